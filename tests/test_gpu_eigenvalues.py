"""Eigenvalues of FP64 solves against the Rayleigh-Ritz values of the vectors
that the same call returns."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
K = np.full(3, np.pi)


@pytest.fixture(scope="module")
def pcx():
    from paper_2511_17107_gb300 import pcx as p
    p.lib()
    return p


# The residual of 1e-8 leaves |res|^2 / gap, about 1e-16, in a Ritz value; the
# products that form the block's small matrices are good to 1e-14 of theirs.
@pytest.mark.parametrize("stencil", [1, 5])
@pytest.mark.parametrize("block", [12, 14])
def test_eigenvalues_are_those_of_the_vectors(pcx, stencil, block):
    """A smooth permittivity between 4 and 22 at k = (pi, pi, pi): a cluster of six eigenvalues, and with 10th-order
    stencils a search space that is ill conditioned late in the solve."""
    n, nev = 32, 8
    i = np.arange(1, n + 1) / n
    z, y, x = np.meshgrid(i, i, i, indexing="ij")
    blocks = np.zeros((n ** 3, 9))
    for c in range(3):
        blocks[:, c] = (1.0 / (8.9 * np.sin(2 * np.pi * (x + y + z - 0.5 / n)) + 13.0)).reshape(-1)
    ctx = pcx.pcx_setup(n, stencil_m=stencil, cell_blocks=blocks)
    for seed in range(1, 7):
        vec = torch.empty((1, nev, 3, n, n, n), dtype=torch.complex128, device="cuda")
        ev, res, _, st = pcx.pcx_solve(ctx, [K], nev, 1e-8, block=block, precision=pcx.PCX_FP64, precond_kind=1,
                                       seed=seed, vec_out=vec)
        assert st == pcx.PCX_OK and np.all(np.diff(ev[0]) >= 0)
        img = torch.empty_like(vec[0])
        pcx.pcx_apply(ctx, K, vec[0], img)
        v, w = vec[0].reshape(nev, -1), img.reshape(nev, -1)
        g, a = (v.conj() @ v.T).cpu().numpy(), (v.conj() @ w.T).cpu().numpy()
        inv = np.linalg.inv(np.linalg.cholesky(g))
        want = np.linalg.eigvalsh(inv @ (0.5 * (a + a.conj().T)) @ inv.conj().T)
        assert np.all(np.abs(ev[0] - want) <= 1e-12 * want), (seed, np.abs(ev[0] - want) / want)
