"""The one-launch apply and T0 of 8^3 and 16^3 complex64 vectors against the
oracle: material ids and dense cell blocks, several vectors and Bloch vectors,
T0 in place.  Tolerance 2e-5 of the largest output, as for every complex64
apply (24 stages of a few 2^-24 each, see test_gpu_apply.py)."""
import numpy as np
import pytest

import workloads as wl
from oracle import fourier, penalty, permittivity

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
KS = np.array([[0.6, 1.3, -0.5], [2.0, -1.0, 3.0], [0.3, 0.2, 0.1]])


@pytest.fixture(scope="module")
def pcx():
    from paper_2511_17107_gb300 import pcx as p
    p.lib()
    return p


def _close(got, want):
    assert np.abs(got - want).max() <= 2e-5 * np.abs(want).max()


@pytest.mark.parametrize("n", [8, 16])
@pytest.mark.parametrize("dense", [False, True])
def test_apply_and_t0(pcx, n, dense):
    s = wl.fcc_air_spheres()
    ctx = pcx.setup_structure(s, n)
    if dense:
        ctx = pcx.pcx_setup(n, lattice=s.lattice, cell_blocks=pcx.pcx_cell_blocks(ctx)[0])
    blocks = permittivity.cell_blocks(s, n)
    x = wl.random_block(2 * len(KS), n, seed=n).reshape(len(KS), 2, 3, n, n, n).astype(np.complex64)
    X = torch.from_numpy(x).cuda()
    Y = torch.empty_like(X)
    pcx.pcx_apply_kbatch(ctx, KS, X, Y)
    for i, k in enumerate(KS):
        kap = fourier.kappa(n, s.lattice, k)
        g = penalty.gamma_practical(k)
        xi = x[i].astype(np.complex128)
        _close(Y[i].cpu().numpy(), fourier.apply_symbols(xi, kap, lambda e: permittivity.apply_m(blocks, e), g))
        one = torch.empty_like(X[i])
        pcx.pcx_apply(ctx, k, X[i].contiguous(), one)
        assert torch.equal(one, Y[i])
        k2 = (np.abs(kap) ** 2).sum(0)
        ka = fourier.ka_matrix(kap)
        u = fourier._per_mode(np.conj(np.swapaxes(ka, -1, -2)), xi) / k2
        w = fourier.f3h(permittivity.apply_m(np.linalg.inv(blocks), fourier.f3(u)))
        want = fourier._per_mode(ka, w) / k2 + fourier._per_mode(fourier.kb_matrix(kap), xi) / (g * k2 ** 2)
        t0 = torch.empty_like(X[i])
        pcx.pcx_sandwich_precond(ctx, k, X[i].contiguous(), t0)
        _close(t0.cpu().numpy(), want)
        inplace = X[i].clone()
        pcx.pcx_sandwich_precond(ctx, k, inplace, inplace)
        assert torch.equal(inplace, t0)
