"""Kernels that take a cell or a mode through a group of vectors (the M_CrossDoF
stencil, K_P^{-1}): counts that give one vector, full groups and ragged last
groups, against the oracle for the vectors at the groups' ends and bit for bit
against the same vectors one at a time.  Tolerances as in test_gpu_apply.py:
1e-12 (complex128), 2e-5 (complex64) of the largest output."""
import numpy as np
import pytest

import workloads as wl
from oracle import crossdof, fourier, penalty

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
TOL = {np.complex64: 2e-5, np.complex128: 1e-12}
K = np.array([0.6, 1.3, -0.5])


@pytest.fixture(scope="module")
def pcx():
    from paper_2511_17107_gb300 import pcx as p
    p.lib()
    return p


def _check(pcx, ctx, call, x, oracle, chunks):
    dtype = x.dtype.type
    X = torch.from_numpy(x).cuda()
    Y = torch.empty_like(X)
    call(ctx, K, X, Y)
    one = torch.empty_like(X[:1])
    for j in range(x.shape[0]):
        call(ctx, K, X[j:j + 1].contiguous(), one)
        assert torch.equal(one[0], Y[j]), j
    for j in sorted({0, x.shape[0] // 2, x.shape[0] - 1}):
        want = oracle(x[j:j + 1].astype(np.complex128))[0]
        assert np.abs(Y[j].cpu().numpy() - want).max() <= TOL[dtype] * np.abs(want).max()
    Z = torch.empty_like(X)
    for chunk in chunks:
        pcx.pcx_set_apply_chunk(ctx, chunk)
        call(ctx, K, X, Z)
        assert torch.equal(Y, Z), chunk
    pcx.pcx_set_apply_chunk(ctx, 0)


@pytest.mark.parametrize("n,nvec", [(8, 40), (16, 17), (32, 18), (64, 2), (64, 17)])
@pytest.mark.parametrize("dtype", [np.complex64, np.complex128])
def test_crossdof(pcx, n, nvec, dtype):
    s = wl.bcc_gyroid()
    m = crossdof.CrossDofM(s, n)
    kap = fourier.kappa(n, s.lattice, K)
    g = penalty.gamma_practical(K)
    ctx = pcx.setup_structure(s, n, m_kind=pcx.PCX_M_CROSSDOF)
    x = wl.random_block(nvec, n, seed=n + nvec).astype(dtype)
    _check(pcx, ctx, pcx.pcx_apply, x, lambda v: fourier.apply_symbols(v, kap, m.apply, g), (1, 5, nvec))


@pytest.mark.parametrize("n,nvec", [(8, 1), (16, 33), (32, 5), (64, 1), (64, 17)])
@pytest.mark.parametrize("dtype", [np.complex64, np.complex128])
def test_precond(pcx, n, nvec, dtype):
    s = wl.fcc_air_spheres()
    kap = fourier.kappa(n, s.lattice, K)
    g = penalty.gamma_practical(K)
    ctx = pcx.setup_structure(s, n)
    x = wl.random_block(nvec, n, seed=n + nvec).astype(dtype)
    _check(pcx, ctx, pcx.pcx_precond, x, lambda v: fourier.precondition(v, kap, g), ())


@pytest.mark.parametrize("call", ["pcx_apply", "pcx_sandwich_precond"])
@pytest.mark.parametrize("dense", [False, True])
def test_lone_vector_of_the_three_pass_chain(pcx, call, dense):
    """A lone 64^3 complex64 vector runs half tiles in the z pass: same bits as in a block."""
    n = 64
    s = wl.fcc_air_spheres()
    ctx = pcx.setup_structure(s, n)
    if dense:
        ctx = pcx.pcx_setup(n, lattice=s.lattice, cell_blocks=pcx.pcx_cell_blocks(ctx)[0])
    x = wl.random_block(3, n, seed=3).astype(np.complex64)
    X = torch.from_numpy(x).cuda()
    Y = torch.empty_like(X)
    getattr(pcx, call)(ctx, K, X, Y)
    one = torch.empty_like(X[:1])
    for j in range(3):
        getattr(pcx, call)(ctx, K, X[j:j + 1].contiguous(), one)
        assert torch.equal(one[0], Y[j]), j


@pytest.mark.parametrize("nvec", [2, 3, 4])
def test_few_vectors_at_128(pcx, nvec):
    """Two and three 128^3 vectors go one by one, four in one launch: same bits either way."""
    n = 128
    ctx = pcx.setup_structure(wl.diamond_rods(), n)
    X = torch.from_numpy(wl.random_block(nvec, n, seed=nvec).astype(np.complex64)).cuda()
    for call in (pcx.pcx_apply, pcx.pcx_sandwich_precond):
        out = []
        for chunk in (0, 1, nvec):
            pcx.pcx_set_apply_chunk(ctx, chunk)
            out.append(torch.empty_like(X))
            call(ctx, K, X, out[-1])
        assert torch.equal(out[0], out[1]) and torch.equal(out[0], out[2])
