"""Norms of the residual kernel: the sums keep the range of FP64 where the
squares of complex64 entries do not fit an FP32 sum, infinities stay infinite,
NaN stays NaN."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pcx():
    from paper_2511_17107_gb300 import pcx as p
    p.lib()
    return p


def _run(pcx, x, ax, theta):
    X, AX = torch.from_numpy(x).cuda(), torch.from_numpy(ax).cuda()
    R = torch.empty_like(X)
    norms = torch.empty(2 * x.shape[0], dtype=torch.float64, device="cuda")
    pcx.pcx_residual(X, AX, torch.from_numpy(theta).cuda(), R, norms)
    return R.cpu().numpy(), norms.cpu().numpy().reshape(2, -1)


# Squares carry two roundings of 2^-24 each, the sums far less.
@pytest.mark.parametrize("L", [1, 7, 255, 257, 20001, 300000])
@pytest.mark.parametrize("nvec", [1, 3, 17])
@pytest.mark.parametrize("size", [1e-6, 1.0, 1e13, 9e18])
def test_norms(pcx, L, nvec, size):
    """At 9e18 four squares exceed the FP32 range; long columns put some ten to some hundred in a thread's sum."""
    rng = np.random.default_rng(L + nvec)
    cx = lambda: (size * np.exp(2j * np.pi * rng.random((nvec, L)))).astype(np.complex64)
    x, ax = cx(), cx()
    theta = np.zeros(nvec)
    r, norms = _run(pcx, x, ax, theta)
    assert np.array_equal(r, ax)
    for got, v in zip(norms, (ax, x)):
        want = (np.abs(v.astype(np.complex128)) ** 2).sum(axis=1)
        assert np.all(np.isfinite(got)) and np.all(np.abs(got - want) <= 2.0 ** -22 * want)


@pytest.mark.parametrize("dtype", [np.complex64, np.complex128])
@pytest.mark.parametrize("L", [1, 100, 100000])
def test_non_finite(pcx, dtype, L):
    rng = np.random.default_rng(5)
    x = (rng.standard_normal((4, L)) + 1j * rng.standard_normal((4, L))).astype(dtype)
    ax = x.copy()
    ax[0, L // 2] = np.inf
    ax[1, L - 1] = complex(0.0, -np.inf)
    ax[2, 0] = np.nan
    if dtype == np.complex64:
        ax[3, 0] = 3e19   # its square is infinite in FP32
    _, norms = _run(pcx, x, ax, np.zeros(4))
    assert np.isposinf(norms[0, 0]) and np.isposinf(norms[0, 1]) and np.isnan(norms[0, 2])
    assert np.isposinf(norms[0, 3]) == (dtype == np.complex64)
    assert np.all(np.isfinite(norms[1]))
