"""The complex128 passes (transforms in 64-bit fixed point): every grid size
against the oracle, independence of the data's scale, sparse lines, and Inf /
NaN.

Tolerance: 1e-14 of the largest output.  A transform of N <= 256 points rounds
its input at 2^-(62 - log2 N) <= 2^-54 of the line's largest entry and every
twiddle product by less; five passes and the FP64 products around them (a few
units of 2^-53 each, symbols normalised by the largest output) stay below
50 x 2^-53 = 5.6e-15.  A scale by a power of two moves only exponents, so the
result is the same bit for bit.
"""
import numpy as np
import pytest

import workloads as wl
from oracle import fourier, penalty, permittivity

pytestmark = pytest.mark.gpu
K = np.array([1.1, -0.4, 2.3])


@pytest.fixture(scope="module")
def pcx():
    from paper_2511_17107_gb300 import pcx as p
    p.lib()
    return p


def _apply(pcx, ctx, x, call="pcx_apply"):
    import torch
    X = torch.from_numpy(np.ascontiguousarray(x)).cuda()
    Y = torch.empty_like(X)
    getattr(pcx, call)(ctx, K, X, Y)
    return Y.cpu().numpy()


def _oracle(s, n, x):
    kap = fourier.kappa(n, s.lattice, K)
    blocks = permittivity.cell_blocks(s, n)
    return fourier.apply_symbols(x, kap, lambda e: permittivity.apply_m(blocks, e), penalty.gamma_practical(K))


@pytest.mark.parametrize("n", [8, 16, 32, 64, 128])
def test_every_grid(pcx, n):
    s = wl.fcc_air_spheres()
    ctx = pcx.setup_structure(s, n)
    x = wl.random_block(3 if n < 64 else 1, n, seed=n)
    got, want = _apply(pcx, ctx, x), _oracle(s, n, x)
    assert np.abs(got - want).max() <= 1e-14 * np.abs(want).max()


def test_sparse_lines(pcx):
    """Lines with one entry, lines of zeros, and magnitudes a million apart in one line."""
    n = 16
    s = wl.sc_gyro_sphere()
    ctx = pcx.setup_structure(s, n)
    x = np.zeros((3, 3, n, n, n), dtype=np.complex128)
    x[0, 1, 3, 5, 7] = 1.0 - 2.0j
    x[1] = wl.random_block(1, n, seed=2)[0] * 10.0 ** np.random.default_rng(3).uniform(-6, 0, size=(3, n, n, n))
    got, want = _apply(pcx, ctx, x), _oracle(s, n, x)
    assert np.abs(got[:2] - want[:2]).max() <= 1e-14 * np.abs(want).max()
    assert np.all(got[2] == 0)


@pytest.mark.parametrize("call", ["pcx_apply", "pcx_sandwich_precond"])
@pytest.mark.parametrize("n", [8, 16, 32, 256])
def test_scale_by_powers_of_two(pcx, n, call):
    s = wl.sc_gyro_sphere()
    ctx = pcx.setup_structure(s, n)
    x = wl.random_block(1, n, seed=n + 1)
    y = _apply(pcx, ctx, x, call)
    assert np.isfinite(y).all()
    for k in ((-900, -60, 60, 950) if n <= 32 else (-900, 950)):
        assert np.array_equal(_apply(pcx, ctx, x * 2.0 ** k, call), y * 2.0 ** k)


@pytest.mark.parametrize("value", [np.inf, -np.inf, np.nan])
def test_non_finite(pcx, value):
    n = 16
    ctx = pcx.setup_structure(wl.sc_gyro_sphere(), n)
    x = wl.random_block(3, n, seed=5)
    clean = _apply(pcx, ctx, x)
    x[1, 2, 4, 9, 11] = complex(1.0, value)
    y = _apply(pcx, ctx, x)
    assert not np.isfinite(y[1]).any()
    assert np.array_equal(y[[0, 2]], clean[[0, 2]])


def test_overflow_gives_infinity(pcx):
    n = 8
    ctx = pcx.setup_structure(wl.sc_gyro_sphere(), n)
    x = wl.random_block(1, n, seed=6) * 2.0 ** 1020
    assert not np.isfinite(_apply(pcx, ctx, x)).all()


@pytest.mark.parametrize("n", [16, 32, 64, 128, 256])
@pytest.mark.parametrize("power", [0.0, 2.0, 4.0])
def test_decaying_modes(pcx, n, power):
    """With M = I the transforms of an apply cancel, y = K_A K_A^H x + gamma K_B x mode by mode, so what is left is
    their rounding.  Modes that fall off as |p|^-power give lines with one large entry, whose transform grows by
    sqrt(N) less than that of an even line.  Each of the six transforms rounds by at most 2^-53 of its norm (as FP64
    does), sqrt(6) 2^-53 = 2.7e-16 in all; the products before and after and those of the expected values add a few
    2^-53 of theirs.  The error of a mode, divided by |kappa_p| (which the last step multiplies in), stays below
    1e-15 in norm."""
    ctx = pcx.pcx_setup(n, eps=np.eye(3)[None], background=0)
    sym, _, b, _ = pcx.pcx_symbols(ctx, K)
    assert np.array_equal(b, np.eye(3))
    kap = [sym[0][None, None, :], sym[1][None, :, None], sym[2][:, None, None]]
    p = np.fft.fftfreq(n, 1.0 / n)
    w = (1.0 + p[:, None, None] ** 2 + p[None, :, None] ** 2 + p[None, None, :] ** 2) ** (-0.5 * power)
    rng = np.random.default_rng(n)
    x = np.empty((1, 3, n, n, n), dtype=np.complex128)
    for c in range(3):
        x[0, c] = w * (rng.standard_normal((n, n, n)) + 1j * rng.standard_normal((n, n, n)))
    import torch
    X = torch.from_numpy(x).cuda()
    Y = torch.empty_like(X)
    pcx.pcx_apply(ctx, K, X, Y, gamma=1.0)
    y = Y.cpu().numpy()[0]
    err = size = 0.0
    for z in range(n):   # a plane of modes at a time
        kz = [kap[0][0], kap[1][0], kap[2][z]]
        kc = [np.conj(v) for v in kz]
        v = x[0, :, z]
        u = [kc[2] * v[1] - kc[1] * v[2], kc[0] * v[2] - kc[2] * v[0], kc[1] * v[0] - kc[0] * v[1]]
        s = kz[0] * v[0] + kz[1] * v[1] + kz[2] * v[2]
        want = [kz[1] * u[2] - kz[2] * u[1] + kc[0] * s, kz[2] * u[0] - kz[0] * u[2] + kc[1] * s,
                kz[0] * u[1] - kz[1] * u[0] + kc[2] * s]
        k2 = sum(np.abs(q) ** 2 for q in kz)
        err += float(sum((np.abs(y[c, z] - want[c]) ** 2 / k2).sum() for c in range(3)))
        size += float(sum((np.abs(q) ** 2).sum() for q in u) + (np.abs(s) ** 2).sum())
    assert np.sqrt(err / size) <= 1e-15


def test_subnormal_results(pcx):
    """Entries around 2^-1022: a result below the normal range is a multiple of 2^-1074, not 0.  Each pass rounds at
    2^-52 of such an entry; passes and symbols of 16^3 leave that below 1e-12 of the largest output."""
    n = 16
    ctx = pcx.setup_structure(wl.sc_gyro_sphere(), n)
    x = wl.random_block(1, n, seed=8)
    y = _apply(pcx, ctx, x)
    small = _apply(pcx, ctx, x * 2.0 ** -1022)
    assert np.abs(small * 2.0 ** 1000 - y * 2.0 ** -22).max() <= 1e-12 * np.abs(y).max() * 2.0 ** -22
