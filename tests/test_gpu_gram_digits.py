"""Digit Gram products (complex128, and complex128 x complex64) against
extended-precision sums at the edges of the kernel: column counts around the
tile and launch sizes, row counts around a chunk, columns whose scale rises
along the rows or differs by hundreds of binary orders, limits of the digits,
zero columns, Inf and NaN.

Tolerance.  An entry is rounded to 2^-50 2^E with 2^E at most twice the
column's largest part M; a complex product has two such errors in each of its
two real terms (2^-46 M M' in all), the digit pairs left out add 2^-45 M M',
the last group's fraction and its rounding less, so |error| <= L 2^-44 M M'.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _scale(kind, ncol, L, single, rng):
    lim = 60 if single else 300
    if kind == "rising":   # grows from row to row: the running exponents change in most chunks
        return np.tile(2.0 ** np.minimum(np.arange(L) / 11.0, lim), (ncol, 1))
    if kind == "spread":
        return np.tile((2.0 ** rng.integers(-lim, lim, size=(ncol, 1))), (1, L))
    return np.ones((ncol, L))


def _block(kind, ncol, L, dtype, seed):
    rng = np.random.default_rng(seed)
    x = rng.standard_normal((ncol, L)) + 1j * rng.standard_normal((ncol, L))
    if kind == "limits":   # powers of two, their neighbours below, zeros, subnormals, constant columns
        eps = np.finfo(np.float32 if dtype == np.complex64 else np.float64).eps
        tiny = 1e-42 if dtype == np.complex64 else 1e-310
        vals = np.array([1.0, -1.0, 1 - eps, -(1 - eps / 2), 0.5, 0.0, tiny, 2.0 ** -49, 513 / 1024, -511.5 / 1024])
        x = rng.choice(vals, size=(ncol, L)) + 1j * rng.choice(vals, size=(ncol, L))
        x[0] = (1 - eps) * (1 - 1j)
        x[-1] = 0.0
    return (x * _scale(kind, ncol, L, dtype == np.complex64, rng)).astype(dtype)


def _gram(pcx, a, b):
    import torch
    A, B = torch.from_numpy(a).cuda(), torch.from_numpy(b).cuda()
    if a is b:
        B = A
    G = torch.empty((a.shape[0], b.shape[0]), dtype=torch.complex128, device="cuda")
    (pcx.pcx_gram if b.dtype == np.complex128 else pcx.pcx_gram_mixed)(A, B, G)
    return G.cpu().numpy()


@pytest.fixture(scope="module")
def pcx():
    from paper_2511_17107_gb300 import pcx as p
    p.lib()
    return p


def _check(a, b, got):
    L = a.shape[1]
    want = a.conj().astype(np.clongdouble) @ b.T.astype(np.clongdouble)
    mag = [np.maximum(np.abs(v.real), np.abs(v.imag)).max(axis=1).astype(np.longdouble) for v in (a, b)]
    bound = L * np.longdouble(2.0) ** -44 * mag[0][:, None] * mag[1][None, :]
    assert np.all(np.abs(got - want) <= bound)
    return want


@pytest.mark.parametrize("na,nb", [(1, 1), (7, 9), (8, 8), (16, 32), (17, 23), (33, 40), (48, 48), (49, 12), (5, 97),
                                   (128, 128)])
@pytest.mark.parametrize("mixed", [False, True])
def test_shapes(pcx, na, nb, mixed):
    for L in (1, 31, 33, 700):
        a = _block("plain", na, L, np.complex128, 1)
        b = _block("plain", nb, L, np.complex64 if mixed else np.complex128, 2)
        got = _gram(pcx, a, b)
        want = _check(a, b, got)
        norms = np.linalg.norm(a, axis=1)[:, None] * np.linalg.norm(b, axis=1)[None, :]
        assert np.all(np.abs(got - want) <= 4e-14 * norms)


@pytest.mark.parametrize("n", [1, 9, 16, 43, 48, 60])
def test_hermitian(pcx, n):
    a = _block("plain", n, 1234, np.complex128, 3)
    got = _gram(pcx, a, a)
    _check(a, a, got)
    if n <= 48:   # one launch: the lower triangle is the exact mirror
        assert np.array_equal(got, got.conj().T)


@pytest.mark.parametrize("kind", ["rising", "spread", "limits"])
@pytest.mark.parametrize("mixed", [False, True])
def test_ranges(pcx, kind, mixed):
    a = _block(kind, 13, 2500, np.complex128, 4)
    b = _block(kind, 10, 2500, np.complex64 if mixed else np.complex128, 5)
    _check(a, b, _gram(pcx, a, b))
    if not mixed:
        _check(a, a, _gram(pcx, a, a))


@pytest.mark.parametrize("row", [31, 32, 63, 64, 96])
@pytest.mark.parametrize("mixed", [False, True])
def test_exponent_steps_between_chunks(pcx, row, mixed):
    """A column's scale jumps 2^40-fold at one row (chunks hold 32) and stays: every lane that cuts the column has
    to see the new exponent in the next chunk, from the first to the second one too."""
    for na, nb in ((1, 1), (16, 16), (48, 31)):
        a = _block("plain", na, 128, np.complex128, 8)
        b = _block("plain", nb, 128, np.complex64 if mixed else np.complex128, 9)
        a[:, row:] *= 2.0 ** 40
        b[:, row:] *= 2.0 ** 40
        _check(a, b, _gram(pcx, a, b))


@pytest.mark.parametrize("value", [np.inf, -np.inf, np.nan])
def test_non_finite(pcx, value):
    a = _block("plain", 9, 300, np.complex128, 6)
    b = _block("plain", 6, 300, np.complex64, 7)
    a[4, 250] = complex(0.0, value)
    b[2, 3] = complex(value, 1.0)
    got = _gram(pcx, a, b)
    bad = np.zeros(got.shape, dtype=bool)
    bad[4], bad[:, 2] = True, True
    assert np.all(np.isnan(got[bad].real)) and np.all(np.isnan(got[bad].imag))
    ra, rb = [i for i in range(9) if i != 4], [j for j in range(6) if j != 2]
    _check(a[ra], b[rb], got[np.ix_(ra, rb)])


def test_long_columns(pcx):
    """More rows than one CTA takes in a launch of one wave: the exact value of a constant column's Gram."""
    import torch
    L = 3 * 10 ** 6
    A = torch.full((2, L), 1.0 - 2.0 ** -52, dtype=torch.complex128, device="cuda")
    A[1] = -1j * A[0]
    G = torch.empty((2, 2), dtype=torch.complex128, device="cuda")
    pcx.pcx_gram(A, A, G)
    v = L * (1.0 - 2.0 ** -52) ** 2
    want = np.array([[v, -1j * v], [1j * v, v]])
    assert np.abs(G.cpu().numpy() - want).max() <= v * 2.0 ** -44


# Columns graded against each other and columns with one dominant entry.
#
# An entry is cut relative to its column's largest part M_c in its chunk of 32
# rows (2^E <= 2 M_c).  The pairs left out and the rounding of the entries come
# to 2^-50 2^(Ea + Eb) rms in a real product, so 2^-47.5 sqrt(sum over rows of
# (M_c M'_c)^2) in an entry of G; the tolerance takes 11 times that.  The sums
# of the chunks are kept to about 2^-49 of the running sum at each addition:
# 2^-47 sum |a||b| holds for them with room.
def _graded_bound(a, b):
    L = a.shape[1]
    mag = [np.maximum(np.abs(v.real), np.abs(v.imag)).reshape(v.shape[0], L // 32, 32).max(axis=2) for v in (a, b)]
    sq = 32 * (mag[0] ** 2 @ (mag[1] ** 2).T)
    return 2.0 ** -44 * np.sqrt(sq) + 2.0 ** -47 * (np.abs(a) @ np.abs(b).T.astype(np.float64))


@pytest.mark.parametrize("decades", [3, 6, 9])
@pytest.mark.parametrize("mixed", [False, True])
@pytest.mark.parametrize("na,nb", [(2, 3), (18, 17), (35, 3)])
def test_graded_columns(pcx, decades, mixed, na, nb):
    """A falls and B rises by `decades` over every 1024 rows, so all rows weigh alike in the products."""
    L = 32 * 6250
    t = 10.0 ** (decades * (np.arange(L) % 1024) / 1024.0)
    rng = np.random.default_rng(decades)
    cx = lambda *sh: rng.standard_normal(sh) + 1j * rng.standard_normal(sh)
    a = cx(na, L) / t
    b = (cx(nb, L) * t).astype(np.complex64 if mixed else np.complex128)
    got = _gram(pcx, a, b)
    want = np.zeros((na, nb), dtype=np.clongdouble)
    for i in range(na):
        for j in range(nb):
            want[i, j] = (a[i].conj().astype(np.clongdouble) * b[j].astype(np.clongdouble)).sum()
    assert np.all(np.abs(got - want) <= _graded_bound(a, b))


@pytest.mark.parametrize("mixed", [False, True])
def test_dominant_entry(pcx, mixed):
    """One entry 1000 times the others in long columns.  Its chunk errs by about 2^-47 M M' (as above); the other
    chunks are cut by their own size, and adding some hundred of them to the large sum costs 2^-45.5 M M' at most
    where all roundings add up as a random walk: 2^-43 M M' in all."""
    L = 2 * 10 ** 6
    rng = np.random.default_rng(11)
    cx = lambda *sh: rng.standard_normal(sh) + 1j * rng.standard_normal(sh)
    a, b = cx(2, L), cx(2, L)
    a[:, 5], b[:, 5] = 1000.0 - 300.0j, 700.0 + 900.0j
    b = b.astype(np.complex64 if mixed else np.complex128)
    got = _gram(pcx, a, b)
    want = np.array([[(x.conj().astype(np.clongdouble) * y.astype(np.clongdouble)).sum() for y in b] for x in a])
    assert np.abs(got - want).max() <= 2.0 ** -43 * 1000.0 * 900.0
