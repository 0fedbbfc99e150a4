"""complex128 combinations in double-float arithmetic: widths of the output
sweeps (4, 8, 12, 16 and remainders), long and ragged columns, entries over
many decades, values at the ends of the FP32 range."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pcx():
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    from paper_2511_17107_gb300 import pcx as m
    return m


def combine(pcx, s, c, y, beta):
    Y = torch.from_numpy(y.copy()).cuda()
    pcx.pcx_combine(torch.from_numpy(s).cuda(), torch.from_numpy(c).cuda(), Y, beta=beta)
    return Y.cpu().numpy()


# Entrywise bound, B = sum |S||C| of an output: entries split to 2^-49 and 2 ns
# products whose compensation (up to 2^-24 B) is rounded to 24 bits each time.
# As a random walk that is about sqrt(4 ns) 2^-50 B; 2^-46 sqrt(2 ns + 8) B
# leaves a factor of 8 and more.
@pytest.mark.parametrize("ns,ny,L,beta", [(1, 1, 1, 0.0), (3, 4, 63, 0.0), (16, 16, 12345, 0.0), (16, 5, 64, 1.0),
                                          (43, 9, 65, -0.5), (7, 17, 257, 0.0), (33, 13, 3 * 16 ** 3, 1.0),
                                          (130, 12, 1000, 0.0), (256, 33, 300, 0.0), (5, 3, 3 * 64 ** 3, 0.0)])
def test_entrywise(pcx, ns, ny, L, beta):
    rng = np.random.default_rng(ns * 100 + ny)
    cx = lambda *sh: rng.standard_normal(sh) + 1j * rng.standard_normal(sh)
    s = cx(ns, L) * 10.0 ** rng.uniform(-9, 0, (1, L)) * 10.0 ** rng.uniform(-3, 0, (ns, 1))
    c = cx(ns, ny) * 10.0 ** rng.uniform(-9, 0, (ns, 1))
    y = cx(ny, L)
    got = combine(pcx, s, c, y, beta)
    want = np.zeros((ny, L), dtype=np.clongdouble)
    for i in range(ns):
        want += c[i][:, None].astype(np.clongdouble) * s[i][None]
    want += beta * y
    bound = 2.0 ** -46 * np.sqrt(2 * ns + 8) * (np.abs(c).T @ np.abs(s)) * 2 + 2.0 ** -52 * np.abs(want).astype(float)
    assert np.all(np.abs(got - want) <= bound)


def test_range_ends(pcx):
    top = np.nextafter(2.0 ** 128, 0)      # rounds to infinity in FP32, its leading 24 bits do not
    s = np.array([[top, -top, 2.0 ** -130, np.inf, np.nan, 1.0]], dtype=np.complex128)
    c = np.array([[0.25]], dtype=np.complex128)
    got = combine(pcx, s, c, np.zeros((1, 6), dtype=np.complex128), 0.0)[0]
    assert abs(got[0] - top / 4) <= 2.0 ** -46 * top and abs(got[1] + top / 4) <= 2.0 ** -46 * top
    assert got[2] == 0 and got[5] == 0.25                # below the FP32 normal range: 0
    assert np.isnan(got[3].real) and np.isnan(got[4].real)
