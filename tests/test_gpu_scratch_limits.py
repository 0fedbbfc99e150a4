"""An apply whose default scratch does not fit the device's free memory goes on
with smaller launches: same bits."""
import numpy as np
import pytest

import workloads as wl

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
K = np.array([0.6, 1.3, -0.5])


@pytest.fixture(scope="module")
def pcx():
    from paper_2511_17107_gb300 import pcx as p
    p.lib()
    return p


def test_little_free_memory(pcx):
    n, count = 128, 16
    s = wl.diamond_rods()
    roomy, tight = pcx.setup_structure(s, n), pcx.setup_structure(s, n)
    X = torch.randn((count, 3, n, n, n), dtype=torch.complex64, device="cuda")
    Y, Z, T = torch.empty_like(X), torch.empty_like(X), torch.empty_like(X)
    pcx.pcx_apply(roomy, K, X, Y)
    pcx.pcx_sandwich_precond(roomy, K, X, T)
    assert not torch.equal(Y, T)   # its kernels are loaded and its workspace cached while there is room
    torch.cuda.synchronize()
    full = pcx.pcx_get_apply_chunk(tight, pcx.PCX_FP32)
    need = full * n ** 3 * 8
    assert full == 16 and need == 256 << 20
    held = []
    try:
        step = 1 << 38
        while step >= 1 << 24:   # fill the memory down to less than the scratch, more than one vector's
            if torch.cuda.mem_get_info()[0] - step < need // 2:
                step //= 2
                continue
            held.append(torch.empty(step, dtype=torch.uint8, device="cuda"))
        assert torch.cuda.mem_get_info()[0] < need
        pcx.pcx_apply(tight, K, X, Z)
        torch.cuda.synchronize()
        assert torch.equal(Y, Z)
        assert pcx.pcx_get_apply_chunk(tight, pcx.PCX_FP32) < full
        pcx.pcx_sandwich_precond(tight, K, X, Z)
        torch.cuda.synchronize()
        assert torch.equal(T, Z)
    finally:
        del held
        torch.cuda.empty_cache()
