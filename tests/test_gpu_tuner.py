"""What the autotuner times, and the one-launch applies it has nothing to tune in."""
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


@pytest.mark.parametrize("n", [8, 16])
def test_one_launch_applies(pcx, n):
    """Nothing to choose, no scratch, and a set chunk does not split the block: same bits."""
    ctx = pcx.setup_structure(wl.sc_gyro_sphere(), n)
    count = 2000
    X = torch.randn((count, 3, n, n, n), dtype=torch.complex64, device="cuda")
    Y, Z = torch.empty_like(X), torch.empty_like(X)
    pcx.pcx_apply(ctx, K, X[:1].contiguous(), Y[:1].contiguous())
    torch.cuda.synchronize()
    free = torch.cuda.mem_get_info()[0]
    pcx.pcx_apply(ctx, K, X, Y)
    torch.cuda.synchronize()
    assert torch.cuda.mem_get_info()[0] == free
    pcx.pcx_set_apply_chunk(ctx, 7)
    pcx.pcx_apply(ctx, K, X, Z)
    assert torch.equal(Y, Z)
    for call in (pcx.pcx_apply_noalloc, pcx.pcx_sandwich_precond):
        a, b = torch.empty_like(X), torch.empty_like(X)
        call(ctx, K, X, a)
        pcx.pcx_set_apply_chunk(ctx, 0)
        call(ctx, K, X, b)
        assert torch.equal(a, b)
