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


def test_the_untuned_chunk_is_among_the_candidates(pcx):
    """Chunks 1, 2, ..., 64 and the 200 of an untuned context, for both pass structures."""
    ctx = pcx.setup_structure(wl.sc_gyro_sphere(), 32)
    assert pcx.pcx_get_apply_chunk(ctx, pcx.PCX_FP32) >= 200
    r = pcx.pcx_autotune(ctx, pcx.PCX_FP32, 200)
    assert r["candidates"] == 2 * 8 + (7 if r["path"] == pcx.PCX_APPLY_THREE_PASS else 0)


def test_a_variant_that_runs_as_another_is_not_timed(pcx):
    """At N = 128 pass B has one kernel: four x variants, z variant 0 reported."""
    ctx = pcx.setup_structure(wl.diamond_rods(), 128)
    r = pcx.pcx_autotune(ctx, pcx.PCX_FP32, 2)
    three = r["path"] == pcx.PCX_APPLY_THREE_PASS
    assert r["candidates"] == 2 * 2 + (3 if three else 0) and r["z_variant"] == (0 if three else -1)


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
    assert pcx.pcx_autotune(ctx, pcx.PCX_FP32, 256)["candidates"] == 1
    pcx.pcx_set_apply_chunk(ctx, 7)
    pcx.pcx_apply(ctx, K, X, Z)
    assert torch.equal(Y, Z)
    for call in (pcx.pcx_apply_noalloc, pcx.pcx_sandwich_precond):
        a, b = torch.empty_like(X), torch.empty_like(X)
        call(ctx, K, X, a)
        pcx.pcx_set_apply_chunk(ctx, 0)
        call(ctx, K, X, b)
        assert torch.equal(a, b)
