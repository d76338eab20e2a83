"""rg_gemm_plan_host in row panels whose parts of a leaf have fewer tiles than the whole leaf: a leaf of as many tiles as
the chip has SMs sums K in one accumulator, and its panels, which alone would sum it in parts, have to do so too.  K beyond
1024 on the tiles that sum in parts; the device path's result bit for bit, and the call did run in panels."""
import numpy as np
import pytest

import synthetic

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def rg():
    from paper_2605_29752_gb300 import rg as _rg
    return _rg


@pytest.fixture(scope="module")
def ctx(rg):
    h = rg.rg_init(0)
    yield h
    rg.rg_destroy(h)


# 2048 x 2048: 256 tiles of 128x128 and of 256x64, half of them (128 < 152 SMs) to a panel; 512 of 128x64 (256 to a panel)
@pytest.mark.parametrize("tile, split", [(0, 1), (0, 2), (1, 1), (3, 1)])
@pytest.mark.parametrize("M, N, K", [(2048, 2048, 2048), (1792, 2560, 1504), (2304, 2304, 2808)])
def test_panels_of_leaves_beyond_one_wave(rg, ctx, tile, split, M, N, K):
    plan = rg.rg_plan_build(rg.make_grid(*((-(-x // 128) * 128, -(-x // 128) * 128, 1) for x in (M, N, K))),
                            np.ones((1, 1), np.int64), [rg.variant(tile, split)])
    try:
        bits = synthetic.operands_bf16(M, N, K, seed=11)
        a, b = (torch.from_numpy(np.ascontiguousarray(x.view(np.int16))).pin_memory() for x in bits)
        A, B = (x.cuda().view(torch.bfloat16) for x in (a, b))
        C = torch.empty((M, N), device="cuda")
        rg.rg_gemm_plan(ctx, plan, M, N, K, A, K, B, N, C, N)
        rg.rg_check(ctx)
        c = torch.full((M, N), float("nan")).pin_memory()
        before = rg.rg_launch_count(ctx)
        rg.rg_gemm_plan_host(ctx, plan, M, N, K, a, K, b, N, c, N)
        assert rg.rg_launch_count(ctx) - before >= 2        # one launch to a panel
        assert torch.equal(C.cpu(), c)
    finally:
        rg.rg_plan_free(plan)
