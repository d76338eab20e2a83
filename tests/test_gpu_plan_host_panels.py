"""rg_gemm_plan_host in row panels (page-locked blocks of memory large enough that copies and GEMMs run side by side): the
device path's result bit for bit, for plans of one leaf in every kind of variant and of many leaves with K phases,
and for the calls that stay whole (stream-K, C over A, pageable C)."""
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


def _check(rg, ctx, plan, M, N, K, out=None, over_a=False):
    a_bits, b_bits = synthetic.operands_bf16(M, N, K, seed=3)
    a, b = (torch.from_numpy(np.ascontiguousarray(x.view(np.int16))).pin_memory() for x in (a_bits, b_bits))
    la, lb = -(-K // 8) * 8, -(-N // 8) * 8
    A, B = torch.zeros((M, la), dtype=torch.int16), torch.zeros((K, lb), dtype=torch.int16)
    A[:, :K], B[:, :N] = a, b
    A, B = A.cuda().view(torch.bfloat16), B.cuda().view(torch.bfloat16)
    C = torch.full((M, lb), float("nan"), device="cuda")
    rg.rg_gemm_plan(ctx, plan, M, N, K, A, la, B, lb, C, lb)
    rg.rg_check(ctx)
    if over_a:  # C starts at A's first element
        buf = torch.zeros(M * N, dtype=torch.float32).pin_memory()
        buf.view(torch.int16)[: M * K] = a.reshape(-1)
        a, c = buf, buf
    else:
        c = torch.full((M, N), float("nan"))
        c = c.pin_memory() if out is None else c
    for _ in range(1 if over_a else 2):
        rg.rg_gemm_plan_host(ctx, plan, M, N, K, a, K, b, N, c, N)
    assert torch.equal(C.cpu()[:, :N], c.reshape(-1)[: M * N].reshape(M, N))


# one leaf: fixed tile, split-K through the workspace and through clusters, the pairs whole and split, stream-K
@pytest.mark.parametrize("tile, split", [(1, 1), (0, 8), (5, 2), (2, 4), (5, "2SM"), (4, ("2SM", 2)), (1, "SK"),
                                         (5, "2SM-SK")])
@pytest.mark.parametrize("shape", [(1537, 2304, 64), (512, 7168, 200), (4000, 1800, 136)])
def test_one_leaf(rg, ctx, tile, split, shape):
    plan = rg.rg_plan_build(rg.make_grid(*((-(-x // 128) * 128, -(-x // 128) * 128, 1) for x in shape)),
                            np.ones((1, 1), np.int64), [rg.variant(tile, split)])
    try:
        _check(rg, ctx, plan, *shape)
    finally:
        rg.rg_plan_free(plan)


@pytest.mark.parametrize("shape", [(2048, 2048, 256), (2000, 1800, 1024), (1600, 2304, 72)])
def test_many_leaves(rg, ctx, shape):
    vids = [0, 5, 10, 14, 17, 21]
    T0 = np.random.default_rng(9).integers(50, 5000, size=(len(vids), 18, 18, 8)).astype(np.int64)
    plan = rg.rg_plan_build(rg.make_grid((128, 128, 18), (128, 128, 18), (128, 128, 8)), T0, vids)
    try:
        _check(rg, ctx, plan, *shape)
    finally:
        rg.rg_plan_free(plan)


def test_whole_calls(rg, ctx):
    M, N, K = 2048, 2048, 256
    plan = rg.rg_plan_build(rg.make_grid(*((x, x, 1) for x in (M, N, K))), np.ones((1, 1), np.int64), [rg.variant(1, 1)])
    try:
        _check(rg, ctx, plan, M, N, K, over_a=True)
        _check(rg, ctx, plan, M, N, K, out="pageable")
    finally:
        rg.rg_plan_free(plan)
