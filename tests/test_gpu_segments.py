"""Unsplit launches whose K blocks are summed in several accumulators in turn (few tiles, K beyond 1024): the bits of
split-K with as many splits, which sums the same K ranges in the same order, alone and in a grouped call."""
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


# K: one accumulator up to 1024; 2 of 8 or 9 and of 16 blocks, 4 with a ragged last block, 8
@pytest.mark.parametrize("K, segs", [(1024, 1), (1032, 2), (2048, 2), (3100, 4), (8000, 8)])
@pytest.mark.parametrize("tile", [0, 1, 3, 6])
@pytest.mark.parametrize("M, N, beta", [(1, 8, 0), (300, 392, 1), (1000, 1096, 0)])
def test_segments(rg, ctx, tile, M, N, beta, K, segs):
    ldk = -(-K // 8) * 8
    a, b = synthetic.operands_bf16(M, N, ldk, seed=2)
    A, B = (torch.from_numpy(x.view(np.int16)).cuda().view(torch.bfloat16) for x in (a, b))
    c0 = torch.from_numpy(synthetic.normal_stream_f32(2, 3, M * N)).cuda().view(M, N)
    C, R, G = c0.clone(), c0.clone(), c0.clone()
    rg.rg_gemm(ctx, M, N, K, A, ldk, B, N, C, N, rg.variant(tile, 1), beta)
    rg.rg_gemm(ctx, M, N, K, A, ldk, B, N, R, N, rg.variant(tile, segs), beta)
    g = rg.rg_group_create(ctx, 1, 4, 1 << 20)
    try:
        rg.rg_gemm_grouped(g, rg.group_problems([(M, N, K, A, ldk, B, N, G, N, beta, 0, 0, 0, rg.variant(tile, 1))]), 1)
        rg.rg_check(ctx)
        assert torch.equal(C, R) and torch.equal(C, G)
    finally:
        rg.rg_group_destroy(g)
