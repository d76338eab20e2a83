"""Launches whose K blocks are summed in several accumulators in turn (few tiles, K beyond 1024): the bits of
split-K with as many splits, which sums the same K ranges in the same order, and the same bits in a grouped call."""
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
@pytest.mark.parametrize("tile", [0, 1, 3])
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


# 128x64 with split-K and K beyond 1024 to a split: alone, in a grouped call of one problem and in one
# that fills the chip; each split's sum is that of its accumulators, in order
@pytest.mark.parametrize("split, K", [(2, 2049), (2, 4096), (4, 5000), (8, 9000)])
@pytest.mark.parametrize("M, N, beta", [(1, 8, 0), (300, 392, 1), (512, 1024, 0)])
def test_split_segments(rg, ctx, split, K, M, N, beta):
    ldk = -(-K // 8) * 8
    a, b = synthetic.operands_bf16(M, N, ldk, seed=4)
    A, B = (torch.from_numpy(x.view(np.int16)).cuda().view(torch.bfloat16) for x in (a, b))
    c0 = torch.from_numpy(synthetic.normal_stream_f32(4, 3, M * N)).cuda().view(M, N)
    v = rg.variant(0, split)
    C, R = c0.clone(), c0.clone()
    rg.rg_gemm(ctx, M, N, K, A, ldk, B, N, C, N, v, beta)
    # the sum by hand: every split's K blocks in as many accumulators, each a launch of its own
    kb = -(-K // 64)
    subs = -(-(-(-kb // split)) // 16)
    total = None
    for s in range(split):
        lo, hi = s * kb // split, (s + 1) * kb // split
        part = None
        for j in range(subs):
            k0, k1 = 64 * (lo + j * (hi - lo) // subs), min(K, 64 * (lo + (j + 1) * (hi - lo) // subs))
            P = torch.zeros((M, N), device="cuda")
            rg.rg_gemm(ctx, M, N, k1 - k0, A[:, k0:], ldk, B[k0:], N, P, N, rg.variant(0, 1))
            part = P if part is None else part + P
        total = part if total is None else total + part
    R = R + total if beta else total
    rg.rg_check(ctx)
    assert subs > 1 and torch.equal(C, R)
    g = rg.rg_group_create(ctx, 1, 64, 64 << 20)
    try:
        for n in (1, 40):  # 40 problems: K blocks enough for every CTA
            outs = [c0.clone() for _ in range(n)]
            rg.rg_gemm_grouped(g, rg.group_problems([(M, N, K, A, ldk, B, N, G, N, beta, 0, 0, 0, v) for G in outs]), n)
            rg.rg_check(ctx)
            assert all(torch.equal(C, G) for G in outs)
    finally:
        rg.rg_group_destroy(g)
