"""Launches of few tiles whose K blocks are summed in parts: as many as a split count, at most 1024 of K each, on 128x64 one
of more than 768 in two halves.  Against the same sums made of launches of one accumulator each, against split-K of as many splits
(the same bits), and, in error, against the split-K that a plan would have taken instead."""
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


def _operands(M, N, K, seed):
    ldk = -(-K // 8) * 8
    a, b = synthetic.operands_bf16(M, N, ldk, seed=seed)
    return ldk, [torch.from_numpy(x.view(np.int16)).cuda().view(torch.bfloat16) for x in (a, b)]


def _accumulators(tile, kb0, kb1, longest):
    """K block ranges of a unit's accumulators: a list of parts, each one or two of them; a launch's units have all as
    many parts, by the longest one's K blocks."""
    n = 1
    while 16 * n < longest:
        n *= 2
    out = []
    for t in range(n):
        lo, hi = kb0 + t * (kb1 - kb0) // n, kb0 + (t + 1) * (kb1 - kb0) // n
        mid = lo + (hi - lo) // 2
        out.append([(lo, mid), (mid, hi)] if hi - lo > 12 and tile == 0 else [(lo, hi)])
    return out


# K blocks: 12 and 13 (one accumulator, two halves), 16, 17 (two parts), 25 (12 and two halves), 32, 33, 64, 65 (eight)
@pytest.mark.parametrize("K", [768, 769, 1024, 1080, 1599, 2048, 2104, 4096, 4104])
@pytest.mark.parametrize("tile, split", [(0, 1), (1, 1), (3, 1), (0, 2), (0, 4)])
@pytest.mark.parametrize("M, N, beta", [(1, 8, 0), (300, 392, 1)])
def test_sums_are_those_of_their_accumulators(rg, ctx, tile, split, M, N, beta, K):
    ldk, (A, B) = _operands(M, N, K, 6)
    c0 = torch.from_numpy(synthetic.normal_stream_f32(6, 3, M * N)).cuda().view(M, N)
    v, kb = rg.variant(tile, split), -(-K // 64)

    def one(lo, hi):
        P = torch.zeros((M, N), device="cuda")
        k0, k1 = 64 * lo, min(K, 64 * hi)
        rg.rg_gemm(ctx, M, N, k1 - k0, A[:, k0:], ldk, B[k0:], N, P, N, rg.variant(tile, 1))
        return P
    total = None
    for s in range(split):
        unit = None
        for part in _accumulators(tile, s * kb // split, (s + 1) * kb // split, -(-kb // split)):
            x = one(*part[0])
            if len(part) == 2:
                x = x + one(*part[1])
            unit = x if unit is None else unit + x
        total = unit if total is None else total + unit
    want = c0 + total if beta else total
    C = c0.clone()
    rg.rg_gemm(ctx, M, N, K, A, ldk, B, N, C, N, v, beta)
    rg.rg_check(ctx)
    assert torch.equal(C, want)
    g = rg.rg_group_create(ctx, 1, 64, 64 << 20)
    try:
        for n in (1, 40):  # 40 problems: K blocks enough for every CTA, so splits run in turn
            outs = [c0.clone() for _ in range(n)]
            rg.rg_gemm_grouped(g, rg.group_problems([(M, N, K, A, ldk, B, N, G, N, beta, 0, 0, 0, v) for G in outs]), n)
            rg.rg_check(ctx)
            assert all(torch.equal(want, G) for G in outs)
    finally:
        rg.rg_group_destroy(g)


@pytest.mark.parametrize("K", [2176, 2560, 2691, 2736, 3072])
@pytest.mark.parametrize("tile", [0, 1, 3])
def test_four_parts_have_the_bits_of_four_splits(rg, ctx, tile, K):
    M, N = 208, 256
    ldk, (A, B) = _operands(M, N, K, 7)
    C, R = (torch.empty((M, N), device="cuda") for _ in range(2))
    rg.rg_gemm(ctx, M, N, K, A, ldk, B, N, C, N, rg.variant(tile, 1))
    rg.rg_gemm(ctx, M, N, K, A, ldk, B, N, R, N, rg.variant(tile, 4))
    rg.rg_check(ctx)
    assert torch.equal(C, R)


@pytest.mark.parametrize("K", [1827, 1920, 2048, 2176, 2736, 3072, 4096])
def test_no_split_is_as_close_as_four(rg, ctx, K):
    """K = 1827..4096 on 128x64: accumulators no longer than those of four splits, so the error (2-norm, relative to the
    result's) differs by the three additions of the partial sums at most, 2^-24 each."""
    M, N = 256, 224
    ldk, (A, B) = _operands(M, N, K, 8)
    exact = A[:, :K].double() @ B[:K].double()

    def error(split):
        C = torch.empty((M, N), device="cuda")
        rg.rg_gemm(ctx, M, N, K, A, ldk, B, N, C, N, rg.variant(0, split))
        rg.rg_check(ctx)
        return float((C.double() - exact).norm() / exact.norm())
    four = error(4)
    assert error(1) <= four + 3 * 2.0 ** -24 and error(2) <= four + 3 * 2.0 ** -24
