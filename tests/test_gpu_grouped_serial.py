"""Grouped launches whose K splits run in turn on one CTA (where the launch's tiles fill the chip), against
rg_gemm with the same variant, whose splits run on S CTAs: the same bits, and within the oracle's bound."""
import numpy as np
import pytest

import synthetic
from oracle import gemm as og

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


def _cuda(bits):
    return torch.from_numpy(bits.view(np.int16)).cuda().view(torch.bfloat16)


# tile, split (2SM: a cta_group::2 pair); K block counts of 2 to 65 on both sides of the split counts
@pytest.mark.parametrize("tile, pair", [(0, False), (1, False), (3, False), (4, True), (2, False), (6, False)])
@pytest.mark.parametrize("split", [2, 4, 8])
def test_serial_splits_equal_rg_gemm(rg, ctx, tile, pair, split):
    v = rg.variant(tile, (rg.TWO_SM, split)) if pair else rg.variant(tile, split)
    shapes = [(1030, 1096, 1003, 0, 0), (1024, 1024, 520, 1, 0), (130, 72, 4104, 0, 0), (2048, 1024, 448, 0, 1024),
              (1500, 2000, 129, 1, 0), (96, 200, 700, 0, 0), (2048, 1536, 1280, 0, 0)]
    g = rg.rg_group_create(ctx, 1, 8, 512 << 20)
    try:
        probs, pairs, hosts = [], [], []
        for i, (M, N, K, beta, pk) in enumerate(shapes):
            ldk, ldn = -(-K // 8) * 8, -(-N // 8) * 8
            a, b = synthetic.operands_bf16(M, ldn, ldk, seed=70 + i)
            A, B = _cuda(a), _cuda(b)
            c0 = torch.from_numpy(synthetic.normal_stream_f32(70 + i, 3, M * ldn)).cuda().view(M, ldn)
            C, R = c0.clone(), c0.clone()
            rg.rg_gemm(ctx, M, N, K, A, ldk, B, ldn, R, ldn, v, beta, M if pk else 0, N if pk else 0, pk)
            probs.append((M, N, K, A, ldk, B, ldn, C, ldn, beta, M if pk else 0, N if pk else 0, pk, v))
            pairs.append((C, R))
            hosts.append((a[:, :K], b[:K, :N], c0 if beta else None, M, N, K))
        rg.rg_gemm_grouped(g, probs)
        rg.rg_check(ctx)
        for (C, R), (a, b, c0, M, N, K) in zip(pairs, hosts):
            assert torch.equal(C, R), (M, N, K)
        a, b, c0, M, N, K = hosts[2]                    # one of them against the oracle
        ok, ratio = og.check(pairs[2][0][:, :N].cpu().numpy(), og.bf16_bits_to_f64(a), og.bf16_bits_to_f64(b))
        assert ok, ratio
    finally:
        rg.rg_group_destroy(g)
