"""Launches whose last, partial wave runs its tiles as two half-width units each: the bits of the 128x64 tile,
which has no halves (every output is summed over K in the same order), and the oracle's bound."""
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


# (tile, pair, M, N): 1 to 76 tiles beyond whole waves of 152 CTAs (76 pairs), with the tail's second halves
# whole, ragged, a single column and wholly outside N
@pytest.mark.parametrize("tile, pair, M, N", [
    (1, False, 2560, 1024), (1, False, 2560, 1000), (1, False, 2500, 961), (1, False, 2560, 960), (1, False, 10240, 130),
    (1, False, 128 * 153, 128), (1, False, 128 * 228, 72), (2, False, 2560, 2048), (2, False, 2500, 1921),
    (2, False, 2560, 1830), (4, False, 2560, 2048), (4, False, 2600, 2000), (5, False, 5120, 2040), (5, False, 5100, 1900),
    (5, True, 2560, 2048), (5, True, 2500, 1930), (5, True, 2560, 1900), (5, True, 256 * 77, 256), (5, True, 256 * 77 - 200, 140),
])
@pytest.mark.parametrize("K, beta", [(64, 0), (200, 1), (1030, 0)])
def test_half_tail_tiles(rg, ctx, tile, pair, M, N, K, beta):
    ldk, ldn = -(-K // 8) * 8, -(-N // 8) * 8
    a, b = synthetic.operands_bf16(M, ldn, ldk, seed=9)
    A, B = (torch.from_numpy(x.view(np.int16)).cuda().view(torch.bfloat16) for x in (a, b))
    c0 = torch.from_numpy(synthetic.normal_stream_f32(9, 3, M * ldn)).cuda().view(M, ldn)
    C, R = c0.clone(), c0.clone()
    bm, bn = rg.TILES[tile]
    units, p = -(-M // bm) * -(-N // bn), 76 if pair else 152
    assert units > p and 0 < 2 * (units % p) <= p            # the shape has a halved tail
    rg.rg_gemm(ctx, M, N, K, A, ldk, B, ldn, C, ldn, rg.variant(tile, rg.TWO_SM) if pair else rg.variant(tile, 1), beta)
    rg.rg_gemm(ctx, M, N, K, A, ldk, B, ldn, R, ldn, rg.variant(0, 1), beta)
    rg.rg_check(ctx)
    assert torch.equal(C, R)                                 # up to ldc: the columns beyond N as well
    if not beta and K == 200:
        ok, ratio = og.check(C[:, :N].cpu().numpy(), og.bf16_bits_to_f64(a[:, :K]), og.bf16_bits_to_f64(b[:K, :N]))
        assert ok, ratio
