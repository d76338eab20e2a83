"""FP8 launches whose last or only wave runs its tiles as two half-width units each: the bits of the
256x256 cta_group::2 pair, which has no halves (every output is summed over K in the same order)."""
import numpy as np
import pytest

import synthetic
from oracle import fp8 as of

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


def _quantized(rg, ctx, rows, cols, seed):
    x = torch.from_numpy(synthetic.normal_stream_f32(seed, 1, rows * cols).reshape(rows, cols)).cuda()
    q = torch.zeros((rows, -(-cols // 16) * 16), dtype=torch.uint8, device="cuda")
    s = torch.empty((-(-rows // 128), -(-cols // 128)), device="cuda")
    rg.rg_fp8_quantize(ctx, x, rows, cols, cols, q, q.stride(0), s)
    return q, s


# M, N of 128x256 tiles: one tile, an only wave with room for the halves, 1 to 76 tiles beyond whole waves
# of 152, and second halves whole, ragged, one column and wholly outside N
@pytest.mark.parametrize("M, N", [
    (128, 256), (100, 130), (90, 129), (60, 128), (512, 1536), (2560, 2048), (2500, 1921), (2560, 1920), (2560, 1830),
    (128 * 153, 129), (128 * 228, 256),
])
@pytest.mark.parametrize("K, beta", [(128, 0), (400, 1), (1500, 0)])
def test_half_tiles(rg, ctx, M, N, K, beta):
    tiles = -(-M // 128) * -(-N // 256)
    assert 0 < 2 * (tiles % 152) <= 152                       # the shape has halves
    qa, sa = _quantized(rg, ctx, M, K, 30)
    qb, sb = _quantized(rg, ctx, K, N, 31)
    ldc = -(-N // 4) * 4
    c0 = torch.from_numpy(synthetic.normal_stream_f32(32, 3, M * ldc)).cuda().view(M, ldc)
    C, R = c0.clone(), c0.clone()
    for out, v in ((C, rg.fp8_variant(0, 1)), (R, rg.fp8_variant(rg.FP8_PAIR_TILE, 1))):
        rg.rg_gemm_fp8_ex(ctx, M, N, K, qa, qa.stride(0), sa, sa.stride(0), qb, qb.stride(0), sb, sb.stride(0), out, ldc,
                          v, beta)
    rg.rg_check(ctx)
    assert torch.equal(C, R)
    if not beta and M <= 512:
        a, b = (of.dequantize(q[:, :w].cpu().numpy(), s.cpu().numpy()) for q, s, w in ((qa, sa, K), (qb, sb, N)))
        err = np.abs(C[:, :N].cpu().numpy() - a @ b) / (np.abs(a) @ np.abs(b))
        assert err.max() <= 4 * K * 2.0 ** -24
