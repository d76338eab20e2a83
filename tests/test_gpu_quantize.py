"""The block quantiser over the alignments, strides and ragged edges that choose between its 16-byte and
its element-wise accesses, and over non-finite input: codes and scales bit-exact against the oracle."""
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


def _run(rg, ctx, x, ldx, x_off, ldq, q_off):
    """x quantised from row stride ldx, x_off floats into a buffer, to row stride ldq, q_off bytes in; the
    bytes around the result must stay as they were."""
    R, N = x.shape
    X = torch.full((x_off + R * ldx + 8,), float("nan"), device="cuda")
    Q = torch.full((q_off + R * ldq + 8,), 0xA5, dtype=torch.uint8, device="cuda")
    X[x_off:x_off + R * ldx].view(R, ldx)[:, :N] = torch.from_numpy(x).cuda()
    S = torch.zeros((-(-R // 128), -(-N // 128)), device="cuda")
    rg.rg_fp8_quantize(ctx, X.data_ptr() + 4 * x_off, R, N, ldx, Q.data_ptr() + q_off, ldq, S)
    rg.rg_check(ctx)
    q = Q.cpu().numpy()
    body = q[q_off:q_off + R * ldq].reshape(R, ldq)
    assert np.all(q[:q_off] == 0xA5) and np.all(q[q_off + R * ldq:] == 0xA5) and np.all(body[:, N:] == 0xA5)
    return body[:, :N], S.cpu().numpy()


@pytest.mark.parametrize("R, N, ldx, x_off, ldq, q_off", [
    (129, 132, 132, 0, 132, 0),        # vector accesses, one row and four columns past a block
    (127, 130, 132, 0, 132, 0),        # a ragged last group of two columns inside a vector row
    (255, 257, 260, 4, 272, 4),        # offsets that keep the alignment
    (130, 131, 131, 0, 131, 0),        # odd strides
    (64, 256, 256, 1, 256, 0),         # X one element off 16 bytes
    (64, 256, 256, 0, 256, 2),         # Q two bytes off four
    (3, 1, 1, 0, 1, 0),                # one column
    (3200, 3200, 3204, 4, 3208, 4),    # more whole blocks than two waves of 512-thread CTAs: the 256-thread kernel
    (3201, 3204, 3204, 0, 3204, 0),    # as many, ragged
])
def test_quantizer_alignments_and_edges(rg, ctx, R, N, ldx, x_off, ldq, q_off):
    x = (synthetic.normal_stream_f32(3, 1, R * N) * np.exp2(synthetic.uniform24(3, 2, R * N) * 60 - 30)).astype(
        np.float32).reshape(R, N)
    q_ref, s_ref = of.quantize_blocks(x)
    q, s = _run(rg, ctx, x, ldx, x_off, ldq, q_off)
    assert np.array_equal(s, s_ref) and np.array_equal(q, q_ref)


@pytest.mark.parametrize("x_off", [0, 1])
def test_quantizer_non_finite(rg, ctx, x_off):
    """amax passes over NaN, whose codes are NaN; an infinite amax makes the scale infinite, the finite
    values' codes zero of their sign and the infinite ones NaN."""
    x = synthetic.normal_stream_f32(5, 1, 128 * 384).reshape(128, 384)
    x[7, 9] = x[100, 120] = np.nan
    x[3, 130] = np.inf
    x[:, 256:] = np.nan
    q, s = _run(rg, ctx, x, 384, x_off, 384, 0)
    first = np.where(np.isnan(x[:, :128]), np.float32(0), x[:, :128])
    q_ref, s_ref = of.quantize_blocks(first)
    q_ref[np.isnan(x[:, :128])] = 0x7F
    assert np.array_equal(q[:, :128], q_ref) and s[0, 0] == s_ref[0, 0]
    mid = x[:, 128:256]
    assert np.isinf(s[0, 1])
    assert np.array_equal(q[:, 128:256], np.where(np.isinf(mid), 0x7F, np.where(np.signbit(mid), 0x80, 0)))
    assert s[0, 2] == 1.0 and np.all(q[:, 256:] == 0x7F)


@pytest.mark.parametrize("exp", [0, 3, 99, 101, -99, -101, -130, -142])
def test_quantizer_at_rounding_boundaries(rg, ctx, exp):
    """Quotients on, and a few units in the last place around, every midpoint and value of e4m3, for scales that
    are and are not powers of two and on both sides of the range in which no division is made."""
    grid = np.unique(np.abs(of.e4m3_decode(np.arange(0x7F, dtype=np.uint8))))
    marks = np.concatenate([grid, (grid[1:] + grid[:-1]) / 2])
    blocks = []
    for m in (1.0, 1.1, 1.7, 1.9999999):
        amax = np.float32(np.ldexp(448.0 * m, exp))
        s = np.float32(amax / np.float32(448.0))
        at = (marks * np.float64(s)).astype(np.float32)
        near = np.concatenate([at] + [at * np.float32(1 + d * 2.0 ** -23) for d in (-9, -5, -3, -1, 1, 3, 5, 9)])
        near = np.minimum(near, amax)
        near = np.resize(np.concatenate([near, -near]), 128 * 128)
        near[-1] = amax
        blocks.append(near.reshape(128, 128))
    x = np.concatenate(blocks, axis=1)
    q_ref, s_ref = of.quantize_blocks(x)
    q, s = _run(rg, ctx, x, 512, 0, 512, 0)
    assert np.array_equal(s, s_ref) and np.array_equal(q, q_ref)
