"""rg_gemm_plan_host on pinned operands whose rows are not one block of memory: the rows are copied in by 16-, 4- or
2-byte loads, by the row starts' alignment, and the result is the device path's bit for bit."""
from __future__ import annotations

import numpy as np
import pytest

import synthetic

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    from paper_2605_29752_gb300 import rg
    c = rg.rg_init(0)
    yield c
    rg.rg_destroy(c)


def _pinned_rows(bits, ld):
    buf = torch.zeros((bits.shape[0], ld), dtype=torch.int16).pin_memory()
    buf[:, : bits.shape[1]] = torch.from_numpy(bits.view(np.int16))
    return buf


# (M, N, K, extra of A's rows, extra of B's rows): odd rows (2-byte loads), even (4), multiples of eight in a wider
# buffer (16); one row, one column, and more columns than one batch of a row's threads
@pytest.mark.parametrize("case", [(1, 1, 1, 0, 0), (3, 130, 129, 0, 0), (300, 255, 1025, 0, 0), (257, 254, 130, 0, 0),
                                  (130, 128, 264, 8, 16), (64, 1031, 2050, 1, 0), (5, 8, 16, 8, 8)])
def test_pinned_rows(ctx, case):
    from paper_2605_29752_gb300 import rg
    M, N, K, xa, xb = case
    a_bits, b_bits = synthetic.operands_bf16(M, N, K, seed=7)
    a, b = _pinned_rows(a_bits, K + xa), _pinned_rows(b_bits, N + xb)
    c = torch.full((M, N), float("nan")).pin_memory()
    up = lambda x, m: (x + m - 1) // m * m  # noqa: E731
    grid = rg.make_grid(*((up(x, 128), up(x, 128), 1) for x in (M, N, K)))
    plan = rg.rg_plan_build(grid, np.ones((1, 1), np.int64), [rg.variant(1, 1)])
    try:
        rg.rg_gemm_plan_host(ctx, plan, M, N, K, a, K + xa, b, N + xb, c, N)
        la, lb = up(K, 8), up(N, 8)
        A, B = torch.zeros((M, la), dtype=torch.int16), torch.zeros((K, lb), dtype=torch.int16)
        A[:, :K], B[:, :N] = torch.from_numpy(a_bits.view(np.int16)), torch.from_numpy(b_bits.view(np.int16))
        A, B = A.cuda().view(torch.bfloat16), B.cuda().view(torch.bfloat16)
        C = torch.full((M, lb), float("nan"), device="cuda")
        rg.rg_gemm_plan(ctx, plan, M, N, K, A, la, B, lb, C, lb)
        rg.rg_check(ctx)
        assert torch.equal(C.cpu()[:, :N], c)
    finally:
        rg.rg_plan_free(plan)
