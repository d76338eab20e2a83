"""Grouped calls of one group whose kernel families change from call to call, over more calls than it has slots: every
slot's work list, and the enabled nodes of its graph, are then reused by calls of other families.  Every result is bitwise
rg_gemm's, and no call touches another's outputs."""
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


def test_families_change_between_calls(rg, ctx):
    # tile, split (2SM: a pair), by family
    kinds = [rg.variant(0, 1), rg.variant(1, 2), rg.variant(2, 1), rg.variant(3, 1), rg.variant(4, (rg.TWO_SM, 1)),
             rg.variant(5, (rg.TWO_SM, 2)), rg.variant(6, 1), rg.variant(7, 1)]
    calls = [(0, 1), (1, 2, 4), (0,), (0, 3), (5,), (5, 6, 7), (1,), (3, 4), (2,), (0, 1, 2, 3, 4, 5, 6, 7), (0,), (7, 4),
             (3,), (1, 0), (6, 2), (4,), (5, 0), (2, 3), (1,), (6, 7, 0)]
    rs = np.random.default_rng(12)
    g = rg.rg_group_create(ctx, 1, 8, 64 << 20)
    try:
        done, keep = [], []
        for c, families in enumerate(calls):
            probs = []
            for f in families:
                for _ in range(int(rs.integers(1, 4))):
                    M, N, K = (int(rs.integers(1, 90)) * 8 for _ in range(3))
                    a, b = synthetic.operands_bf16(M, N, K, seed=100 + len(done))
                    A, B = (torch.from_numpy(x.view(np.int16)).cuda().view(torch.bfloat16) for x in (a, b))
                    C, R = (torch.full((M, N), float("nan"), device="cuda") for _ in range(2))
                    rg.rg_gemm(ctx, M, N, K, A, K, B, N, R, N, kinds[f])
                    probs.append((M, N, K, A, K, B, N, C, N, 0, 0, 0, 0, kinds[f]))
                    done.append((c, f, C, R))
                    keep.append((A, B))
            torch.cuda.synchronize()
            rg.rg_gemm_grouped(g, probs)
        rg.rg_check(ctx)
        for c, f, C, R in done:
            assert torch.equal(C, R), (c, f)
        # the same calls' outputs, cleared: later calls of other families leave them alone
        for _, _, C, _ in done:
            C.fill_(3.0)
        A, B = keep[0]
        M, K, N = A.shape[0], A.shape[1], B.shape[1]
        last = [torch.full((M, N), float("nan"), device="cuda") for _ in range(9)]
        for i, C in enumerate(last):  # every slot once more, with one family or two
            more = [(M, N, K, A, K, B, N, C, N, 0, 0, 0, 0, kinds[i % 3])]
            extra = torch.empty_like(C)
            rg.rg_gemm_grouped(g, more + [(M, N, K, A, K, B, N, extra, N, 0, 0, 0, 0, kinds[3])] * (i % 2))
        rg.rg_check(ctx)
        assert all(bool((C == 3.0).all()) for _, _, C, _ in done)
        assert all(bool(torch.isfinite(C).all()) for C in last)
    finally:
        rg.rg_group_destroy(g)
