"""The quantiser on what the stream's previous kernel has just written, both launched without a wait in between (the
quantiser may start before that kernel has ended): the codes of the finished values, for vector and element loads."""
import numpy as np
import pytest

import synthetic

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


# Q's leading dimension odd: X is read element by element; a multiple of 4: by vectors but for the ragged right edge
@pytest.mark.parametrize("M, N, ldq", [(1000, 131, 131), (1000, 131, 132), (640, 515, 515), (256, 512, 512)])
def test_quantize_what_a_gemm_writes(M, N, ldq):
    from paper_2605_29752_gb300 import rg
    ctx = rg.rg_init(0)
    try:
        K, ldn, ldc = 512, -(-N // 8) * 8, -(-N // 4) * 4
        pairs = []
        for seed in range(3):
            a, b = synthetic.operands_bf16(M, ldn, K, seed=30 + seed)
            pairs.append([torch.from_numpy(x.view(np.int16)).cuda().view(torch.bfloat16) for x in (a, b)])
        C = torch.zeros((M, ldc), device="cuda")
        blocks = (-(-M // 128), -(-N // 128))

        def outputs():
            return torch.zeros((M, ldq), dtype=torch.uint8, device="cuda"), torch.zeros(blocks, device="cuda")
        got = [outputs() for _ in range(12)]
        torch.cuda.synchronize()
        for i, (q, s) in enumerate(got):
            A, B = pairs[i % 3]
            rg.rg_gemm(ctx, M, N, K, A, K, B, ldn, C, ldc, rg.variant(1, 1))
            rg.rg_fp8_quantize(ctx, C, M, N, ldc, q, ldq, s)
        rg.rg_check(ctx)
        for i, (q, s) in enumerate(got):
            A, B = pairs[i % 3]
            rg.rg_gemm(ctx, M, N, K, A, K, B, ldn, C, ldc, rg.variant(1, 1))
            rg.rg_check(ctx)
            want, scales = outputs()
            torch.cuda.synchronize()
            rg.rg_fp8_quantize(ctx, C, M, N, ldc, want, ldq, scales)
            rg.rg_check(ctx)
            assert torch.equal(q, want) and torch.equal(s, scales), i
    finally:
        rg.rg_destroy(ctx)
