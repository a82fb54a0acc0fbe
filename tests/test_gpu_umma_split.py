"""The BF16 GEMM with its columns shared by several CTAs (few row tiles), at the row counts where the
share changes, against a float64 product: BF16 products are exact in FP32 and only the FP32
accumulation rounds, so the error is bounded by K 2^-23 of the sum of |products|; and the same rows
give the same bits whatever the share."""
import ctypes

import pytest

from gpu_common import engine

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,K", [(128, 128), (384, 128), (96, 64), (32, 96), (512, 64)])
def test_column_shares(N, K):
    import torch
    eng = engine()
    from paper_2506_04055_gb300 import _lib
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    g = torch.Generator(device="cpu").manual_seed(N + K)
    tiles = sorted({1, 2} | {sms // s + d for s in range(1, N // 32 + 1) for d in (0, 1)})
    rows = [t * 128 for t in tiles] + [t * 128 - 1 for t in tiles]
    A = torch.randn(max(rows), K, generator=g).to(torch.bfloat16).cuda()
    B = torch.randn(N, K, generator=g).to(torch.bfloat16).cuda()
    ref = A.double() @ B.double().T
    bound = (A.double().abs() @ B.double().abs().T) * (K * 2.0 ** -23) + 1e-30
    P = lambda t: ctypes.c_void_p(t.data_ptr())
    whole = None
    with eng.Potential(64, T=1, n_species=1) as pot:
        for M in sorted(rows, reverse=True):
            C = torch.zeros(M, N, dtype=torch.float32, device="cuda")
            torch.cuda.synchronize()
            _lib.ctd_gemm_bf16(pot.ctx, M, N, K, P(A), K, P(B), P(C), N)
            assert bool(((C.double() - ref[:M]).abs() <= bound[:M]).all()), M
            whole = C if whole is None else whole
            assert torch.equal(C, whole[:M]), M
