"""The fused epilogues of the BF16 GEMM by themselves, through a small library linked to the engine's:
the same rows give the same bits whatever the number of CTAs that share a row tile's columns, and
SiLU' of the residual epilogue is as accurate as FP32 exponential and division make it."""
import ctypes
import os
import subprocess

import pytest

from gpu_common import engine

pytestmark = pytest.mark.gpu

PROGRAM = r"""
#include "ctd_internal.cuh"
using namespace ctd;
#define RUN(E)                                                                                              \
  case E: return gemm_bf16<E>(0, M, N, K, (const __nv_bfloat16*)A, K, (const __nv_bfloat16*)W, bias, aux, ldaux, out, \
                              ldo, (__nv_bfloat16*)outb, ldob, status, (__half*)outh, aux2, (const __half*)auxh);
extern "C" int run(int epi, int64_t M, int N, int K, const void* A, const void* W, const float* bias, const float* aux,
                   int ldaux, float* out, int ldo, void* outb, int ldob, int* status, void* outh, const float* aux2,
                   const void* auxh) {
  switch (epi) { RUN(0) RUN(1) RUN(2) RUN(3) RUN(4) RUN(5) RUN(6) RUN(7) }
  return -1;
}
"""


@pytest.fixture(scope="module")
def run(tmp_path_factory):
    engine()
    from paper_2506_04055_gb300 import buildlib
    d = tmp_path_factory.mktemp("epi")
    src, so = d / "epi.cu", d / "epi.so"
    src.write_text(PROGRAM)
    subprocess.run([buildlib.nvcc(), *buildlib.ARCH, "-O1", "-std=c++17", "-Xcompiler", "-fPIC", "-shared", "-cudart", "shared",
                    "-I", buildlib.SRC, str(src), buildlib.OUT, "-o", str(so),
                    "-Xlinker", "-rpath," + os.path.dirname(buildlib.OUT) + ":/usr/local/cuda/lib64"], check=True)
    lib = ctypes.CDLL(str(so))
    P, I, L = ctypes.c_void_p, ctypes.c_int, ctypes.c_int64
    lib.run.argtypes = [I, L, I, I, P, P, P, P, I, P, I, P, I, P, P, P, P]
    lib.run.restype = I
    return lib.run


def _call(run, epi, M, N, K, A, W, bias=None, aux=None, out=None, outb=None, outh=None, aux2=None, auxh=None, ldaux=0):
    import torch
    p = lambda t: None if t is None else t.data_ptr()
    status = torch.zeros(4, dtype=torch.int32, device="cuda")
    ldo = 6 * (N // 3) if epi == 4 else N
    torch.cuda.synchronize()
    assert run(epi, M, N, K, p(A), p(W), p(bias), p(aux), ldaux, p(out), ldo, p(outb), N, p(status), p(outh), p(aux2), p(auxh)) == 0
    torch.cuda.synchronize()
    assert int(status[0]) == 0


@pytest.mark.parametrize("epi,N,K", [(0, 384, 128), (1, 128, 256), (1, 64, 64), (2, 64, 64), (2, 128, 256), (3, 128, 64),
                                     (4, 384, 128), (4, 192, 64), (5, 128, 256), (5, 64, 128), (6, 128, 384), (7, 64, 64),
                                     (7, 128, 64)])
def test_column_shares_leave_the_bits(run, epi, N, K):
    import torch
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    rt = 126 if epi == 5 else 128
    most = (sms + 1) * rt
    g = torch.Generator(device="cuda").manual_seed(epi * 1000 + N)
    rnd = lambda *s: torch.randn(*s, generator=g, device="cuda")
    A, W = rnd(most, K).bfloat16(), (rnd(N, K) / K ** 0.5).bfloat16()
    bias = rnd(N) if epi in (0, 1, 4) else None
    aux = rnd(most, N) if epi in (2, 3, 4, 5, 7) else None   # PHI packing: v is [M][3F] and N = 3F
    aux2 = rnd(most // 3, N) if epi == 5 else rnd(most, N) if epi == 7 else None
    auxh = rnd(most, N).half() if epi == 6 else None

    def outputs(M):
        o = {}
        if epi == 5:
            o["out"] = torch.zeros(M // 3, N, 4, device="cuda")
        elif epi == 4:
            o["out"], o["outh"] = torch.zeros(M, 2 * N, device="cuda"), torch.zeros(M, 2 * N, device="cuda").half()
        else:
            o["out"] = torch.zeros(M, N, device="cuda")
            if epi:
                o["outb"] = torch.zeros(M, N, device="cuda").bfloat16()
            if epi < 2:
                o["outh"] = torch.zeros(M, N, device="cuda").half()
        _call(run, epi, M, N, K, A, W, bias, aux, aux2=aux2, auxh=auxh, ldaux=N if epi > 1 else 0, **o)
        return o

    whole = outputs(most)   # more row tiles than SMs: one CTA per tile
    assert all(bool(torch.isfinite(t.float()).all()) and float(t.float().abs().max()) > 0 for t in whole.values())
    for tiles in sorted({1, 2, 3} | {sms // s + d for s in range(1, N // 32 + 1) for d in (0, 1)}):
        for M in (tiles * rt, tiles * rt - 3):
            for k, t in outputs(M).items():
                assert torch.equal(t, whole[k][:t.shape[0]]), (M, k)


@pytest.mark.parametrize("M", [300, 40000])
def test_silu_derivative_of_the_residual_epilogue(run, M):
    """A = 0 and aux = 1 leave SiLU'(z) itself.  With s = 1 / (1 + exp(-z)): expf within 1 ulp and a rounded sum
    and division give s a relative error of 2^-22; z (1 - s), 1 + z (1 - s) and the last product round once each."""
    import torch
    N = K = 64
    z = torch.linspace(-80.0, 80.0, M * N, device="cuda").reshape(M, N).contiguous()
    A, W = torch.zeros(M, K, device="cuda").bfloat16(), torch.zeros(N, K, device="cuda").bfloat16()
    out = torch.zeros(M, N, device="cuda")
    _call(run, 7, M, N, K, A, W, aux=torch.ones(M, N, device="cuda"), aux2=z, out=out, ldaux=N)
    x = z.double()
    s = torch.sigmoid(x)
    u = x * torch.sigmoid(-x)
    bound = s * ((1 + u).abs() * (2.0 ** -22 + 2.0 ** -23) + x.abs() * (s * 2.0 ** -22 + 2.0 ** -23)) * (1 + 2.0 ** -20)
    err = (out.double() - s * (1 + u)).abs()
    assert bool((err <= bound + 1e-37).all()), float((err / (bound + 1e-37)).max())
