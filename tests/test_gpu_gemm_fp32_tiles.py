"""The FP32 GEMM where the tile rule changes with the number of rows, narrow outputs among them: every
output is the same chain of fused multiply-adds whatever the tile, so the first rows of a large problem and
the same rows alone give the same bits, for every epilogue; and they are right, against a float64 product
(K terms, one rounding each: an error of at most K 2^-24 of the sum of |products|, doubled for the
epilogue's own roundings)."""
import ctypes
import os
import subprocess

import pytest

from gpu_common import engine

pytestmark = pytest.mark.gpu

PROGRAM = r"""
#include "ctd_internal.cuh"
extern "C" void run(int epi, int64_t M, int N, int K, const float* A, const float* B, const float* bias, const float* aux,
                    float* out, float* out2) {
  ctd::gemm_f32(0, epi, M, N, K, A, K, B, bias, aux, N, out, N, out2, N);
}
"""


@pytest.fixture(scope="module")
def run(tmp_path_factory):
    engine()
    from paper_2506_04055_gb300 import buildlib
    d = tmp_path_factory.mktemp("gemm")
    src, so = d / "g.cu", d / "g.so"
    src.write_text(PROGRAM)
    subprocess.run([buildlib.nvcc(), *buildlib.ARCH, "-O1", "-std=c++17", "-Xcompiler", "-fPIC", "-shared", "-cudart", "shared",
                    "-I", buildlib.SRC, str(src), buildlib.OUT, "-o", str(so),
                    "-Xlinker", "-rpath," + os.path.dirname(buildlib.OUT) + ":/usr/local/cuda/lib64"], check=True)
    lib = ctypes.CDLL(str(so))
    P, I = ctypes.c_void_p, ctypes.c_int
    lib.run.argtypes = [I, ctypes.c_int64, I, I, P, P, P, P, P, P]
    lib.run.restype = None
    return lib.run


@pytest.mark.parametrize("N,K", [(4, 8), (16, 32), (24, 64), (28, 64), (32, 64), (32, 96), (32, 192), (32, 512), (32, 768), (64, 192),
                                 (96, 32), (128, 128), (128, 256), (128, 384), (256, 768)])
@pytest.mark.parametrize("epi", [0, 1, 2, 3, 4])
def test_rows_do_not_depend_on_the_tile(run, epi, N, K):
    import torch
    most = 80000
    g = torch.Generator(device="cuda").manual_seed(100 * N + K)
    rnd = lambda *s: torch.randn(*s, generator=g, device="cuda")
    A, B, bias, aux, arg = rnd(most, K), rnd(K, N) / K ** 0.5, rnd(N), rnd(most, N), rnd(most, N)

    def product(M):
        out = torch.zeros(M, N, device="cuda")
        out2 = torch.zeros(M, N, device="cuda") if epi == 1 else arg
        torch.cuda.synchronize()
        run(epi, M, N, K, A.data_ptr(), B.data_ptr(), bias.data_ptr() if epi < 2 else None, aux.data_ptr(), out.data_ptr(),
            out2.data_ptr())
        torch.cuda.synchronize()
        return (out, out2) if epi == 1 else (out,)

    whole = product(most)
    if epi in (0, 2):
        extra = bias.double() if epi == 0 else aux.double()
        ref, size = A.double() @ B.double() + extra, A.double().abs() @ B.double().abs() + extra.abs()
        assert bool(((whole[0].double() - ref).abs() <= 2 * K * 2.0 ** -24 * size).all())
    for M in (1, 15, 17, 700, 1500, 2432, 2433, 4832, 4833, 4865, 9727, 9729, 19457, 30001, 38913, 45003, 58369, 77824, 77825):
        for a, b in zip(product(M), whole):
            assert torch.equal(a, b[:M]), M
