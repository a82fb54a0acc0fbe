// edge_fp32.cu -- the message step and its adjoint over the active edges in FP32 on CUDA cores
// (every width of the FP32 path; F = 64 of the BF16 path, whose edge step stays in FP32).
//
// The message function is PaiNN's (arXiv 2506.04055, Methods "Graph Neural Networks" message
// equation, "Chosen Architectures"): W_e = (Wf rbf(d_e) + bf) f_c(d_e) per edge and channel, an
// [3F x K] contraction that is most of the work of an edge, so the kernels are bound by the FMA
// pipes, by issue and by the latency that few register-heavy warps leave open.  What they are built
// around:
//   * A warp takes a receiver's (adjoint: sender's) row alone, two channels per lane (rows wider than
//     64 channels are shared by F / 64 warps), so the row's sums need no atomics, and the geometry,
//     the row bookkeeping and the reduction over the features are paid once for 64 channels.  A
//     thread's two channels are one operand of the packed f32x2 instructions (FFMA2 has FFMA's
//     arithmetic rate at half its issue slots: measured 1.9 against 3.9 warp instructions per clock
//     and SM); in the contraction a packed instruction takes a pair of centres instead, even and odd
//     centres being added at the end.
//   * The Gaussians whose terms are lost in the rounding are not visited.  The basis is ordered by its
//     centres: every edge takes the last three (K > 20: four) groups of four centres, their weights in
//     registers, in one straight run of independent chains; an edge takes an earlier group, its
//     weights in shared memory, only if one of its centres lies within the layer's reach of the
//     distance: 6.3 widths or more, worked out from the weights (gauss_reach.h) so that in every channel
//     and at every distance the terms left out add up to at most 2^-26 of the largest one kept, where
//     FP32 rounds that one to 2^-24.  Weights of one scale give 6.6 to 7.1 widths (K = 20 centres
//     over a 5 A cutoff: 14 of 20 centres on average in water and in fcc crystals); far weights that
//     dwarf the near ones a longer reach, up to every Gaussian that FP32 can tell from zero.  The
//     branch is uniform over the warp.
//   * The cutoff is folded into the staged basis (b_k f_c, and its distance derivative for the
//     adjoint), so the contraction gives W and dW/dd themselves.
//   * The 32 lanes of a warp stage the next 32 edges at once, across the rows of a chunk of
//     consecutive rows; an edge's gathered rows are loaded one edge ahead, into two sets of registers
//     in turn.
//   * First layer (L0): v = 0, so the psi channels and W_vv are neither gathered nor formed, and
//     the adjoint forms only dW_s, W_vs and dW_vs.
// What bounds them: operand reads.  FFMA2 with three register operands takes 2.5 cycles of a scheduler
// (two FFMA without a reused operand 3.6), and each other instruction among them about two, which
// makes the measured 208 (adjoint) and 106 (message) warp instructions per edge at F = 64 107 and 59
// cycles of an SM; taking two edges at once or more warps changes nothing.
// 96,000-atom water, F = 64, per launch: adjoint 1.82 ms (first layer 1.19), message 1.02 (0.67); one
// thread per channel and all 20 centres took 2.76 and 1.41.  32,000-atom fcc, F = 128: 0.80 (0.49) and
// 0.46 (0.29) against 1.26 and 0.68.
// Every sum runs in an order that depends on the row alone (a row's edges in list order, an edge's
// features in a fixed tree), so results do not depend on which rows share a launch.
#include "ctd_internal.cuh"

namespace ctd {
namespace {

__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c) {
  uint64_t r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;"
      : "=l"(r)
      : "l"(reinterpret_cast<uint64_t&>(a)), "l"(reinterpret_cast<uint64_t&>(b)), "l"(reinterpret_cast<uint64_t&>(c)));
  return reinterpret_cast<float2&>(r);
}
__device__ __forceinline__ float2 mul2(float2 a, float2 b) {
  uint64_t r;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(reinterpret_cast<uint64_t&>(a)), "l"(reinterpret_cast<uint64_t&>(b)));
  return reinterpret_cast<float2&>(r);
}
__device__ __forceinline__ float2 zero2() { return make_float2(0.f, 0.f); }
__device__ __forceinline__ float2 lo2(float4 v) { return make_float2(v.x, v.y); }
__device__ __forceinline__ float2 hi2(float4 v) { return make_float2(v.z, v.w); }

// The FPL channels of a thread (one for F = 32, else two).
template <int FPL>
struct FV;
template <>
struct FV<1> {
  float v;
  static __device__ __forceinline__ FV zero() { return {0.f}; }
  static __device__ __forceinline__ FV ld(const float* p) { return {__ldg(p)}; }
  static __device__ __forceinline__ FV pair(float2 x) { return {x.x}; }   // a value held twice
  __device__ __forceinline__ void st(float* p) const { *p = v; }
  __device__ __forceinline__ void st(__nv_bfloat16* p) const { *p = __float2bfloat16_rn(v); }
  __device__ __forceinline__ float sum() const { return v; }
};
template <>
struct FV<2> {
  float2 v;
  static __device__ __forceinline__ FV zero() { return {zero2()}; }
  static __device__ __forceinline__ FV ld(const float* p) { return {__ldg(reinterpret_cast<const float2*>(p))}; }
  static __device__ __forceinline__ FV pair(float2 x) { return {x}; }
  __device__ __forceinline__ void st(float* p) const { *reinterpret_cast<float2*>(p) = v; }
  __device__ __forceinline__ void st(__nv_bfloat16* p) const {
    *reinterpret_cast<__nv_bfloat162*>(p) = __floats2bfloat162_rn(v.x, v.y);
  }
  __device__ __forceinline__ float sum() const { return v.x + v.y; }
};
__device__ __forceinline__ FV<1> fma(FV<1> a, FV<1> b, FV<1> c) { return {fmaf(a.v, b.v, c.v)}; }
__device__ __forceinline__ FV<2> fma(FV<2> a, FV<2> b, FV<2> c) { return {fma2(a.v, b.v, c.v)}; }
__device__ __forceinline__ FV<1> mul(FV<1> a, FV<1> b) { return {a.v * b.v}; }
__device__ __forceinline__ FV<2> mul(FV<2> a, FV<2> b) { return {mul2(a.v, b.v)}; }
__device__ __forceinline__ FV<1> add(FV<1> a, FV<1> b) { return {a.v + b.v}; }
__device__ __forceinline__ FV<2> add(FV<2> a, FV<2> b) { return {make_float2(a.v.x + b.v.x, a.v.y + b.v.y)}; }
// even + odd centres of each of the thread's channels
__device__ __forceinline__ FV<1> fold(const float2 (&a)[1]) { return {a[0].x + a[0].y}; }
__device__ __forceinline__ FV<2> fold(const float2 (&a)[2]) { return {make_float2(a[0].x + a[0].y, a[1].x + a[1].y)}; }

constexpr int kStage = 32;             // edges staged at a time, one per lane
constexpr int kBatch = 8;              // edges whose partials are reduced over the features together
constexpr int kPartStride = 36;        // float4 per edge of a batch (32 lanes, padded: conflict-free)
constexpr int64_t kChunkRows = 8;      // consecutive rows a warp group takes at a time, at most

// How many of the last groups of four centres keep their weights in registers.
template <int KR>
constexpr int reg_groups() { return KR > 20 ? 4 : KR >= 12 ? 3 : KR / 4; }

struct Args {
  int64_t n, nchunks;
  int K, KP;
  float rc, reach;
  int accumulate;
  const int32_t* __restrict__ arow;
  const int32_t* __restrict__ acol;
  const float4* __restrict__ ar;
  const float* __restrict__ PHI;   // [n][6F]
  const float* __restrict__ Wf;    // [3F][KP]
  const float* __restrict__ bf;    // [3F]
  const float *S, *V;              // message step: residuals
  float *SM, *VM;
  __nv_bfloat16* VMb;              // BF16 copy of VM, or null
  const float *Gsm, *Gvm;          // adjoint: the receivers' gradients
  float* GPHI;                     // [n][5F]
  float4* hedge;
  float* wst;                      // stored filters [E][6F]: written (message) or read (adjoint)
};

// An edge's staged scalars: the direction and the cutoff, each twice (the operand of a packed
// instruction over two channels), its column and its first group.
struct __align__(16) EdgeGeo {
  float4 xy;        // (ux, ux, uy, uy)
  float4 zf;        // (uz, uz, f_c, f_c)
  float2 dfc;       // f_c'
  int col, lo;
};

// Floats of an edge's staged basis: an odd number of 16-byte words, so that the lanes' 16-byte
// stores of their own edges fall in distinct banks.
template <int KR, bool GRAD>
constexpr int basis_stride() {
  constexpr int q = (GRAD ? 2 : 1) * KR / 4;
  return 4 * (q % 2 ? q : q + 1);
}

// Stage edge e: direction (negated for the adjoint, where the edge carries the message of its
// reverse), cutoff, basis.  Group g: (b_0..3) f_c, or with GRAD two pairs (b_0, b_1, b_0', b_1') of
// b f_c and its distance derivative.  Columns from K on meet zero weights.
template <int KR, bool GRAD>
__device__ __forceinline__ void stage_edge(const Args& a, float4 r, int col, float sign, EdgeGeo& geo, float* bas) {
  const float d = r.w, id = sign / d, inv_rc = 1.0f / a.rc;
  const float sig = a.rc / (float)(a.K - 1), inv2s2 = 1.0f / (2.0f * sig * sig), inv_s2 = 1.0f / (sig * sig);
  const float fc = 0.5f * (cospif(d * inv_rc) + 1.0f);
  const float dfc = GRAD ? -0.5f * 3.14159265358979f * inv_rc * sinpif(d * inv_rc) : 0.0f;
  const float ux = r.x * id, uy = r.y * id, uz = r.z * id;
  const int first = (int)ceilf((d - a.reach * sig) / sig);
  geo.xy = make_float4(ux, ux, uy, uy);
  geo.zf = make_float4(uz, uz, fc, fc);
  *reinterpret_cast<float4*>(&geo.dfc) =
      make_float4(dfc, dfc, __int_as_float(col), __int_as_float(max(0, min(first, KR - 1)) >> 2));
#pragma unroll
  for (int k = 0; k < KR; k += 4) {
    float v[4], w[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const float t = d - (float)(k + j) * sig;
      const float b = expf(-t * t * inv2s2);
      v[j] = b * fc;
      w[j] = GRAD ? fmaf(-b * t * inv_s2, fc, b * dfc) : 0.0f;
    }
    if (GRAD) {
      *reinterpret_cast<float4*>(bas + 2 * k) = make_float4(v[0], v[1], w[0], w[1]);
      *reinterpret_cast<float4*>(bas + 2 * k + 4) = make_float4(v[2], v[3], w[2], w[3]);
    } else {
      *reinterpret_cast<float4*>(bas + k) = make_float4(v[0], v[1], v[2], v[3]);
    }
  }
}

// row `col` of a table of `bytes` per row
__device__ __forceinline__ const float* row_of(const float* base, int col, uint32_t bytes) {
  return reinterpret_cast<const float*>(reinterpret_cast<const char*>(base) + (uint64_t)(uint32_t)col * bytes);
}

// A chunk of consecutive rows: lane l holds arow[r0 + l].
struct RowChunk {
  int64_t r0;
  int nrows, rp;
  __device__ __forceinline__ RowChunk(const Args& a, int64_t ck, int lane) {
    r0 = ck * a.n / a.nchunks;
    nrows = (int)((ck + 1) * a.n / a.nchunks - r0);
    rp = nrows > 0 ? a.arow[r0 + min(lane, nrows)] : 0;
  }
  __device__ __forceinline__ int at(int k) const { return __shfl_sync(0xffffffffu, rp, k); }
};

// Filter weights of the thread's channels of one block (s, vv or vs): groups NL.. in registers,
// the first NL groups in shared memory as [group][channel of the thread][thread of the row].
template <int KR, int F, int FPL>
struct Filter {
  static constexpr int NG = KR / 4, NL = NG - reg_groups<KR>();
  float2 w[FPL][2 * (NG - NL)];
  FV<FPL> b;
  const float4* low;
  // shared-memory copy of the first NL groups of one block, filled by the whole thread block
  static __device__ __forceinline__ void fill(const Args& a, int row, float4* dst) {
    for (int i = threadIdx.x; i < NL * F; i += blockDim.x) {
      const int g = i / F, c = i % F;   // channel c = FPL * thread + j
      dst[g * F + (c % FPL) * (F / FPL) + c / FPL] = weights(a, row + c, g);
    }
  }
  static __device__ __forceinline__ float4 weights(const Args& a, int row, int g) {
    return 4 * g < a.KP ? *reinterpret_cast<const float4*>(a.Wf + (size_t)row * a.KP + 4 * g) : make_float4(0.f, 0.f, 0.f, 0.f);
  }
  __device__ __forceinline__ void load(const Args& a, int row, int f, const float4* shared) {
#pragma unroll
    for (int c = 0; c < FPL; ++c)
#pragma unroll
      for (int g = NL; g < NG; ++g) {
        const float4 q = weights(a, row + f + c, g);
        w[c][2 * (g - NL)] = lo2(q);
        w[c][2 * (g - NL) + 1] = hi2(q);
      }
    b = FV<FPL>::ld(a.bf + row + f);
    low = shared + f / FPL;
  }
  // weights of group g < NL of the thread's channel c
  __device__ __forceinline__ float4 lower(int g, int c) const { return low[g * F + c * (F / FPL)]; }
};

// x += the products of a group's weights (w0, w1) and basis (b0, b1)
__device__ __forceinline__ void mac(float2& x, float2 w0, float2 w1, float2 b0, float2 b1) {
  x = fma2(w1, b1, fma2(w0, b0, x));
}

// ---------------------------------------------------------------------------- message step
// STORE: also writes, per edge, [W_s | W_vv | W_vs | dW_s | dW_vv | dW_vs] for the adjoint.
template <int KR, int F, int FPL, int W, bool L0, bool STORE>
__global__ __launch_bounds__(32 * W, 1) void k_edge_msg(const __grid_constant__ Args a) {
  using V = FV<FPL>;
  using Fil = Filter<KR, F, FPL>;
  constexpr int NG = KR / 4, NL = Fil::NL, BS = basis_stride<KR, STORE>(), GS = STORE ? 8 : 4, NWR = F / (32 * FPL), groups = W / NWR;
  static_assert(W % NWR == 0, "whole rows per block");
  extern __shared__ float4 edge_smem4[];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, f = (warp % NWR) * 32 * FPL + FPL * lane;
  float4* low = edge_smem4;
  EdgeGeo* geo = reinterpret_cast<EdgeGeo*>(low + 3 * Fil::NL * F) + warp * kStage;
  float* bas = reinterpret_cast<float*>(reinterpret_cast<EdgeGeo*>(low + 3 * Fil::NL * F) + W * kStage) + warp * kStage * BS;
  Fil ws, wv, wx;   // s, vv, vs
  for (int q = 0; q < 3; ++q) Fil::fill(a, q * F, low + q * Fil::NL * F);
  __syncthreads();
  ws.load(a, 0, f, low);
  if (!L0) wv.load(a, F, f, low + Fil::NL * F);
  wx.load(a, 2 * F, f, low + 2 * Fil::NL * F);

  for (int64_t ck = (int64_t)blockIdx.x * groups + warp / NWR; ck < a.nchunks; ck += (int64_t)gridDim.x * groups) {
    const RowChunk C(a, ck, lane);
    if (C.nrows == 0) continue;
    const int e0 = C.at(0), e1 = C.at(C.nrows);
    int k = 0, rend = C.at(1);
    V as = V::zero(), av0 = as, av1 = as, av2 = as;
    auto flush = [&]() {
      const int64_t i = C.r0 + k;
      if (!L0) {
        av0 = add(V::ld(a.V + i * 3 * F + f), av0);
        av1 = add(V::ld(a.V + i * 3 * F + F + f), av1);
        av2 = add(V::ld(a.V + i * 3 * F + 2 * F + f), av2);
      }
      add(V::ld(a.S + i * F + f), as).st(a.SM + i * F + f);
      av0.st(a.VM + i * 3 * F + f);
      av1.st(a.VM + i * 3 * F + F + f);
      av2.st(a.VM + i * 3 * F + 2 * F + f);
      if (a.VMb) {
        av0.st(a.VMb + i * 3 * F + f);
        av1.st(a.VMb + i * 3 * F + F + f);
        av2.st(a.VMb + i * 3 * F + 2 * F + f);
      }
      as = av0 = av1 = av2 = V::zero();
    };
    float4 rn = make_float4(0.f, 0.f, 0.f, 1.f);   // the next stage's edge of this lane
    int cn = 0;
    auto fetch = [&](int e) {
      if (e < e1) { rn = a.ar[e]; cn = a.acol[e]; }
    };
    fetch(e0 + lane);
    for (int c0 = e0; c0 < e1; c0 += kStage) {
      const int cnt = min(kStage, e1 - c0);
      __syncwarp();
      if (lane < cnt) stage_edge<KR, STORE>(a, rn, cn, 1.0f, geo[lane], bas + lane * BS);
      __syncwarp();
      fetch(c0 + kStage + lane);
      struct Row { V p, x, y0, y1, y2; int lo; } ra, rb;   // an edge's gathered values and first group
      auto gather = [&](int t, Row& r) {
        const int2 cl = *reinterpret_cast<const int2*>(&geo[t].col);
        r.lo = cl.y;
        const float* p = row_of(a.PHI + f, cl.x, 24 * F);
        r.p = V::ld(p);
        r.x = V::ld(p + 4 * F);
        if (!L0) { r.y0 = V::ld(p + F); r.y1 = V::ld(p + 2 * F); r.y2 = V::ld(p + 3 * F); }
      };
      auto edge = [&](int t, const Row& r, Row& next) {
        if (t + 1 < cnt) gather(t + 1, next);
        const float4 gxy = geo[t].xy, gzf = geo[t].zf;
        const float* bp = bas + t * BS;
        float2 xs[FPL], xv[FPL], xx[FPL];
#pragma unroll
        for (int c = 0; c < FPL; ++c) xs[c] = xv[c] = xx[c] = zero2();
#pragma unroll
        for (int g = NL; g < NG; ++g) {
          const float4 q = *reinterpret_cast<const float4*>(bp + GS * g);
          const float2 b0 = lo2(q), b1 = STORE ? *reinterpret_cast<const float2*>(bp + GS * g + 4) : hi2(q);
#pragma unroll
          for (int c = 0; c < FPL; ++c) {
            mac(xs[c], ws.w[c][2 * (g - NL)], ws.w[c][2 * (g - NL) + 1], b0, b1);
            if (!L0) mac(xv[c], wv.w[c][2 * (g - NL)], wv.w[c][2 * (g - NL) + 1], b0, b1);
            mac(xx[c], wx.w[c][2 * (g - NL)], wx.w[c][2 * (g - NL) + 1], b0, b1);
          }
        }
#pragma unroll 1
        for (int g = NL - 1; g >= r.lo; --g) {
          const float4 q = *reinterpret_cast<const float4*>(bp + GS * g);
          const float2 b0 = lo2(q), b1 = STORE ? *reinterpret_cast<const float2*>(bp + GS * g + 4) : hi2(q);
#pragma unroll
          for (int c = 0; c < FPL; ++c) {
            const float4 us = ws.lower(g, c), ux = wx.lower(g, c);
            mac(xs[c], lo2(us), hi2(us), b0, b1);
            if (!L0) {
              const float4 uv = wv.lower(g, c);
              mac(xv[c], lo2(uv), hi2(uv), b0, b1);
            }
            mac(xx[c], lo2(ux), hi2(ux), b0, b1);
          }
        }
        const V fc = V::pair(hi2(gzf));
        const V Ws = fma(ws.b, fc, fold(xs)), Wx = fma(wx.b, fc, fold(xx));
        const V Wv = L0 ? V::zero() : fma(wv.b, fc, fold(xv));
        if constexpr (STORE) {
          const V dfc = V::pair(geo[t].dfc);
          float2 ds[FPL], dv[FPL], dx[FPL];
#pragma unroll
          for (int c = 0; c < FPL; ++c) ds[c] = dv[c] = dx[c] = zero2();
#pragma unroll
          for (int g = 0; g < NG; ++g) {
            const float2 b0 = *reinterpret_cast<const float2*>(bp + GS * g + 2);
            const float2 b1 = *reinterpret_cast<const float2*>(bp + GS * g + 6);
#pragma unroll
            for (int c = 0; c < FPL; ++c) {
              if (g < NL) {
                const float4 us = ws.lower(g, c), uv = wv.lower(g, c), ux = wx.lower(g, c);
                mac(ds[c], lo2(us), hi2(us), b0, b1);
                mac(dv[c], lo2(uv), hi2(uv), b0, b1);
                mac(dx[c], lo2(ux), hi2(ux), b0, b1);
              } else {
                mac(ds[c], ws.w[c][2 * (g - NL)], ws.w[c][2 * (g - NL) + 1], b0, b1);
                mac(dv[c], wv.w[c][2 * (g - NL)], wv.w[c][2 * (g - NL) + 1], b0, b1);
                mac(dx[c], wx.w[c][2 * (g - NL)], wx.w[c][2 * (g - NL) + 1], b0, b1);
              }
            }
          }
          float* o = a.wst + (int64_t)(c0 + t) * 6 * F + f;
          Ws.st(o); Wv.st(o + F); Wx.st(o + 2 * F);
          fma(ws.b, dfc, fold(ds)).st(o + 3 * F);
          fma(wv.b, dfc, fold(dv)).st(o + 4 * F);
          fma(wx.b, dfc, fold(dx)).st(o + 5 * F);
        }
        as = fma(r.p, Ws, as);
        const V tx = mul(r.x, Wx);
        av0 = fma(V::pair(lo2(gxy)), tx, av0);
        av1 = fma(V::pair(hi2(gxy)), tx, av1);
        av2 = fma(V::pair(lo2(gzf)), tx, av2);
        if (!L0) {
          av0 = fma(r.y0, Wv, av0);
          av1 = fma(r.y1, Wv, av1);
          av2 = fma(r.y2, Wv, av2);
        }
      };
      gather(0, ra);
      for (int t = 0; t < cnt;) {
        while (c0 + t == rend) {
          flush();
          rend = C.at(++k + 1);
        }
        const int tend = min(cnt, rend - c0);
#pragma unroll 1
        for (; t + 2 <= tend; t += 2) {
          edge(t, ra, rb);
          edge(t + 1, rb, ra);
        }
        if (t < tend) {
          edge(t++, ra, rb);
          ra = rb;
        }
      }
    }
    for (; k < C.nrows; ++k) flush();
  }
}

// ---------------------------------------------------------------------------- adjoint
// Sender-side: row j holds the edges e' = (j <- i); the reverse (i <- j) carried phi_j, v_j into
// receiver i with direction -u_e'.  Per edge the partials of dU/dd and dU/du of a thread's
// channels go to shared memory and are summed over the features eight edges at a time (four lanes
// per edge, eight 16-byte reads and two shuffle steps each), then turned into
// hedge[e'] = dU/dr_(i<-j), 32 edges at a time.
// STORED: the filter and its distance derivative are read from wst (the message step of the same
// edge list wrote them; an edge's distance equals its reverse's).
template <int KR, int F, int FPL, int W, bool L0, bool STORED>
__global__ __launch_bounds__(32 * W, 1) void k_edge_adj(const __grid_constant__ Args a) {
  using V = FV<FPL>;
  using Fil = Filter<KR, F, FPL>;
  constexpr int NG = KR / 4, NL = Fil::NL, BS = STORED ? 4 : basis_stride<KR, true>(), NWR = F / (32 * FPL), groups = W / NWR;
  constexpr int NLOW = STORED ? 0 : 3 * Fil::NL * F;
  static_assert(W % NWR == 0, "whole rows per block");
  extern __shared__ float4 edge_smem4[];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, wir = warp % NWR, f = wir * 32 * FPL + FPL * lane;
  float4* low = edge_smem4;
  float4* part = low + NLOW + warp * kBatch * kPartStride;
  float4* red = low + NLOW + W * kBatch * kPartStride + (warp - wir) * 2 * kStage;   // [2][kStage][NWR] per group
  EdgeGeo* geo0 = reinterpret_cast<EdgeGeo*>(low + NLOW + W * (kBatch * kPartStride + 2 * kStage));
  EdgeGeo* geo = geo0 + warp * kStage;
  float* bas = reinterpret_cast<float*>(geo0 + W * kStage) + warp * kStage * BS;
  Fil ws, wv, wx;
  if constexpr (!STORED) {
    for (int q = 0; q < 3; ++q) Fil::fill(a, q * F, low + q * Fil::NL * F);
    __syncthreads();
    ws.load(a, 0, f, low);
    if (!L0) wv.load(a, F, f, low + Fil::NL * F);
    wx.load(a, 2 * F, f, low + 2 * Fil::NL * F);
  }
  int buf = 0;

  for (int64_t ck = (int64_t)blockIdx.x * groups + warp / NWR; ck < a.nchunks; ck += (int64_t)gridDim.x * groups) {
    const RowChunk C(a, ck, lane);
    if (C.nrows == 0) continue;
    const int e0 = C.at(0), e1 = C.at(C.nrows);
    int k = 0, rend = C.at(1);
    V ps, pvs, y0, y1, y2, gps, gy0, gy1, gy2, gpvs;
    auto begin = [&]() {
      const float* p = a.PHI + (C.r0 + k) * 6 * F + f;
      ps = V::ld(p);
      pvs = V::ld(p + 4 * F);
      if (!L0) { y0 = V::ld(p + F); y1 = V::ld(p + 2 * F); y2 = V::ld(p + 3 * F); }
      gps = gy0 = gy1 = gy2 = gpvs = V::zero();
    };
    auto flush = [&]() {
      if (L0) return;   // the first layer's inputs do not depend on positions
      float* o = a.GPHI + (C.r0 + k) * 5 * F + f;
      gps.st(o); gy0.st(o + F); gy1.st(o + 2 * F); gy2.st(o + 3 * F); gpvs.st(o + 4 * F);
    };
    begin();
    float4 rn = make_float4(0.f, 0.f, 0.f, 1.f);   // the next stage's edge of this lane
    int cn = 0;
    auto fetch = [&](int e) {
      if (e < e1) { rn = a.ar[e]; cn = a.acol[e]; }
    };
    fetch(e0 + lane);
    for (int c0 = e0; c0 < e1; c0 += kStage, buf ^= 1) {
      const int cnt = min(kStage, e1 - c0);
      __syncwarp();
      if (lane < cnt) stage_edge<STORED ? 0 : KR, true>(a, rn, cn, -1.0f, geo[lane], bas + lane * BS);
      __syncwarp();
      const float dist = rn.w;   // of the edge this lane finishes
      fetch(c0 + kStage + lane);
      struct Row { V s, v0, v1, v2; int lo; } ra, rb;   // an edge's gathered values and first group
      auto gather = [&](int t, Row& r) {
        const int2 cl = *reinterpret_cast<const int2*>(&geo[t].col);
        r.lo = cl.y;
        r.s = V::ld(row_of(a.Gsm + f, cl.x, 4 * F));
        const float* p = row_of(a.Gvm + f, cl.x, 12 * F);
        r.v0 = V::ld(p); r.v1 = V::ld(p + F); r.v2 = V::ld(p + 2 * F);
      };
      // the feature sums of the batch that ends at edge t (inclusive)
      auto reduce = [&](int t) {
        __syncwarp();
        const int b = lane >> 2, p = lane & 3, base = t & ~(kBatch - 1);
        const float4* src = part + b * kPartStride + 8 * p;
        float4 s = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
        for (int i = 0; i < 8; ++i) {
          const float4 v = src[(i + p) & 7];
          s.x += v.x; s.y += v.y; s.z += v.z; s.w += v.w;
        }
#pragma unroll
        for (int o = 1; o < 4; o <<= 1) {
          s.x += __shfl_xor_sync(0xffffffffu, s.x, o);
          s.y += __shfl_xor_sync(0xffffffffu, s.y, o);
          s.z += __shfl_xor_sync(0xffffffffu, s.z, o);
          s.w += __shfl_xor_sync(0xffffffffu, s.w, o);
        }
        if (p == 0) red[(buf * kStage + base + b) * NWR + wir] = s;
        __syncwarp();
      };
      auto edge = [&](int t, const Row& r, Row& next) {
        if (t + 1 < cnt) gather(t + 1, next);
        const float4 gxy = geo[t].xy, gzf = geo[t].zf;
        V Ws, Wv, Wx, Ds, Dv, Dx;
        if constexpr (STORED) {
          const float* w = a.wst + (int64_t)(c0 + t) * 6 * F + f;
          Ws = V::ld(w); Wv = V::ld(w + F); Wx = V::ld(w + 2 * F);
          Ds = V::ld(w + 3 * F); Dv = V::ld(w + 4 * F); Dx = V::ld(w + 5 * F);
        } else {
          const float* bp = bas + t * BS;
          float2 xs[FPL], xv[FPL], xx[FPL], ds[FPL], dv[FPL], dx[FPL];
#pragma unroll
          for (int c = 0; c < FPL; ++c) xs[c] = xv[c] = xx[c] = ds[c] = dv[c] = dx[c] = zero2();
#pragma unroll
          for (int g = NL; g < NG; ++g) {
            const float4 b0 = *reinterpret_cast<const float4*>(bp + 8 * g);
            const float4 b1 = *reinterpret_cast<const float4*>(bp + 8 * g + 4);
#pragma unroll
            for (int c = 0; c < FPL; ++c) {
              const float2 s0 = ws.w[c][2 * (g - NL)], s1 = ws.w[c][2 * (g - NL) + 1];
              const float2 u0 = wx.w[c][2 * (g - NL)], u1 = wx.w[c][2 * (g - NL) + 1];
              if (!L0) mac(xs[c], s0, s1, lo2(b0), lo2(b1));
              mac(ds[c], s0, s1, hi2(b0), hi2(b1));
              if (!L0) {
                const float2 v0 = wv.w[c][2 * (g - NL)], v1 = wv.w[c][2 * (g - NL) + 1];
                mac(xv[c], v0, v1, lo2(b0), lo2(b1));
                mac(dv[c], v0, v1, hi2(b0), hi2(b1));
              }
              mac(xx[c], u0, u1, lo2(b0), lo2(b1));
              mac(dx[c], u0, u1, hi2(b0), hi2(b1));
            }
          }
#pragma unroll 1
          for (int g = NL - 1; g >= r.lo; --g) {
            const float4 b0 = *reinterpret_cast<const float4*>(bp + 8 * g);
            const float4 b1 = *reinterpret_cast<const float4*>(bp + 8 * g + 4);
#pragma unroll
            for (int c = 0; c < FPL; ++c) {
              const float4 us = ws.lower(g, c), ux = wx.lower(g, c);
              if (!L0) mac(xs[c], lo2(us), hi2(us), lo2(b0), lo2(b1));
              mac(ds[c], lo2(us), hi2(us), hi2(b0), hi2(b1));
              if (!L0) {
                const float4 uv = wv.lower(g, c);
                mac(xv[c], lo2(uv), hi2(uv), lo2(b0), lo2(b1));
                mac(dv[c], lo2(uv), hi2(uv), hi2(b0), hi2(b1));
              }
              mac(xx[c], lo2(ux), hi2(ux), lo2(b0), lo2(b1));
              mac(dx[c], lo2(ux), hi2(ux), hi2(b0), hi2(b1));
            }
          }
          const V fc = V::pair(hi2(gzf)), dfc = V::pair(geo[t].dfc);
          Ds = fma(ws.b, dfc, fold(ds));
          Wx = fma(wx.b, fc, fold(xx));
          Dx = fma(wx.b, dfc, fold(dx));
          if (!L0) {
            Ws = fma(ws.b, fc, fold(xs));
            Wv = fma(wv.b, fc, fold(xv));
            Dv = fma(wv.b, dfc, fold(dv));
          }
        }
        // the staged direction is that of the reverse edge, -u
        const V qv = fma(r.v2, V::pair(lo2(gzf)), fma(r.v1, V::pair(hi2(gxy)), mul(r.v0, V::pair(lo2(gxy)))));
        V pd = fma(mul(qv, pvs), Dx, mul(mul(r.s, ps), Ds));
        if (!L0) {
          gps = fma(r.s, Ws, gps);
          gy0 = fma(r.v0, Wv, gy0);
          gy1 = fma(r.v1, Wv, gy1);
          gy2 = fma(r.v2, Wv, gy2);
          gpvs = fma(qv, Wx, gpvs);
          pd = fma(fma(r.v2, y2, fma(r.v1, y1, mul(r.v0, y0))), Dv, pd);
        }
        const V tv = mul(pvs, Wx);
        part[(t & (kBatch - 1)) * kPartStride + lane] =
            make_float4(pd.sum(), mul(r.v0, tv).sum(), mul(r.v1, tv).sum(), mul(r.v2, tv).sum());
        if ((t & (kBatch - 1)) == kBatch - 1) reduce(t);
      };
      gather(0, ra);
      for (int t = 0; t < cnt;) {
        while (c0 + t == rend) {
          flush();
          rend = C.at(++k + 1);
          begin();
        }
        const int tend = min(cnt, rend - c0);
#pragma unroll 1
        for (; t + 2 <= tend; t += 2) {
          edge(t, ra, rb);
          edge(t + 1, rb, ra);
        }
        if (t < tend) {
          edge(t++, ra, rb);
          ra = rb;
        }
      }
      if (cnt & (kBatch - 1)) reduce(cnt - 1);
      // the group's warps have written their sums; the buffer alternates, so one barrier per stage
      // separates a buffer's reads from its next writes
      if (NWR > 1) asm volatile("bar.sync %0, %1;" ::"r"(1 + warp / NWR), "n"(32 * NWR) : "memory");
      if (wir == 0 && lane < cnt) {
        float4 s = red[(buf * kStage + lane) * NWR];
#pragma unroll
        for (int w = 1; w < NWR; ++w) {
          const float4 o = red[(buf * kStage + lane) * NWR + w];
          s.x += o.x; s.y += o.y; s.z += o.z; s.w += o.w;
        }
        const EdgeGeo& g = geo[lane];
        const float ux = g.xy.x, uy = g.xy.z, uz = g.zf.x, id = 1.0f / dist;
        const float gdu = s.y * ux + s.z * uy + s.w * uz;
        float4 h = make_float4(s.x * ux + (s.y - gdu * ux) * id, s.x * uy + (s.z - gdu * uy) * id,
                               s.x * uz + (s.w - gdu * uz) * id, 0.f);
        if (a.accumulate) {
          const float4 o = a.hedge[c0 + lane];
          h.x += o.x; h.y += o.y; h.z += o.z;
        }
        a.hedge[c0 + lane] = h;
      }
    }
    for (;;) {
      flush();
      if (++k == C.nrows) break;
      begin();
    }
  }
}

// ---------------------------------------------------------------------------- host side
// Warps of a block (one block per SM): what the registers allow, 168 a thread for twelve warps and
// 255 for eight.  Twelve of the wide kernels spill (adjoint, F = 64, 24,000 atoms: 698 us against 455).
template <int KR, int F, int FPL, bool L0>
constexpr int warps() { return (L0 && KR <= 20) || KR <= 8 ? 12 : 8; }
template <int KR, int F, int FPL, int W, bool STORE>
constexpr size_t msg_smem() {
  return sizeof(float4) * 3 * Filter<KR, F, FPL>::NL * F +
         (size_t)W * kStage * (sizeof(float) * basis_stride<KR, STORE>() + sizeof(EdgeGeo));
}
template <int KR, int F, int FPL, int W, bool STORED>
constexpr size_t adj_smem() {
  return (STORED ? 0 : sizeof(float4) * 3 * Filter<KR, F, FPL>::NL * F) +
         (size_t)W * (sizeof(float4) * (kBatch * kPartStride + 2 * kStage) +
                      kStage * (sizeof(EdgeGeo) + sizeof(float) * (STORED ? 4 : basis_stride<KR, true>())));
}

int edge_sms() {
  static const int sms = [] {
    int dev = 0, count = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&count, cudaDevAttrMultiProcessorCount, dev);
    return count > 0 ? count : 152;
  }();
  return sms;
}

// One persistent block per SM; the rows are cut into w chunks of consecutive rows per warp group, taken
// block-cyclically: the groups of an SM work on neighbouring rows, whose gathered rows overlap in
// L1.  Chunks hold at most kChunkRows rows; among the w that allow it the one that leaves no group more
// rows than it must (6,000 rows on 1,216 groups in two chunks are 4 or 6 rows a group, in one 4 or 5:
// adjoint 143 against 121 us).
template <typename Kern>
void launch(cudaStream_t st, Kern kern, int warps, int groups, size_t smem, Args& a) {
  const int64_t blocks = edge_sms(), G = blocks * groups, w0 = (a.n + G * kChunkRows - 1) / (G * kChunkRows);
  int64_t best = 0, most = 0;
  for (int64_t w = w0; w <= 2 * w0; ++w) {
    const int64_t rows = w * ((a.n + G * w - 1) / (G * w));   // of the group with the most
    if (best == 0 || rows <= most) { best = w; most = rows; }
  }
  a.nchunks = G * best;
  cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  LaunchScope ls_(st);
  kern<<<(unsigned)blocks, 32 * warps, smem, st>>>(a);
}

template <int KR, int F, int FPL>
void msg_go(cudaStream_t st, Args& a, bool first) {
  constexpr int NWR = F / (32 * FPL), W = warps<KR, F, FPL, false>(), W0 = warps<KR, F, FPL, true>();
  if (a.wst) launch(st, k_edge_msg<KR, F, FPL, W, false, true>, W, W / NWR, msg_smem<KR, F, FPL, W, true>(), a);
  else if (first) launch(st, k_edge_msg<KR, F, FPL, W0, true, false>, W0, W0 / NWR, msg_smem<KR, F, FPL, W0, false>(), a);
  else launch(st, k_edge_msg<KR, F, FPL, W, false, false>, W, W / NWR, msg_smem<KR, F, FPL, W, false>(), a);
}

template <int KR, int F, int FPL>
void adj_go(cudaStream_t st, Args& a, bool first) {
  constexpr int NWR = F / (32 * FPL), W = warps<KR, F, FPL, false>(), W0 = warps<KR, F, FPL, true>();
  // stored filters: nothing depends on the basis size
  if (a.wst && first) launch(st, k_edge_adj<16, F, FPL, 16, true, true>, 16, 16 / NWR, adj_smem<16, F, FPL, 16, true>(), a);
  else if (a.wst) launch(st, k_edge_adj<16, F, FPL, 16, false, true>, 16, 16 / NWR, adj_smem<16, F, FPL, 16, true>(), a);
  else if (first) launch(st, k_edge_adj<KR, F, FPL, W0, true, false>, W0, W0 / NWR, adj_smem<KR, F, FPL, W0, false>(), a);
  else launch(st, k_edge_adj<KR, F, FPL, W, false, false>, W, W / NWR, adj_smem<KR, F, FPL, W, false>(), a);
}

}  // namespace

#define CTD_WIDTH(GO, KR)                           \
  switch (m.F) {                                    \
    case 32: GO<KR, 32, 1>(st, a, t == 0); break;   \
    case 64: GO<KR, 64, 2>(st, a, t == 0); break;   \
    case 128: GO<KR, 128, 2>(st, a, t == 0); break; \
    default: GO<KR, 256, 2>(st, a, t == 0); break;  \
  }
// Basis sizes are rounded up to 8, 16, 20 or 32 centres.  (K = 4, calls of 20,000-atom water: 2.28 ms at F = 64, 4.75 at
// F = 128; rounded up to 16 centres 2.99 and 5.97, with a thread per channel 2.89 and 5.59.)
#define CTD_DISPATCH(GO)                     \
  if (m.KP <= 8) { CTD_WIDTH(GO, 8) }        \
  else if (m.KP <= 16) { CTD_WIDTH(GO, 16) } \
  else if (m.KP <= 20) { CTD_WIDTH(GO, 20) } \
  else { CTD_WIDTH(GO, 32) }

void edge_msg_f32(cudaStream_t st, const ModelW& m, int t, int64_t n, const int32_t* arow, const int32_t* acol,
                  const float4* ar, const float* PHI, const float* S, const float* V, float* SM, float* VM,
                  __nv_bfloat16* VMb, float* wst) {
  if (n == 0) return;
  Args a{};
  a.n = n; a.K = m.K; a.KP = m.KP; a.rc = m.rc; a.reach = m.L[t].reach; a.arow = arow; a.acol = acol; a.ar = ar; a.PHI = PHI;
  a.Wf = m.L[t].Wf; a.bf = m.L[t].bf; a.S = S; a.V = V; a.SM = SM; a.VM = VM; a.VMb = VMb; a.wst = wst;
  CTD_DISPATCH(msg_go)
}

void edge_adj_f32(cudaStream_t st, const ModelW& m, int t, int accumulate, int64_t n, const int32_t* arow,
                  const int32_t* acol, const float4* ar, const float* PHI, const float* Gsm, const float* Gvm,
                  float* GPHI, float4* hedge, const float* wst) {
  if (n == 0) return;
  Args a{};
  a.n = n; a.K = m.K; a.KP = m.KP; a.rc = m.rc; a.reach = m.L[t].reach; a.accumulate = accumulate; a.arow = arow; a.acol = acol;
  a.ar = ar; a.PHI = PHI; a.Wf = m.L[t].Wf; a.bf = m.L[t].bf; a.Gsm = Gsm; a.Gvm = Gvm; a.GPHI = GPHI;
  a.hedge = hedge; a.wst = const_cast<float*>(wst);
  CTD_DISPATCH(adj_go)
}

}  // namespace ctd
