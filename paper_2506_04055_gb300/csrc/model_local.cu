// model_local.cu -- the strictly local equivariant edge model (Allegro form, rotation orders
// <= 1), forward and hand-written adjoint, FP32 on CUDA cores.
//
// Methods, "(Semi-)Local Potential Models" and "Chosen Architectures": information moves only
// between directed edges that leave the same atom, so an atom's energy depends on its own
// cutoff sphere alone, whatever the number of layers.  Every quantity lives on an edge
// e = (i -> j) of the active CSR list (row i = the edges leaving atom i, r_e = x_j - x_i):
//   x = silu([b f_c | onehot Z_i | onehot Z_j] A0 + c0)             two-body latent   [E][F]
//   s = (x P0)[0:C], v = (x P0)[C:2C] u                             edge features     [E][C], [E][3][C]
//   layer l: om = x Q_l;  Gs_i = sum_{e from i} f_c om[0:C],  Gv_i = sum f_c om[C:2C] u
//            ts = [s Gs_i | v . Gv_i], tv = [s Gv_i | v Gs_i]        tensor-product paths
//            x = silu([x | ts] M_l + m_l);  (l < L) s = ts Gs_l, v = tv Gv_l
//   E_i = e_scale w_i sum_{e from i} f_c (silu(x R1 + d1) . R2 + d2)
// The dense contractions are GEMMs over edge rows (the FP32 SIMT GEMM of model_fp32.cu); the
// centre sums are one thread per (atom, channel) over its row in a fixed order; everything
// else is one thread per edge or per (edge, channel).  The adjoint reverses each step and ends
// in hedge = -dE/dr_e, from which the shared force kernel assembles forces and virial through
// the reverse-edge index (no atomics anywhere, so results do not depend on the batch).
#include "ctd_internal.cuh"

namespace ctd {
namespace {

constexpr float kPiF = 3.14159265358979323846f;

// Eight FP32 values as one 16-byte store of BF16 (a thread writing its own edge's row: one
// store per 8 columns instead of one per column)
__device__ __forceinline__ void st8_bf16(__nv_bfloat16* p, const float (&v)[8]) {
  uint32_t w[4];
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    const __nv_bfloat162 b = __floats2bfloat162_rn(v[2 * j], v[2 * j + 1]);
    w[j] = *reinterpret_cast<const uint32_t*>(&b);
  }
  *reinterpret_cast<uint4*>(p) = make_uint4(w[0], w[1], w[2], w[3]);
}
__device__ __forceinline__ float4 ld4f(const float* p) { return *reinterpret_cast<const float4*>(p); }
__device__ __forceinline__ void st4_bf16(__nv_bfloat16* p, float4 v) {
  const __nv_bfloat162 a = __floats2bfloat162_rn(v.x, v.y), b = __floats2bfloat162_rn(v.z, v.w);
  *reinterpret_cast<uint2*>(p) = make_uint2(*reinterpret_cast<const uint32_t*>(&a), *reinterpret_cast<const uint32_t*>(&b));
}

// Blocks of eight warps over w rows, at most a few per resident block.
inline unsigned row_blocks(int64_t w, int C) {
  const int64_t b = (w + kThreads / 32 - 1) / (kThreads / 32), most = 152 * 4 * (C == 16 ? 2 : 1);
  return (unsigned)(b < 1 ? 1 : b < most ? b : most);
}
inline unsigned nblocks(int64_t w) { return (unsigned)((w + kThreads - 1) / kThreads); }

// Per-edge and per-atom arrays, carved from one allocation (128-byte aligned pieces).
struct LocalBufs {
  int32_t* erow;                      // [E] row (centre atom) of each edge
  float *geo, *in, *z0, *w0, *zh, *h;  // [E][8] (d, f_c, f_c', u, 0, 0), [E][KA], [E][F], [E][2C], [E][F/2] x2
  float* X[kMaxT + 1];                // [E][F+2C]: x^l in columns 0..F-1, ts of layer l+1 after it
  float *S[kMaxT], *V[kMaxT];         // s^l [E][C], v^l [E][3][C], l = 0..L-1
  float *OM[kMaxT + 1], *Z[kMaxT + 1];  // l = 1..L: [E][2C], [E][F]
  float* TV[kMaxT];                   // l = 1..L-1: [E][3][2C]
  float *gamS[kMaxT + 1], *gamV[kMaxT + 1];  // l = 1..L: [n][C], [n][3][C]
  // adjoint
  float *gzh, *gx, *gxc, *gts, *gtv, *gs[2], *gv[2], *gom, *gw0, *gin, *ggamS, *ggamV;
  float4* gg;                         // [E]: (dE/df_c, dE/du)
  // BF16 path: the tensor-core GEMMs' A operands, rows zero-padded to >= 64 columns
  __nv_bfloat16 *inb, *Xb[kMaxT + 1], *gzhb, *gomb, *gw0b, *gxb;   // [E][KAb], [E][F+2C], [E][Kh], [E][Kc] x2, [E][F]
};

// The one-pass tensor-product kernels are built for these channel counts.
inline bool local_fused(const LocalW& w) { return w.C == 16 || w.C == 32; }

inline int local_kc(const LocalW& w) { return 2 * w.C < 64 ? 64 : 2 * w.C; }   // padded K of 2C-wide gradients

struct Carver {
  float* base;
  int64_t off = 0;
  float* take(int64_t cnt) {
    off = (off + 31) / 32 * 32;
    float* p = base ? base + off : nullptr;
    off += cnt;
    return p;
  }
};

int64_t carve(const LocalW& w, int64_t n, int64_t E, float* base, LocalBufs* b) {
  const int64_t F = w.F, C = w.C, C2 = 2 * w.C, FX = F + C2, Fh = w.F / 2;
  Carver cv{base};
  b->erow = reinterpret_cast<int32_t*>(cv.take(E));
  b->geo = cv.take(E * 8);
  b->in = cv.take(w.bf16 ? 0 : E * w.KA);   // the BF16 path has inb
  b->z0 = cv.take(E * F);
  b->w0 = cv.take(E * C2);
  for (int l = 0; l <= w.L; ++l) b->X[l] = cv.take(E * FX);
  for (int l = 0; l < w.L; ++l) {
    b->S[l] = cv.take(E * C);
    b->V[l] = cv.take(E * 3 * C);
  }
  for (int l = 1; l <= w.L; ++l) {
    b->OM[l] = cv.take(E * C2);
    b->Z[l] = cv.take(E * F);
    b->gamS[l] = cv.take(n * C);
    b->gamV[l] = cv.take(n * 3 * C);
    if (l < w.L) b->TV[l] = cv.take(local_fused(w) ? 0 : E * 3 * C2);
  }
  b->zh = cv.take(E * Fh);
  b->h = cv.take(w.bf16 ? 0 : E * Fh);
  b->gzh = cv.take(w.bf16 ? 0 : E * Fh);
  b->gx = cv.take(E * F);
  b->gxc = cv.take(E * FX);
  b->gts = cv.take(local_fused(w) ? 0 : E * C2);
  b->gtv = cv.take(local_fused(w) ? 0 : E * 3 * C2);
  for (int q = 0; q < 2; ++q) {
    b->gs[q] = cv.take(E * C);
    b->gv[q] = cv.take(E * 3 * C);
  }
  b->gom = cv.take(w.bf16 ? 0 : E * C2);
  b->gw0 = cv.take(w.bf16 ? 0 : E * C2);
  b->gin = cv.take(E * w.KA);
  b->gg = reinterpret_cast<float4*>(cv.take(E * 4));
  b->ggamS = cv.take(n * C);
  b->ggamV = cv.take(n * 3 * C);
  auto tb = [&](int64_t cnt) { return reinterpret_cast<__nv_bfloat16*>(cv.take((cnt + 1) / 2)); };
  if (w.bf16) {
    const int64_t Kc = local_kc(w);
    b->inb = tb(E * w.KAb);
    for (int l = 0; l <= w.L; ++l) b->Xb[l] = tb(E * FX);
    b->gzhb = tb(E * w.Kh);
    b->gomb = tb(E * Kc);
    b->gw0b = tb(E * Kc);
    b->gxb = tb(E * F);
  } else {
    b->inb = b->gzhb = b->gomb = b->gw0b = b->gxb = nullptr;
    for (int l = 0; l <= w.L; ++l) b->Xb[l] = nullptr;
  }
  return cv.off;
}

// ---------------------------------------------------------------------------- forward kernels
__global__ void k_loc_erow(int64_t n, const int32_t* __restrict__ arow, int32_t* __restrict__ erow) {
  const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (i >= n) return;
  for (int32_t e = arow[i]; e < arow[i + 1]; ++e) erow[e] = (int32_t)i;
}

// geo[e] = (d, f_c, f_c', u_x, u_y, u_z, 0, 0); in[e] = [b_k(d) f_c (K) | onehot Z_i | onehot Z_j | 0].
// b_k = exp(-(d - k sigma)^2 / (2 sigma^2)), sigma = rc / (K - 1); f_c = (cos(pi d / rc) + 1) / 2.
// The row goes to in (FP32, KA columns) or, on the BF16 path, to inb (KAb >= KA columns, a multiple of
// 32, zeros after KA).  Four lanes per edge, each over every fourth 16-byte piece of the row: with a
// thread per edge each store touched 32 lines, and the BF16 path also wrote the FP32 row, which
// nothing reads there (96,000 atoms, BF16: 1.40 ms, now 0.31).
__global__ void k_loc_geom(int64_t E, int K, int S, int KA, float rc, const float4* __restrict__ ar,
                           const int32_t* __restrict__ acol, const int32_t* __restrict__ erow,
                           const int32_t* __restrict__ Z, float* __restrict__ geo, float* __restrict__ in,
                           __nv_bfloat16* __restrict__ inb, int KAb) {
  const int64_t t4 = blockIdx.x * (int64_t)blockDim.x + threadIdx.x, e = t4 >> 2;
  const int j = (int)(t4 & 3);
  if (e >= E) return;
  const float4 r = ar[e];
  const float d = sqrtf(r.x * r.x + r.y * r.y + r.z * r.z);
  const float inv = 1.0f / d;
  const float a = kPiF / rc;
  const float fc = 0.5f * (cosf(a * d) + 1.0f);
  if (j == 0) {
    const float dfc = -0.5f * a * sinf(a * d);
    *reinterpret_cast<float4*>(geo + e * 8) = make_float4(d, fc, dfc, r.x * inv);
    *reinterpret_cast<float4*>(geo + e * 8 + 4) = make_float4(r.y * inv, r.z * inv, 0.0f, 0.0f);
  }
  const float sig = rc / (float)(K - 1);
  const float c = 1.0f / (2.0f * sig * sig);
  const int zi = Z[erow[e]], zj = Z[acol[e]];
  const int hi = zi >= 0 && zi < S ? K + zi : -1, hj = zj >= 0 && zj < S ? K + S + zj : -1;
  auto value = [&](int k) {
    const float t = d - (float)k * sig;
    return k < K ? expf(-t * t * c) * fc : (k == hi || k == hj ? 1.0f : 0.0f);
  };
  if (inb) {
    for (int k0 = 8 * j; k0 < KAb; k0 += 32) {
      float v[8];
#pragma unroll
      for (int q = 0; q < 8; ++q) v[q] = value(k0 + q);
      st8_bf16(inb + e * KAb + k0, v);
    }
  } else {
    for (int k0 = 4 * j; k0 < KA; k0 += 16)
      *reinterpret_cast<float4*>(in + e * KA + k0) = make_float4(value(k0), value(k0 + 1), value(k0 + 2), value(k0 + 3));
  }
}

// s[e][c] = w0[e][c], v[e][a][c] = w0[e][C+c] u_a
__global__ void k_loc_init(int64_t E, int C, const float* __restrict__ w0, const float* __restrict__ geo,
                           float* __restrict__ S0, float* __restrict__ V0) {
  const int64_t idx = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (idx >= E * C) return;
  const int64_t e = idx / C;
  const int c = (int)(idx % C);
  const float* g = geo + e * 8;
  const float wv = w0[e * 2 * C + C + c];
  S0[e * C + c] = w0[e * 2 * C + c];
  for (int q = 0; q < 3; ++q) V0[(e * 3 + q) * C + c] = wv * g[3 + q];
}

// Gs[i][c] = sum_{e in row i} f_c om[e][c];  Gv[i][a][c] = sum_{e in row i} f_c om[e][C+c] u_a
__global__ void k_loc_env(int64_t n, int C, const int32_t* __restrict__ arow, const float* __restrict__ geo,
                          const float* __restrict__ om, float* __restrict__ gamS, float* __restrict__ gamV) {
  const int64_t idx = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (idx >= n * C) return;
  const int64_t i = idx / C;
  const int c = (int)(idx % C);
  float gs = 0.0f, gv0 = 0.0f, gv1 = 0.0f, gv2 = 0.0f;
  for (int64_t e = arow[i]; e < arow[i + 1]; ++e) {
    const float* g = geo + e * 8;
    const float fc = g[1];
    gs = fmaf(fc, om[e * 2 * C + c], gs);
    const float t = fc * om[e * 2 * C + C + c];
    gv0 = fmaf(t, g[3], gv0);
    gv1 = fmaf(t, g[4], gv1);
    gv2 = fmaf(t, g[5], gv2);
  }
  gamS[i * C + c] = gs;
  gamV[(i * 3 + 0) * C + c] = gv0;
  gamV[(i * 3 + 1) * C + c] = gv1;
  gamV[(i * 3 + 2) * C + c] = gv2;
}

// ts[e] = [s Gs_i | v . Gv_i] (row stride ld), tv[e][a] = [s Gv_i[a] | v[a] Gs_i] (may be null)
__global__ void k_loc_tp(int64_t E, int C, const int32_t* __restrict__ erow, const float* __restrict__ S,
                         const float* __restrict__ V, const float* __restrict__ gamS, const float* __restrict__ gamV,
                         float* __restrict__ ts, int ld, float* __restrict__ tv, __nv_bfloat16* __restrict__ tsb) {
  const int64_t idx = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (idx >= E * C) return;
  const int64_t e = idx / C;
  const int c = (int)(idx % C);
  const int64_t i = erow[e];
  const float s = S[e * C + c];
  const float v0 = V[(e * 3 + 0) * C + c], v1 = V[(e * 3 + 1) * C + c], v2 = V[(e * 3 + 2) * C + c];
  const float gs = gamS[i * C + c];
  const float g0 = gamV[(i * 3 + 0) * C + c], g1 = gamV[(i * 3 + 1) * C + c], g2 = gamV[(i * 3 + 2) * C + c];
  const float t0 = s * gs, t1 = fmaf(v2, g2, fmaf(v1, g1, v0 * g0));
  ts[e * ld + c] = t0;
  ts[e * ld + C + c] = t1;
  if (tsb) {   // BF16 copy, same row stride
    tsb[e * ld + c] = __float2bfloat16_rn(t0);
    tsb[e * ld + C + c] = __float2bfloat16_rn(t1);
  }
  if (tv) {
    float* t = tv + e * 6 * C;
    t[0 * 2 * C + c] = s * g0;
    t[1 * 2 * C + c] = s * g1;
    t[2 * 2 * C + c] = s * g2;
    t[0 * 2 * C + C + c] = v0 * gs;
    t[1 * 2 * C + C + c] = v1 * gs;
    t[2 * 2 * C + C + c] = v2 * gs;
  }
}

// E_i = e_scale w_i sum_{e in row i} f_c (h_e . R2 + d2), FP64 Neumaier sums per warp; with gradients
// also the adjoint's seed per edge, g = e_scale w_i: gg[e] = (dE/df_c, 0, 0, 0) with dE/df_c = g (h . R2 + d2), and
// g_zh = g f_c R2 silu'(zh) (gzh, or on the BF16 path gzhb, Kh columns).  A warp per row, eight lanes per
// edge: zh is read once (a thread per row for the energies and a warp per edge for the seed took 0.76
// and 1.31 ms at 96,000 atoms, BF16; now 0.53).  H = silu(zh) as stored, or computed here where null.
__global__ void k_loc_readout(int64_t n, int Fh, float e_scale, const int32_t* __restrict__ arow,
                              const float* __restrict__ geo, const float* __restrict__ H,
                              const float* __restrict__ ZH, const float* __restrict__ R2,
                              const float* __restrict__ d2, const float* __restrict__ ew, float* __restrict__ e_atom,
                              double* __restrict__ partials, int need_grad, float* __restrict__ gzh,
                              float4* __restrict__ gg, __nv_bfloat16* __restrict__ gzhb, int Kh) {
  __shared__ double sbuf[kThreads / 32];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, sub = lane >> 3, j = lane & 7;
  double acc = 0.0, comp = 0.0;
  for (int64_t i = (int64_t)blockIdx.x * (kThreads / 32) + w; i < n; i += (int64_t)gridDim.x * (kThreads / 32)) {
    const int r0 = arow[i], r1 = arow[i + 1];
    const float g = ew ? e_scale * ew[i] : e_scale;
    float es = 0.0f;   // of the edges r0 + sub, r0 + sub + 4, ...
    for (int e0 = r0; e0 < r1; e0 += 4) {
      const bool live = e0 + sub < r1;
      const int64_t e = live ? e0 + sub : r0;
      const float fc = geo[e * 8 + 1];
      float y = 0.0f;
      for (int k = 4 * j; k < Fh; k += 32) {
        const float4 q = ld4f((H ? H : ZH) + e * Fh + k), r = ld4f(R2 + k);
        const float4 h = H ? q : make_float4(silu_f(q.x), silu_f(q.y), silu_f(q.z), silu_f(q.w));
        y = fmaf(r.w, h.w, fmaf(r.z, h.z, fmaf(r.y, h.y, fmaf(r.x, h.x, y))));
      }
#pragma unroll
      for (int o = 1; o < 8; o <<= 1) y += __shfl_xor_sync(0xffffffffu, y, o);
      y += d2[0];
      if (live) es = fmaf(fc, y, es);
      if (live && need_grad) {
        if (j == 0) gg[e] = make_float4(g * y, 0.0f, 0.0f, 0.0f);
        const float a = g * fc;
        for (int k = 4 * j; k < (gzhb ? Kh : Fh); k += 32) {
          float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
          if (k < Fh) {
            const float4 z = ld4f(ZH + e * Fh + k), r = ld4f(R2 + k);
            v = make_float4(a * r.x * dsilu_f(z.x), a * r.y * dsilu_f(z.y), a * r.z * dsilu_f(z.z), a * r.w * dsilu_f(z.w));
          }
          if (gzhb) st4_bf16(gzhb + e * Kh + k, v);
          else *reinterpret_cast<float4*>(gzh + e * Fh + k) = v;
        }
      }
    }
    es += __shfl_xor_sync(0xffffffffu, es, 8);
    es += __shfl_xor_sync(0xffffffffu, es, 16);
    es *= e_scale;
    if (ew) es *= ew[i];
    if (lane == 0 && e_atom) e_atom[i] = es;
    const double x = (double)es, t = acc + x;
    comp += fabs(acc) >= fabs(x) ? (acc - t) + x : (x - t) + acc;
    acc = t;
  }
  if (lane == 0) sbuf[w] = acc + comp;
  __syncthreads();
  if (threadIdx.x == 0) {
    double s = 0.0;
    for (int k = 0; k < kThreads / 32; ++k) s += sbuf[k];
    partials[blockIdx.x] = s;
  }
}

// The tensor products and the channel mixings of a layer in one pass over the rows, for C = 16 and 32:
// ts = [s Gs_i | v . Gv_i] (row stride ld, and its BF16 copy), s' = ts Gs, v'_a = [s Gv_i[a] | v_a Gs_i] Gv.
// A warp per row, 32 / C edges at a time, lane = channel; an edge's 8C products are exchanged through
// shared memory, a lane's 4C weights are in registers, the next edges' features are loaded while one
// set is computed.  The separate passes wrote and read the 6C products of v and ran the mixings as
// GEMMs with 16 of 32 columns idle (96,000 atoms, C = 16: 2.1 ms, now 0.94).  The sums run over the
// inputs in order as the GEMM's.
template <int C>
__global__ void __launch_bounds__(kThreads, C == 16 ? 2 : 1) k_loc_tp_mix(
    int64_t n, const int32_t* __restrict__ arow, const float* __restrict__ S, const float* __restrict__ V,
    const float* __restrict__ gamS, const float* __restrict__ gamV, const float* __restrict__ Gs,
    const float* __restrict__ Gv, float* __restrict__ ts, int ld, __nv_bfloat16* __restrict__ tsb, float* __restrict__ So,
    float* __restrict__ Vo) {
  constexpr int HW = 32 / C;
  __shared__ __align__(16) float sm[kThreads / 32][HW][8 * C];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, h = lane / C, c = lane % C;
  float ws[2 * C], wv[2 * C];
#pragma unroll
  for (int k = 0; k < 2 * C; ++k) {
    ws[k] = Gs[k * C + c];
    wv[k] = Gv[k * C + c];
  }
  float* x = sm[w][h];
  for (int64_t i = (int64_t)blockIdx.x * (kThreads / 32) + w; i < n; i += (int64_t)gridDim.x * (kThreads / 32)) {
    const int r0 = arow[i], r1 = arow[i + 1];
    const float gs = gamS[i * C + c];
    const float g0 = gamV[(i * 3 + 0) * C + c], g1 = gamV[(i * 3 + 1) * C + c], g2 = gamV[(i * 3 + 2) * C + c];
    float ns = 0.f, nv0 = 0.f, nv1 = 0.f, nv2 = 0.f;
    auto load = [&](int e0) {
      const int64_t e = min(e0 + h, r1 - 1);   // lanes without an edge repeat the row's last one
      ns = S[e * C + c];
      nv0 = V[(e * 3 + 0) * C + c];
      nv1 = V[(e * 3 + 1) * C + c];
      nv2 = V[(e * 3 + 2) * C + c];
    };
    if (r0 < r1) load(r0);
    for (int e0 = r0; e0 < r1; e0 += HW) {
      const bool live = e0 + h < r1;
      const int64_t e = e0 + h;
      const float s = ns, v0 = nv0, v1 = nv1, v2 = nv2;
      if (e0 + HW < r1) load(e0 + HW);
      const float t0 = s * gs, t1 = fmaf(v2, g2, fmaf(v1, g1, v0 * g0));
      if (live) {
        ts[e * ld + c] = t0;
        ts[e * ld + C + c] = t1;
        if (tsb) {
          tsb[e * ld + c] = __float2bfloat16_rn(t0);
          tsb[e * ld + C + c] = __float2bfloat16_rn(t1);
        }
      }
      __syncwarp();   // the previous edges' products have been read
      x[c] = t0;
      x[C + c] = t1;
      x[2 * C + c] = s * g0;
      x[3 * C + c] = v0 * gs;
      x[4 * C + c] = s * g1;
      x[5 * C + c] = v1 * gs;
      x[6 * C + c] = s * g2;
      x[7 * C + c] = v2 * gs;
      __syncwarp();
      float o[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
      for (int k = 0; k < 2 * C; k += 4)
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          const float4 y = *reinterpret_cast<const float4*>(x + q * 2 * C + k);
          const float* u = q == 0 ? ws : wv;
          o[q] = fmaf(y.w, u[k + 3], fmaf(y.z, u[k + 2], fmaf(y.y, u[k + 1], fmaf(y.x, u[k], o[q]))));
        }
      if (live) {
        So[e * C + c] = o[0];
        Vo[(e * 3 + 0) * C + c] = o[1];
        Vo[(e * 3 + 1) * C + c] = o[2];
        Vo[(e * 3 + 2) * C + c] = o[3];
      }
    }
  }
}

// ---------------------------------------------------------------------------- adjoint kernels
// The tensor-product adjoint of a layer in one pass over the rows, for C = 16 and 32.  MIX (a layer that
// feeds another): the channel mixings' adjoint comes first, g_ts = g_s Gs^T + g_x's part (gts), g_tv = g_v Gv^T.
// Edge side: g_s = g_ts0 Gs + g_tv0 . Gv, g_v[a] = g_ts1 Gv[a] + g_tv1[a] Gs; centre side:
// g_Gs_i = sum_e (g_ts0 s + g_tv1 . v), g_Gv_i[a] = sum_e (g_ts1 v[a] + g_tv0[a] s).
// A warp per row, 32 / C edges at a time, lane = channel; the incoming gradients are exchanged
// through shared memory, the next edges' values loaded while one set is computed.  The separate passes
// read g_ts and g_tv twice and wrote g_tv (96,000 atoms, C = 16, with the GEMMs: 3.3 ms for a layer that
// mixes and 1.4 for one that does not, now 1.01 and 0.60).
template <int C, bool MIX>
__global__ void __launch_bounds__(kThreads, C == 16 ? 2 : 1) k_loc_tp_bwd(
    int64_t n, const int32_t* __restrict__ arow, const float* __restrict__ S, const float* __restrict__ V,
    const float* __restrict__ gamS, const float* __restrict__ gamV, const float* __restrict__ gts, int ldg,
    const float* __restrict__ gsi, const float* __restrict__ gvi, const float* __restrict__ Gst,
    const float* __restrict__ Gvt, float* __restrict__ GS, float* __restrict__ GV, float* __restrict__ ggamS,
    float* __restrict__ ggamV) {
  constexpr int HW = 32 / C;
  __shared__ __align__(16) float sm[kThreads / 32][HW][4 * C];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, h = lane / C, c = lane % C;
  float u0[MIX ? C : 1], u1[MIX ? C : 1], w0[MIX ? C : 1], w1[MIX ? C : 1];   // columns c and C + c of Gs^T, Gv^T
  if (MIX)
#pragma unroll
    for (int k = 0; k < C; ++k) {
      u0[k] = Gst[k * 2 * C + c];
      u1[k] = Gst[k * 2 * C + C + c];
      w0[k] = Gvt[k * 2 * C + c];
      w1[k] = Gvt[k * 2 * C + C + c];
    }
  float* x = sm[w][h];
  struct In { float a0, a1, s, v[3], g[4]; };
  for (int64_t i = (int64_t)blockIdx.x * (kThreads / 32) + w; i < n; i += (int64_t)gridDim.x * (kThreads / 32)) {
    const int r0 = arow[i], r1 = arow[i + 1];
    const float gs = gamS[i * C + c];
    const float g0 = gamV[(i * 3 + 0) * C + c], g1 = gamV[(i * 3 + 1) * C + c], g2 = gamV[(i * 3 + 2) * C + c];
    float qs = 0.f, q0 = 0.f, q1 = 0.f, q2 = 0.f;
    auto load = [&](int e0, In& in) {
      const int64_t e = min(e0 + h, r1 - 1);   // lanes without an edge repeat the row's last one
      in.a0 = gts[e * ldg + c];
      in.a1 = gts[e * ldg + C + c];
      in.s = S[e * C + c];
#pragma unroll
      for (int q = 0; q < 3; ++q) in.v[q] = V[(e * 3 + q) * C + c];
      if (MIX) {
        in.g[0] = gsi[e * C + c];
#pragma unroll
        for (int q = 0; q < 3; ++q) in.g[1 + q] = gvi[(e * 3 + q) * C + c];
      }
    };
    In nx;
    if (r0 < r1) load(r0, nx);
    for (int e0 = r0; e0 < r1; e0 += HW) {
      In in = nx;
      if (MIX) {
        __syncwarp();
#pragma unroll
        for (int q = 0; q < 4; ++q) x[q * C + c] = in.g[q];
        __syncwarp();
      }
      if (e0 + HW < r1) load(e0 + HW, nx);
      float t0[3] = {0.f, 0.f, 0.f}, t1[3] = {0.f, 0.f, 0.f};
      if (MIX) {
        float b0 = 0.f, b1 = 0.f;
#pragma unroll
        for (int k = 0; k < C; k += 4) {
          const float4 y = *reinterpret_cast<const float4*>(x + k);
          b0 = fmaf(y.w, u0[k + 3], fmaf(y.z, u0[k + 2], fmaf(y.y, u0[k + 1], fmaf(y.x, u0[k], b0))));
          b1 = fmaf(y.w, u1[k + 3], fmaf(y.z, u1[k + 2], fmaf(y.y, u1[k + 1], fmaf(y.x, u1[k], b1))));
#pragma unroll
          for (int q = 0; q < 3; ++q) {
            const float4 z = *reinterpret_cast<const float4*>(x + (1 + q) * C + k);
            t0[q] = fmaf(z.w, w0[k + 3], fmaf(z.z, w0[k + 2], fmaf(z.y, w0[k + 1], fmaf(z.x, w0[k], t0[q]))));
            t1[q] = fmaf(z.w, w1[k + 3], fmaf(z.z, w1[k + 2], fmaf(z.y, w1[k + 1], fmaf(z.x, w1[k], t1[q]))));
          }
        }
        in.a0 = b0 + in.a0;
        in.a1 = b1 + in.a1;
      }
      const float a0 = in.a0, a1 = in.a1;
      if (e0 + h < r1) {
        const int64_t e = e0 + h;
        float s = a0 * gs, v0 = a1 * g0, v1 = a1 * g1, v2 = a1 * g2;
        qs = fmaf(a0, in.s, qs);
        q0 = fmaf(a1, in.v[0], q0);
        q1 = fmaf(a1, in.v[1], q1);
        q2 = fmaf(a1, in.v[2], q2);
        if (MIX) {
          s = fmaf(t0[2], g2, fmaf(t0[1], g1, fmaf(t0[0], g0, s)));
          v0 = fmaf(t1[0], gs, v0);
          v1 = fmaf(t1[1], gs, v1);
          v2 = fmaf(t1[2], gs, v2);
          qs = fmaf(t1[2], in.v[2], fmaf(t1[1], in.v[1], fmaf(t1[0], in.v[0], qs)));
          q0 = fmaf(t0[0], in.s, q0);
          q1 = fmaf(t0[1], in.s, q1);
          q2 = fmaf(t0[2], in.s, q2);
        }
        GS[e * C + c] = s;
        GV[(e * 3 + 0) * C + c] = v0;
        GV[(e * 3 + 1) * C + c] = v1;
        GV[(e * 3 + 2) * C + c] = v2;
      }
    }
    if (HW == 2) {   // even and odd edges of the row
      qs += __shfl_xor_sync(0xffffffffu, qs, 16);
      q0 += __shfl_xor_sync(0xffffffffu, q0, 16);
      q1 += __shfl_xor_sync(0xffffffffu, q1, 16);
      q2 += __shfl_xor_sync(0xffffffffu, q2, 16);
    }
    if (h == 0) {
      ggamS[i * C + c] = qs;
      ggamV[(i * 3 + 0) * C + c] = q0;
      ggamV[(i * 3 + 1) * C + c] = q1;
      ggamV[(i * 3 + 2) * C + c] = q2;
    }
  }
}

// The same in separate passes, for other channel counts.  Edge side: g_s = g_ts0 Gs + g_tv0 . Gv, g_v[a] = g_ts1 Gv[a] + g_tv1[a] Gs.
__global__ void k_loc_tp_bwd_edge(int64_t E, int C, const int32_t* __restrict__ erow, const float* __restrict__ gamS,
                                  const float* __restrict__ gamV, const float* __restrict__ gts, int ldg,
                                  const float* __restrict__ gtv, float* __restrict__ GS, float* __restrict__ GV) {
  const int64_t idx = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (idx >= E * C) return;
  const int64_t e = idx / C;
  const int c = (int)(idx % C);
  const int64_t i = erow[e];
  const float a0 = gts[e * ldg + c], a1 = gts[e * ldg + C + c];
  const float gs = gamS[i * C + c];
  const float g0 = gamV[(i * 3 + 0) * C + c], g1 = gamV[(i * 3 + 1) * C + c], g2 = gamV[(i * 3 + 2) * C + c];
  float s = a0 * gs, v0 = a1 * g0, v1 = a1 * g1, v2 = a1 * g2;
  if (gtv) {
    const float* t = gtv + e * 6 * C;
    s = fmaf(t[0 * 2 * C + c], g0, s);
    s = fmaf(t[1 * 2 * C + c], g1, s);
    s = fmaf(t[2 * 2 * C + c], g2, s);
    v0 = fmaf(t[0 * 2 * C + C + c], gs, v0);
    v1 = fmaf(t[1 * 2 * C + C + c], gs, v1);
    v2 = fmaf(t[2 * 2 * C + C + c], gs, v2);
  }
  GS[e * C + c] = s;
  GV[(e * 3 + 0) * C + c] = v0;
  GV[(e * 3 + 1) * C + c] = v1;
  GV[(e * 3 + 2) * C + c] = v2;
}

// Centre side: g_Gs_i = sum_e (g_ts0 s + g_tv1 . v), g_Gv_i[a] = sum_e (g_ts1 v[a] + g_tv0[a] s).
__global__ void k_loc_tp_bwd_atom(int64_t n, int C, const int32_t* __restrict__ arow, const float* __restrict__ S,
                                  const float* __restrict__ V, const float* __restrict__ gts, int ldg,
                                  const float* __restrict__ gtv, float* __restrict__ ggamS, float* __restrict__ ggamV) {
  const int64_t idx = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (idx >= n * C) return;
  const int64_t i = idx / C;
  const int c = (int)(idx % C);
  float gs = 0.0f, g0 = 0.0f, g1 = 0.0f, g2 = 0.0f;
  for (int64_t e = arow[i]; e < arow[i + 1]; ++e) {
    const float s = S[e * C + c];
    const float v0 = V[(e * 3 + 0) * C + c], v1 = V[(e * 3 + 1) * C + c], v2 = V[(e * 3 + 2) * C + c];
    const float a0 = gts[e * ldg + c], a1 = gts[e * ldg + C + c];
    gs = fmaf(a0, s, gs);
    g0 = fmaf(a1, v0, g0);
    g1 = fmaf(a1, v1, g1);
    g2 = fmaf(a1, v2, g2);
    if (gtv) {
      const float* t = gtv + e * 6 * C;
      gs = fmaf(t[0 * 2 * C + C + c], v0, gs);
      gs = fmaf(t[1 * 2 * C + C + c], v1, gs);
      gs = fmaf(t[2 * 2 * C + C + c], v2, gs);
      g0 = fmaf(t[0 * 2 * C + c], s, g0);
      g1 = fmaf(t[1 * 2 * C + c], s, g1);
      g2 = fmaf(t[2 * 2 * C + c], s, g2);
    }
  }
  ggamS[i * C + c] = gs;
  ggamV[(i * 3 + 0) * C + c] = g0;
  ggamV[(i * 3 + 1) * C + c] = g1;
  ggamV[(i * 3 + 2) * C + c] = g2;
}

// Environment sums, reversed: g_om[c] = f_c g_Gs[c], g_om[C+c] = f_c (g_Gv[c] . u);
// dE/df_c += om[c] g_Gs[c] + om[C+c] (g_Gv[c] . u);  dE/du += f_c om[C+c] g_Gv[c].
// Four lanes per edge, each over channel quads j, j + 4, ... (16-byte accesses; C a multiple of 4,
// of 16 when gomb is written), the sums over channels by two shuffle steps in a fixed order.  The
// BF16 path writes only the GEMM's BF16 operand gomb.
__global__ void k_loc_env_bwd(int64_t E, int C, const int32_t* __restrict__ erow, const float* __restrict__ geo,
                              const float* __restrict__ om, const float* __restrict__ ggamS,
                              const float* __restrict__ ggamV, float* __restrict__ gom, float4* __restrict__ gg,
                              __nv_bfloat16* __restrict__ gomb, int Kc) {
  const int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  const int64_t e = t >> 2;
  const int j = (int)(t & 3);
  const bool live = e < E;
  const int64_t es = live ? e : 0;
  const int64_t i = erow[es];
  const float* g = geo + es * 8;
  const float fc = g[1], u0 = g[3], u1 = g[4], u2 = g[5];
  float gfc = 0.0f, gu0 = 0.0f, gu1 = 0.0f, gu2 = 0.0f;
  for (int c = 4 * j; live && c < C; c += 16) {
    const float4 gs = ld4f(ggamS + i * C + c);
    const float4 q0 = ld4f(ggamV + (i * 3 + 0) * C + c), q1 = ld4f(ggamV + (i * 3 + 1) * C + c),
                 q2 = ld4f(ggamV + (i * 3 + 2) * C + c);
    const float4 o0 = ld4f(om + es * 2 * C + c), o1 = ld4f(om + es * 2 * C + C + c);
    float4 va, vb;
    auto one = [&](float s_, float a0, float a1, float a2, float p0, float p1, float& ra, float& rb) {
      const float gd = fmaf(a2, u2, fmaf(a1, u1, a0 * u0));
      ra = fc * s_;
      rb = fc * gd;
      gfc = fmaf(p0, s_, fmaf(p1, gd, gfc));
      const float tt = fc * p1;
      gu0 = fmaf(tt, a0, gu0);
      gu1 = fmaf(tt, a1, gu1);
      gu2 = fmaf(tt, a2, gu2);
    };
    one(gs.x, q0.x, q1.x, q2.x, o0.x, o1.x, va.x, vb.x);
    one(gs.y, q0.y, q1.y, q2.y, o0.y, o1.y, va.y, vb.y);
    one(gs.z, q0.z, q1.z, q2.z, o0.z, o1.z, va.z, vb.z);
    one(gs.w, q0.w, q1.w, q2.w, o0.w, o1.w, va.w, vb.w);
    if (gomb) {
      st4_bf16(gomb + es * Kc + c, va);
      st4_bf16(gomb + es * Kc + C + c, vb);
    } else {
      *reinterpret_cast<float4*>(gom + es * 2 * C + c) = va;
      *reinterpret_cast<float4*>(gom + es * 2 * C + C + c) = vb;
    }
  }
  if (live && gomb)
    for (int k = 2 * C + 4 * j; k < Kc; k += 16) st4_bf16(gomb + es * Kc + k, make_float4(0.f, 0.f, 0.f, 0.f));
  // the four lanes of an edge are consecutive lanes of one warp (t & 3)
#pragma unroll
  for (int o = 1; o < 4; o <<= 1) {
    gfc += __shfl_xor_sync(0xffffffffu, gfc, o);
    gu0 += __shfl_xor_sync(0xffffffffu, gu0, o);
    gu1 += __shfl_xor_sync(0xffffffffu, gu1, o);
    gu2 += __shfl_xor_sync(0xffffffffu, gu2, o);
  }
  if (live && j == 0) {
    float4 a = gg[e];
    a.x += gfc; a.y += gu0; a.z += gu1; a.w += gu2;
    gg[e] = a;
  }
}

// Initial features, reversed: g_w0[c] = g_s[c], g_w0[C+c] = g_v[c] . u;  dE/du += w0[C+c] g_v[c].
// Four lanes per edge over channel quads, as k_loc_env_bwd.
__global__ void k_loc_init_bwd(int64_t E, int C, const float* __restrict__ w0, const float* __restrict__ geo,
                               const float* __restrict__ GS, const float* __restrict__ GV, float* __restrict__ gw0,
                               float4* __restrict__ gg, __nv_bfloat16* __restrict__ gw0b, int Kc) {
  const int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  const int64_t e = t >> 2;
  const int j = (int)(t & 3);
  const bool live = e < E;
  const int64_t es = live ? e : 0;
  const float* g = geo + es * 8;
  const float u0 = g[3], u1 = g[4], u2 = g[5];
  float gu0 = 0.0f, gu1 = 0.0f, gu2 = 0.0f;
  for (int c = 4 * j; live && c < C; c += 16) {
    const float4 q0 = ld4f(GV + (es * 3 + 0) * C + c), q1 = ld4f(GV + (es * 3 + 1) * C + c),
                 q2 = ld4f(GV + (es * 3 + 2) * C + c);
    const float4 va = ld4f(GS + es * C + c), wv = ld4f(w0 + es * 2 * C + C + c);
    const float4 vb = make_float4(fmaf(q2.x, u2, fmaf(q1.x, u1, q0.x * u0)), fmaf(q2.y, u2, fmaf(q1.y, u1, q0.y * u0)),
                                  fmaf(q2.z, u2, fmaf(q1.z, u1, q0.z * u0)), fmaf(q2.w, u2, fmaf(q1.w, u1, q0.w * u0)));
    if (gw0b) {
      st4_bf16(gw0b + es * Kc + c, va);
      st4_bf16(gw0b + es * Kc + C + c, vb);
    } else {
      *reinterpret_cast<float4*>(gw0 + es * 2 * C + c) = va;
      *reinterpret_cast<float4*>(gw0 + es * 2 * C + C + c) = vb;
    }
    gu0 = fmaf(wv.w, q0.w, fmaf(wv.z, q0.z, fmaf(wv.y, q0.y, fmaf(wv.x, q0.x, gu0))));
    gu1 = fmaf(wv.w, q1.w, fmaf(wv.z, q1.z, fmaf(wv.y, q1.y, fmaf(wv.x, q1.x, gu1))));
    gu2 = fmaf(wv.w, q2.w, fmaf(wv.z, q2.z, fmaf(wv.y, q2.y, fmaf(wv.x, q2.x, gu2))));
  }
  if (live && gw0b)
    for (int k = 2 * C + 4 * j; k < Kc; k += 16) st4_bf16(gw0b + es * Kc + k, make_float4(0.f, 0.f, 0.f, 0.f));
#pragma unroll
  for (int o = 1; o < 4; o <<= 1) {
    gu0 += __shfl_xor_sync(0xffffffffu, gu0, o);
    gu1 += __shfl_xor_sync(0xffffffffu, gu1, o);
    gu2 += __shfl_xor_sync(0xffffffffu, gu2, o);
  }
  if (live && j == 0) {
    float4 a = gg[e];
    a.y += gu0; a.z += gu1; a.w += gu2;
    gg[e] = a;
  }
}

// Geometry, reversed: dE/dd = sum_k g_in[k] (b_k' f_c + b_k f_c') + (dE/df_c) f_c';
// dE/dr = dE/dd u + (dE/du - (dE/du . u) u) / d;  hedge = -dE/dr.
__global__ void k_loc_geom_bwd(int64_t E, int K, float rc, const float* __restrict__ geo, const float* __restrict__ gin,
                               int KA, const float4* __restrict__ gg, float4* __restrict__ hedge) {
  const int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (e >= E) return;
  const float* g = geo + e * 8;
  const float d = g[0], fc = g[1], dfc = g[2], u0 = g[3], u1 = g[4], u2 = g[5];
  const float sig = rc / (float)(K - 1);
  const float c = 1.0f / (2.0f * sig * sig);
  float gd = 0.0f;
  for (int k = 0; k < K; ++k) {
    const float t = d - (float)k * sig;
    const float b = expf(-t * t * c);
    const float db = b * (-2.0f * c * t);
    gd = fmaf(gin[e * KA + k], fmaf(db, fc, b * dfc), gd);
  }
  const float4 a = gg[e];
  gd = fmaf(a.x, dfc, gd);
  const float gu = fmaf(a.w, u2, fmaf(a.z, u1, a.y * u0));
  const float inv = 1.0f / d;
  hedge[e] = make_float4(-(gd * u0 + (a.y - gu * u0) * inv), -(gd * u1 + (a.z - gu * u1) * inv),
                         -(gd * u2 + (a.w - gu * u2) * inv), 0.0f);
}

}  // namespace

int64_t local_buffer_floats(const LocalW& w, int64_t n, int64_t E) {
  LocalBufs b;
  return carve(w, n, E, nullptr, &b) + 32;
}

int local_forward_backward(cudaStream_t st, const LocalW& w, int64_t n, int64_t E, const int32_t* species_s,
                            const int32_t* arow, const int32_t* acol, const float4* ar, float* buf,
                            bool need_grad, const float* ew, double* energy_partials, int n_energy_partials,
                            float* e_atom, float4* hedge, int* status) {
  const int F = w.F, C = w.C, C2 = 2 * w.C, FX = w.F + 2 * w.C, Fh = w.F / 2, L = w.L, KA = w.KA;
  const bool bf = w.bf16;   // BF16 path: the dense edge GEMMs on tcgen05 (BF16 operands, FP32 accumulation)
  const int Kc = local_kc(w), Kh = w.Kh, KAb = w.KAb;
  int bad = 0;   // a GEMM shape the tensor-core GEMM rejects (checked on the host)
  LocalBufs b;
  carve(w, n, E, buf, &b);
  StageGuard fwd_stage(STG_EDGE_FWD);   // the whole forward is edge work
  if (E > 0) {
    { LaunchScope ls_(st); k_loc_erow<<<nblocks(n), kThreads, 0, st>>>(n, arow, b.erow); }
    {
      LaunchScope ls_(st);
      k_loc_geom<<<nblocks(E * 4), kThreads, 0, st>>>(E, w.K, w.S, KA, w.rc, ar, acol, b.erow, species_s, b.geo, b.in,
                                                  b.inb, KAb);
    }
    if (bf) {
      bad |= gemm_bf16<1>(st, E, F, KAb, b.inb, KAb, w.wb.A0t, w.c0, nullptr, 0, b.z0, F, b.Xb[0], FX, status);
      bad |= gemm_bf16<0>(st, E, C2, F, b.Xb[0], FX, w.wb.P0t, nullptr, nullptr, 0, b.w0, C2, nullptr, 0, status);
    } else {
      gemm_f32(st, 1, E, F, KA, b.in, KA, w.A0, w.c0, nullptr, 0, b.z0, F, b.X[0], FX);
      gemm_f32(st, 0, E, C2, F, b.X[0], FX, w.P0, nullptr, nullptr, 0, b.w0, C2, nullptr, 0);
    }
    { LaunchScope ls_(st); k_loc_init<<<nblocks(E * C), kThreads, 0, st>>>(E, C, b.w0, b.geo, b.S[0], b.V[0]); }
    for (int l = 1; l <= L; ++l) {
      const LocalLayerW& lw = w.Lw[l - 1];
      if (bf)
        bad |= gemm_bf16<0>(st, E, C2, F, b.Xb[l - 1], FX, w.wb.Qt[l - 1], nullptr, nullptr, 0, b.OM[l], C2, nullptr, 0, status);
      else
        gemm_f32(st, 0, E, C2, F, b.X[l - 1], FX, lw.Q, nullptr, nullptr, 0, b.OM[l], C2, nullptr, 0);
      { LaunchScope ls_(st); k_loc_env<<<nblocks(n * C), kThreads, 0, st>>>(n, C, arow, b.geo, b.OM[l], b.gamS[l], b.gamV[l]); }
      if (l < L && local_fused(w)) {
        LaunchScope ls_(st);
        (C == 16 ? k_loc_tp_mix<16> : k_loc_tp_mix<32>)<<<row_blocks(n, C), kThreads, 0, st>>>(
            n, arow, b.S[l - 1], b.V[l - 1], b.gamS[l], b.gamV[l], lw.Gs, lw.Gv, b.X[l - 1] + F, FX,
            bf ? b.Xb[l - 1] + F : nullptr, b.S[l], b.V[l]);
      } else {
        LaunchScope ls_(st);
        k_loc_tp<<<nblocks(E * C), kThreads, 0, st>>>(E, C, b.erow, b.S[l - 1], b.V[l - 1], b.gamS[l], b.gamV[l],
                                                      b.X[l - 1] + F, FX, l < L ? b.TV[l] : nullptr,
                                                      bf ? b.Xb[l - 1] + F : nullptr);
      }
      if (bf)
        bad |= gemm_bf16<1>(st, E, F, FX, b.Xb[l - 1], FX, w.wb.Mt[l - 1], lw.m, nullptr, 0, b.Z[l], F, b.Xb[l], FX, status);
      else
        gemm_f32(st, 1, E, F, FX, b.X[l - 1], FX, lw.M, lw.m, nullptr, 0, b.Z[l], F, b.X[l], FX);
      if (l < L && !local_fused(w)) {   // the 2C -> C channel mixings stay on the SIMT GEMM (N = C below a tensor-core tile)
        gemm_f32(st, 0, E, C, C2, b.X[l - 1] + F, FX, lw.Gs, nullptr, nullptr, 0, b.S[l], C, nullptr, 0);
        gemm_f32(st, 0, 3 * E, C, C2, b.TV[l], C2, lw.Gv, nullptr, nullptr, 0, b.V[l], C, nullptr, 0);
      }
    }
    if (bf)   // zh only; the readout applies silu itself
      bad |= gemm_bf16<0>(st, E, Fh, F, b.Xb[L], FX, w.wb.R1t, w.d1, nullptr, 0, b.zh, Fh, nullptr, 0, status);
    else
      gemm_f32(st, 1, E, Fh, F, b.X[L], FX, w.R1, w.d1, nullptr, 0, b.zh, Fh, b.h, Fh);
  }
  {
    LaunchScope ls_(st);
    k_loc_readout<<<n_energy_partials, kThreads, 0, st>>>(n, Fh, w.e_scale, arow, b.geo, bf ? nullptr : b.h, b.zh, w.R2,
                                                          w.d2, ew, e_atom, energy_partials, need_grad, b.gzh, b.gg,
                                                          b.gzhb, Kh);
  }
  if (!need_grad || E == 0) return bad;
  StageGuard bwd_stage(STG_EDGE_BWD);
  // g_z of layer L
  if (bf)
    bad |= gemm_bf16<3>(st, E, F, Kh, b.gzhb, Kh, w.wb.R1, nullptr, b.Z[L], F, nullptr, F, b.gxb, F, status);
  else
    gemm_f32(st, 3, E, F, Fh, b.gzh, Fh, w.R1t, nullptr, b.Z[L], F, b.gx, F, nullptr, 0);
  float *gs_in = b.gs[0], *gv_in = b.gv[0], *gs_out = b.gs[1], *gv_out = b.gv[1];
  for (int l = L; l >= 1; --l) {
    const LocalLayerW& lw = w.Lw[l - 1];
    // [g_x^{l-1} | g_ts] = g_z M_l^T
    if (bf)
      bad |= gemm_bf16<0>(st, E, FX, F, b.gxb, F, w.wb.M[l - 1], nullptr, nullptr, 0, b.gxc, FX, nullptr, 0, status);
    else
      gemm_f32(st, 0, E, FX, F, b.gx, F, lw.Mt, nullptr, nullptr, 0, b.gxc, FX, nullptr, 0);
    const float* gts = b.gxc + F;
    int ldg = FX;
    const float* gtv = nullptr;
    if (l < L && !local_fused(w)) {   // the channel mixings of layer l feed layer l+1
      gemm_f32(st, 2, E, C2, C, gs_in, C, lw.Gst, nullptr, b.gxc + F, FX, b.gts, C2, nullptr, 0);
      gts = b.gts;
      ldg = C2;
      gemm_f32(st, 0, 3 * E, C2, C, gv_in, C, lw.Gvt, nullptr, nullptr, 0, b.gtv, C2, nullptr, 0);
      gtv = b.gtv;
    }
    if (local_fused(w)) {
      auto go = C == 16 ? (l < L ? k_loc_tp_bwd<16, true> : k_loc_tp_bwd<16, false>)
                        : (l < L ? k_loc_tp_bwd<32, true> : k_loc_tp_bwd<32, false>);
      LaunchScope ls_(st);
      go<<<row_blocks(n, C), kThreads, 0, st>>>(n, arow, b.S[l - 1], b.V[l - 1], b.gamS[l], b.gamV[l], gts, ldg, gs_in,
                                                gv_in, lw.Gst, lw.Gvt, gs_out, gv_out, b.ggamS, b.ggamV);
    } else {
      {
        LaunchScope ls_(st);
        k_loc_tp_bwd_edge<<<nblocks(E * C), kThreads, 0, st>>>(E, C, b.erow, b.gamS[l], b.gamV[l], gts, ldg, gtv, gs_out,
                                                               gv_out);
      }
      LaunchScope ls_(st);
      k_loc_tp_bwd_atom<<<nblocks(n * C), kThreads, 0, st>>>(n, C, arow, b.S[l - 1], b.V[l - 1], gts, ldg, gtv, b.ggamS,
                                                             b.ggamV);
    }
    {
      LaunchScope ls_(st);
      k_loc_env_bwd<<<nblocks(E * 4), kThreads, 0, st>>>(E, C, b.erow, b.geo, b.OM[l], b.ggamS, b.ggamV, b.gom, b.gg,
                                                     b.gomb, Kc);
    }
    // g_x^{l-1} = g_xc[:, 0:F] + g_om Q_l^T, and for l > 1 g_z = g_x * silu'(z) of the layer below
    if (bf && l > 1)
      bad |= gemm_bf16<7>(st, E, F, Kc, b.gomb, Kc, w.wb.Q[l - 1], nullptr, b.gxc, FX, nullptr, F, b.gxb, F, status,
                          nullptr, b.Z[l - 1]);
    else if (bf)
      bad |= gemm_bf16<2>(st, E, F, Kc, b.gomb, Kc, w.wb.Q[l - 1], nullptr, b.gxc, FX, b.gx, F, nullptr, 0, status);
    else
      gemm_f32(st, l > 1 ? 4 : 2, E, F, C2, b.gom, C2, lw.Qt, nullptr, b.gxc, FX, b.gx, F, l > 1 ? b.Z[l - 1] : nullptr, F);
    std::swap(gs_in, gs_out);
    std::swap(gv_in, gv_out);
  }
  // gs_in, gv_in: gradients of the initial edge features
  { LaunchScope ls_(st); k_loc_init_bwd<<<nblocks(E * 4), kThreads, 0, st>>>(E, C, b.w0, b.geo, gs_in, gv_in, b.gw0, b.gg, b.gw0b, Kc); }
  if (bf)   // g_x0 * silu'(z0)
    bad |= gemm_bf16<7>(st, E, F, Kc, b.gw0b, Kc, w.wb.P0, nullptr, b.gx, F, nullptr, F, b.gxb, F, status, nullptr, b.z0);
  else
    gemm_f32(st, 4, E, F, C2, b.gw0, C2, w.P0t, nullptr, b.gx, F, b.gxc, FX, b.z0, F);
  if (bf)
    bad |= gemm_bf16<0>(st, E, KA, F, b.gxb, F, w.wb.A0, nullptr, nullptr, 0, b.gin, KA, nullptr, 0, status);
  else
    gemm_f32(st, 0, E, KA, F, b.gxc, FX, w.A0t, nullptr, nullptr, 0, b.gin, KA, nullptr, 0);
  { LaunchScope ls_(st); k_loc_geom_bwd<<<nblocks(E), kThreads, 0, st>>>(E, w.K, w.rc, b.geo, b.gin, KA, b.gg, hedge); }
  return bad;
}

}  // namespace ctd
