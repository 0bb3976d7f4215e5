// kdn_chunked_fwd.cu -- general chunked forward of the Diagonal and Isotropic KDN
// on CUDA cores (float32 arithmetic, any dk, dv in {32,64,128}, float32 or
// bfloat16 activations), the two-stage scheme of App. F in four kernels:
//   k_gain_comp_*  per 32-token chunk, in parallel over chunks: the ordered
//                  product of the tokens' 2 x 2 Moebius matrices (eq.
//                  chunk-gain-summary) on homogeneous coordinates (n, d), p = n / d;
//   k_gain_scan    the uncertainty entering every chunk (eq. chunk-gain-carry);
//   k_chunk_prep   per chunk, in parallel over chunks: the uncertainty recursion
//                  over the chunk's tokens and the gain emission (eq.
//                  chunk-gain-emission), the cumulative log-decay G and gamma =
//                  exp(G) (eq. chunk-memory-normalization), the scaled keys and
//                  queries (eq. chunk-memory-scaled-keys), T and A_qk, A = (I + T)^-1,
//                  W = A Kbar, U = A V and K_tail (eq. chunk-memory-wy, -tail-output);
//   k_state_fwd    the sequential inter-chunk pass R = U - W S_in,
//                  O = Qbar S_in + A_qk R, S_out = diag(gamma_C) S_in + K_tail^T R
//                  (eq. chunk-memory-output-state), columns of S split across
//                  CTAs (the columns of S are independent given kappa).
//
// All chunk-local matrices are float32 in shared memory; intermediates that
// cross kernels live in the caller's workspace.
//
// Diagonal prefill B8 H16 T2048 d = 64 bf16, us: 33 + 11 + 264 + 267, 578 a call.  With the
// uncertainty run token by token (1406), one output a thread in the chunk kernel (763) and two
// loads a multiply-add in the memory pass (790) it was 2922.
#include <float.h>

#include "kdn_chunked.cuh"

namespace kdn {
namespace {

constexpr int PT = 128;  // threads of k_chunk_prep

// ---------------------------------------------------------------------------
// Uncertainty: chunk summaries and their scan.

// The power of two that brings x >= 0 into [1, 2) (subnormals: as near as a normal factor gets).
__device__ __forceinline__ float pow2_to_one(float x) {
  const int e = (__float_as_int(x) >> 23) & 0xff;
  return __int_as_float((254 - min(max(e, 1), 253)) << 23);
}
// A 2x2 matrix of non-negative entries times the power of two that brings its
// largest entry into [1, 2): exact, and the ratio it represents is unchanged.
__device__ __forceinline__ void renorm_pow2(float *m) {
  const float inv = pow2_to_one(fmaxf(fmaxf(m[0], m[1]), fmaxf(m[2], m[3])));
#pragma unroll
  for (int q = 0; q < 4; ++q) m[q] *= inv;
}
// m <- M_t m with M_t = [[r a, r w], [n a, r + n w]], p -> phat / (1 + (n / r) phat) with
// phat = a p + w and n = mu k^2 (n / r = u): multiplied by r, so that no noise, however small,
// brings a large entry in.  The result is scaled, exactly, by the powers of two of max(r, n) and of
// m's largest entry: products of a few tokens' matrices leave the range of float32, a step
// leaves entries of at most ~4 (1 + w).
__device__ __forceinline__ void moebius_step(float *m, float a, float w, float r, float n) {
  const float sc = pow2_to_one(fmaxf(r, n) * fmaxf(fmaxf(m[0], m[1]), fmaxf(m[2], m[3])));
  const float r1 = r * sc, n1 = n * sc;
  const float x0 = fmaf(a, m[0], w * m[2]), x1 = fmaf(a, m[1], w * m[3]);
  m[2] = fmaf(n1, x0, r1 * m[2]);
  m[3] = fmaf(n1, x1, r1 * m[3]);
  m[0] = r1 * x0;
  m[1] = r1 * x1;
}
__device__ __forceinline__ float moebius_apply(const float *m, float p) {
  return fmaf(m[0], p, m[1]) / fmaf(m[2], p, m[3]);
}

// Diagonal KDN: DK / 4 threads per chunk, four adjacent channels each (8- or 16-byte loads).
// Reads k, g, omega once; bound by issue (~40 instructions a channel and token): 33 us for the 100 MB of
// B8 H16 T2048 d = 64 (26 with a rescaling every four tokens, which overflowed at small noises).
template <typename DT, int DK>
__global__ void __launch_bounds__(128) k_gain_comp_diag(Args a) {
  constexpr int L = DK / 4;
  const size_t n = (size_t)a.B * a.H * a.NC, idx = blockIdx.x * (size_t)(128 / L) + KDN_TID / L;
  if (idx >= n) return;
  const int bh = (int)(idx / a.NC), c = (int)(idx % a.NC), b = bh / a.H, h = bh % a.H;
  const int i0 = 4 * (KDN_TID % L);
  float m[4][4];
#pragma unroll
  for (int q = 0; q < 4; ++q) { m[q][0] = 1.f; m[q][1] = 0.f; m[q][2] = 0.f; m[q][3] = 1.f; }
  const int tn = min(CC, a.T - c * CC);
  for (int t0 = 0; t0 < tn; t0 += 4) {
    float kv[4][4], gv[4][4], wv[4][4], rr[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const size_t th = tok_index(a, b, c * CC + min(t0 + u, tn - 1), h);
      ld4<DT>(a.k, th * DK + i0, kv[u]);
      ld4<DT>(a.g, th * DK + i0, gv[u]);
      ld4<DT>(a.omega, th * DK + i0, wv[u]);
      rr[u] = gate_r(a.gates, a.rmin, ld<DT>(a.r, th));
    }
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      if (t0 + u >= tn) break;
#pragma unroll
      for (int q = 0; q < 4; ++q)
        moebius_step(m[q], expf(2.f * gate_logalpha(a.gates, gv[u][q])), gate_omega(a.gates, wv[u][q]), rr[u],
                     a.mu * kv[u][q] * kv[u][q]);
    }
  }
#pragma unroll
  for (int q = 0; q < 4; ++q) renorm_pow2(m[q]);
  float4 *dst = reinterpret_cast<float4 *>(a.comp) + idx * DK + i0;
#pragma unroll
  for (int q = 0; q < 4; ++q) dst[q] = f4(m[q]);
}

// Isotropic KDN: one warp per chunk, one lane per token: a_t and |k_t|^2 (kept in
// isotok), and the ordered product of the lanes' matrices by a shuffle tree.
template <typename DT, int DK>
__global__ void __launch_bounds__(128) k_gain_comp_iso(Args a) {
  const size_t n = (size_t)a.B * a.H * a.NC, idx = blockIdx.x * (size_t)4 + KDN_TID / 32;
  if (idx >= n) return;
  const int bh = (int)(idx / a.NC), c = (int)(idx % a.NC), b = bh / a.H, h = bh % a.H;
  const int lane = KDN_TID % 32, t = c * CC + lane;
  float aa = 1.f, n2 = 0.f, w = 0.f, rr = 1.f;
  if (t < a.T) {
    const size_t th = tok_index(a, b, t, h);
    float sa = 0.f;
#pragma unroll 4
    for (int i = 0; i < DK; i += 4) {
      float kv[4], gv[4];
      ld4<DT>(a.k, th * DK + i, kv);
      if (a.pcd) ld4<DT>(a.g, th * DK + i, gv);
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        n2 = fmaf(kv[q], kv[q], n2);
        if (a.pcd) sa += expf(2.f * gate_logalpha(a.gates, gv[q]));
      }
    }
    aa = a.pcd ? sa / DK : expf(2.f * gate_logalpha(a.gates, ld<DT>(a.g, th)));
    w = gate_omega(a.gates, ld<DT>(a.omega, th));
    rr = gate_r(a.gates, a.rmin, ld<DT>(a.r, th));
  }
  const size_t row = (size_t)bh * a.Tp + t;
  a.isotok[row * 2] = aa;
  a.isotok[row * 2 + 1] = n2;
  float m[4] = {1.f, 0.f, 0.f, 1.f};
  moebius_step(m, aa, w, DK * rr, a.mu * n2);
  renorm_pow2(m);
#pragma unroll
  for (int off = 1; off < 32; off <<= 1) {
    float p[4], x[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) p[q] = __shfl_down_sync(0xffffffffu, m[q], off);
    x[0] = fmaf(p[0], m[0], p[1] * m[2]);
    x[1] = fmaf(p[0], m[1], p[1] * m[3]);
    x[2] = fmaf(p[2], m[0], p[3] * m[2]);
    x[3] = fmaf(p[2], m[1], p[3] * m[3]);
    if ((lane & (2 * off - 1)) == 0) {
#pragma unroll
      for (int q = 0; q < 4; ++q) m[q] = x[q];
    }
    renorm_pow2(m);
  }
  if (lane == 0) reinterpret_cast<float4 *>(a.comp)[idx] = f4(m);
}

// One thread per (sequence, channel): the uncertainty entering every chunk.  A chain of NC
// Moebius applications, its matrices loaded eight chunks ahead: 11 us for 64 chunks.
__global__ void __launch_bounds__(128) k_gain_scan(Args a) {
  const size_t e = blockIdx.x * (size_t)128 + KDN_TID, n = (size_t)a.B * a.H * a.P;
  if (e >= n) return;
  const size_t bh = e / a.P, i = e % a.P;
  float p = a.p0 ? a.p0[e] : 1.f;
  const float4 *cm = reinterpret_cast<const float4 *>(a.comp) + bh * a.NC * a.P + i;
  float *pin = a.pin + bh * a.NC * a.P + i;
  for (int c0 = 0; c0 < a.NC; c0 += 8) {
    float4 x[8];
#pragma unroll
    for (int u = 0; u < 8; ++u)
      if (c0 + u < a.NC) x[u] = cm[(size_t)(c0 + u) * a.P];
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      if (c0 + u < a.NC) {
        pin[(size_t)(c0 + u) * a.P] = p;
        const float m[4] = {x[u].x, x[u].y, x[u].z, x[u].w};
        p = moebius_apply(m, p);
      }
    }
  }
}

// ---------------------------------------------------------------------------
// Chunk-local factors.
// Tokens past T are identity tokens: k = q = v = 0, g = 0, omega = 0, r = 1, kappa = 0.

// row stride (elements) of the V tile, kept in the activations' dtype: 16-byte rows
template <typename DT> __host__ __device__ constexpr int v_stride(int dv) { return dv + 16 / (int)sizeof(DT); }
// Diagonal KDN: Kk before the division by s_t is scaled down, exactly, so that phat k / gamma stays in
// range with it: phat k / (s_t gamma) does wherever gamma is a normal number, phat k / gamma alone
// overflows where a strong decay meets a large process noise.
constexpr float kKkDown = 0x1p-20f, kKkUp = 0x1p20f;
template <typename DT, int DK>
constexpr size_t prep_smem_bytes(int dv) {
  return sizeof(float) * (3 * CC * (DK + 4) + 2 * CC * LC + 16 * 20 + 8 * CC + DK + PT * 5) +
         sizeof(DT) * CC * v_stride<DT>(dv);
}

// A = (I + T)^-1 (32 x 32, T strictly lower in sT; zero above the diagonal of A):
// the two 16 x 16 diagonal blocks by forward substitution, one column a lane with
// its entries in registers, then A_10 = -D_1 T_10 D_0.  PT threads.
__device__ __forceinline__ void inverse32(const float *sT, float *sA, float *sX) {
  const int tid = KDN_TID;
  if (tid < 32) {
    const int o = tid & 16, col = tid & 15;
    float x[16];
#pragma unroll
    for (int r = 0; r < 16; ++r) {
      float a0 = (r == col) ? 1.f : 0.f, a1 = 0.f;
#pragma unroll
      for (int s = 0; s < r; s += 4) {
        float t4[4];
        ld4<float>(sT + (o + r) * LC + o + s, 0, t4);
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          if (s + u < r) {
            if (u & 1) a1 = fmaf(-t4[u], x[s + u], a1);
            else a0 = fmaf(-t4[u], x[s + u], a0);
          }
        }
      }
      x[r] = a0 + a1;
    }
#pragma unroll
    for (int r = 0; r < 16; ++r) sA[(o + r) * LC + o + col] = x[r];
  } else if (tid < 96) {
    const int e = tid - 32;  // upper right block
    const float z[4] = {0.f, 0.f, 0.f, 0.f};
    st4(sA + (e >> 2) * LC + 16 + 4 * (e & 3), z);
  }
  __syncthreads();
  const int r = tid >> 3, c2 = 2 * (tid & 7);
  {
    float x0 = 0.f, x1 = 0.f;
#pragma unroll
    for (int k = 0; k < 16; k += 4) {
      float t4[4];
      ld4<float>(sT + (16 + r) * LC + k, 0, t4);
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const float2 d = *reinterpret_cast<const float2 *>(sA + (k + u) * LC + c2);
        x0 = fmaf(t4[u], d.x, x0);
        x1 = fmaf(t4[u], d.y, x1);
      }
    }
    *reinterpret_cast<float2 *>(sX + r * 20 + c2) = make_float2(x0, x1);
  }
  __syncthreads();
  {
    float x0 = 0.f, x1 = 0.f;
#pragma unroll
    for (int k = 0; k < 16; k += 4) {
      float t4[4];
      ld4<float>(sA + (16 + r) * LC + 16 + k, 0, t4);
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const float2 d = *reinterpret_cast<const float2 *>(sX + (k + u) * 20 + c2);
        x0 = fmaf(t4[u], d.x, x0);
        x1 = fmaf(t4[u], d.y, x1);
      }
    }
    *reinterpret_cast<float2 *>(sA + (16 + r) * LC + c2) = make_float2(-x0, -x1);
  }
  __syncthreads();
}

// Reduce-scatter of N = 8 or 16 per-lane values over a warp: the warp-wide sum of v[lane / (32 / N)],
// by pairs.
template <int N>
__device__ __forceinline__ float warp_sums(const float *v, int lane) {
  float w[N];
#pragma unroll
  for (int j = 0; j < N; ++j) w[j] = v[j];
  int o = 16;
#pragma unroll
  for (int n = N / 2; n > 0; n >>= 1, o >>= 1) {
    const bool up = lane & o;
#pragma unroll
    for (int j = 0; j < n; ++j) {
      const float keep = up ? w[n + j] : w[j], send = up ? w[j] : w[n + j];
      w[j] = keep + __shfl_xor_sync(0xffffffffu, send, o);
    }
  }
  for (; o > 0; o >>= 1) w[0] += __shfl_xor_sync(0xffffffffu, w[0], o);
  return w[0];
}

// SAVE: also keep phat, gamma, A and s_t (iso: beta_t) for the backward.
// One CTA of 128 threads per chunk; five of them on an SM cover each other's load and barrier
// latencies.  Bound by shared-memory loads and issue (ncu, B8 H16 T2048 d = 64: 58 % of the
// shared-memory cycles, 51 % of the issue slots, the rest waits for the first loads); register
// tiles of 4 x 4 outputs, since a 16-byte load costs four cycles of the SM.  264 us (763 with
// one output a thread).
template <int V, typename DT, int DK, int SAVE>
__global__ void __launch_bounds__(PT, DK < 128 ? 5 : 3) k_chunk_prep(Args a) {
  constexpr int LD = DK + 4, NSEG = PT / DK, SL = CC / NSEG;  // token segments per channel
  extern __shared__ __align__(16) float sm[];
  const int dv = a.dv, lv = v_stride<DT>(dv);
  float *sK = sm, *sQ = sK + CC * LD, *sKk = sQ + CC * LD, *sT = sKk + CC * LD, *sA = sT + CC * LC;
  float *sX = sA + CC * LC, *s_r = sX + 16 * 20, *s_mr = s_r + CC;
  float *s_is = s_mr + CC, *s_be = s_is + CC, *s_k2 = s_be + CC, *s_gC = s_k2 + 4 * CC, *s_seg = s_gC + DK;
  DT *sV = reinterpret_cast<DT *>(s_seg + PT * 5);
  const int tid = KDN_TID;
  const int bh = (int)(blockIdx.x / (unsigned)a.NC), c = (int)(blockIdx.x % (unsigned)a.NC);
  const int b = bh / a.H, h = bh % a.H, tn = min(CC, a.T - c * CC);
  const size_t base = (size_t)bh * a.NC + c;

  // this thread's channel and tokens; all loads issued ahead of their uses
  const int i = tid % DK, t0 = (tid / DK) * SL;
  constexpr int LB = SL > 16 ? 16 : SL;  // tokens held in registers at a time
  float kv[LB], qv[LB], gv[LB], wv[LB], a2[LB];
  const size_t tok0 = tok_index(a, b, c * CC, h), row_e = (size_t)a.H * DK;
  auto load = [&](int tb) {
    const size_t o = (tok0 + (size_t)tb * a.H) * DK + i;
#pragma unroll
    for (int j = 0; j < LB; ++j) {
      kv[j] = qv[j] = gv[j] = wv[j] = 0.f;
      if (tb + j < tn) {
        kv[j] = ld<DT>(a.k, o + j * row_e);
        qv[j] = ld<DT>(a.q, o + j * row_e);
        gv[j] = ld<DT>(a.g, a.pcd ? o + j * row_e : tok0 + (size_t)(tb + j) * a.H);
        if (V == 0) wv[j] = ld<DT>(a.omega, o + j * row_e);
      }
    }
  };
  auto gates = [&](int tb) {  // log alpha (gv), alpha^2, omega; identity tokens past T
    if (a.gates) {
#pragma unroll
      for (int j = 0; j < LB; ++j) {
        gv[j] = tb + j < tn ? gate_logalpha(1, gv[j]) : 0.f;
        if (V == 0) wv[j] = tb + j < tn ? gate_omega(1, wv[j]) : 0.f;
      }
    }
    if (V == 0) {
#pragma unroll
      for (int j = 0; j < LB; ++j) a2[j] = expf(2.f * gv[j]);
    }
  };
  load(t0);
  float p = 1.f;
  if (V == 0) p = a.pin[base * DK + i];
  {  // V by asynchronous copies, waited for ahead of U = A V
    constexpr int EP = 16 / (int)sizeof(DT);  // elements per 16-byte piece
    const int pieces = dv / EP;
    for (int e = tid; e < CC * pieces; e += PT) {
      const int t = e / pieces, j = EP * (e % pieces);
      cp16(sV + t * lv + j, static_cast<const DT *>(a.v) + (tok0 + (size_t)(t < tn ? t : 0) * a.H) * dv + j, t < tn);
    }
    cp_commit();
  }
  if (tid < CC) {
    const float rr =
        tid < tn ? gate_r(a.gates, a.rmin, ld<DT>(a.r, tok_index(a, b, c * CC + tid, h))) : 1.f;
    s_r[tid] = rr;
    s_mr[tid] = fminf(a.mu / rr, FLT_MAX);  // (finite, so that k = 0 gives u = 0)
    if (V == 1) {  // the scalar uncertainty of the chunk's tokens: ordered products of M_t by shuffles
      const size_t row = (size_t)bh * a.Tp + c * CC + tid;
      const float aa = a.isotok[row * 2], n2 = a.isotok[row * 2 + 1];
      const float w = tid < tn ? gate_omega(a.gates, ld<DT>(a.omega, tok_index(a, b, c * CC + tid, h))) : 0.f;
      const float pin = a.pin[base];
      float m[4] = {1.f, 0.f, 0.f, 1.f};
      moebius_step(m, aa, w, DK * rr, a.mu * n2);
  renorm_pow2(m);
#pragma unroll
      for (int off = 1; off < 32; off <<= 1) {
        float p[4], x[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) p[q] = __shfl_up_sync(0xffffffffu, m[q], off);
        x[0] = fmaf(m[0], p[0], m[1] * p[2]);
        x[1] = fmaf(m[0], p[1], m[1] * p[3]);
        x[2] = fmaf(m[2], p[0], m[3] * p[2]);
        x[3] = fmaf(m[2], p[1], m[3] * p[3]);
        if (tid >= off) {
#pragma unroll
          for (int q = 0; q < 4; ++q) m[q] = x[q];
        }
        renorm_pow2(m);
      }
      // b_t, then twice one step of the recursion from b_{t-1}, which damps the products' rounding
      float bt = moebius_apply(m, pin), bhat;
      const float u = fminf(a.mu * n2 / (DK * rr), FLT_MAX);
#pragma unroll
      for (int it = 0; it < 3; ++it) {
        float bp = __shfl_up_sync(0xffffffffu, bt, 1);
        if (tid == 0) bp = pin;
        bhat = fmaf(aa, bp, w);  // eq. iso-kla-box-cov-update
        if (it < 2) bt = bhat / fmaf(u, bhat, 1.f);
      }
      const float beta = tid < tn ? bhat / (rr + bhat * n2) : 0.f;
      s_be[tid] = beta;
      if (SAVE) {
        a.phat[row] = bhat;
        a.stok[row] = beta;
      }
      if (a.pT && c == a.NC - 1 && tid == tn - 1) a.pT[bh] = bt;
    }
  }
  __syncthreads();

  // gains and decay of the segment's tokens
  float G = 0.f;
  gates(t0);
  if (NSEG > 1) {  // the segments before this one: their decay sums and Moebius products
    float m[4] = {1.f, 0.f, 0.f, 1.f}, gs = 0.f;
#pragma unroll
    for (int j = 0; j < LB; ++j) {
      gs += gv[j];
      if (V == 0) moebius_step(m, a2[j], wv[j], s_r[t0 + j], a.mu * kv[j] * kv[j]);
    }
    renorm_pow2(m);
    float *mine = s_seg + tid * 5;
#pragma unroll
    for (int q = 0; q < 4; ++q) mine[q] = m[q];
    mine[4] = gs;
    __syncthreads();
    for (int s = 0; s < tid / DK; ++s) {
      const float *o = s_seg + (s * DK + i) * 5;
      G += o[4];
      if (V == 0) p = moebius_apply(o, p);
    }
  }
  float gam = expf(G);
  const size_t grow = ((size_t)bh * a.Tp + c * CC) * DK + i;
  for (int tb = t0; tb < t0 + SL; tb += LB) {
    if (tb > t0) {
      load(tb);
      gates(tb);
    }
#pragma unroll
    for (int j = 0; j < LB; ++j) {
      const int t = tb + j;
      float ph = 0.f, kk;
      G += gv[j];
      gam = expf(G);
      if (V == 0) {
        ph = fmaf(a2[j], p, wv[j]);                             // eq. diag-covariance-prediction
        p = ph / fmaf(s_mr[t] * kv[j] * kv[j], ph, 1.f);        // eq. diag-cov-update
        kk = kKkDown * ph * kv[j];
        a2[j] = ph * kv[j] * kv[j];
      } else {
        kk = s_be[t] * kv[j];
      }
      sK[t * LD + i] = kv[j] * gam;
      sQ[t * LD + i] = a.tau * qv[j] * gam;
      sKk[t * LD + i] = kk / gam;  // (diag: kKkDown s_t Kk)
      if (SAVE) {
        if (V == 0) a.phat[grow + (size_t)t * DK] = ph;
        a.gam[grow + (size_t)t * DK] = gam;
      }
    }
    if (V == 0) {  // sum_i phat k^2 over this warp's channels
      const float s = warp_sums<LB>(a2, tid & 31);
      if ((tid & (32 / LB - 1)) == 0) s_k2[(i >> 5) * CC + tb + (tid & 31) / (32 / LB)] = s;
    }
  }
  if (t0 + SL == CC) {
    s_gC[i] = gam;
    a.gC[base * DK + i] = gam;
    if (V == 0 && a.pT && c == a.NC - 1) a.pT[(size_t)bh * DK + i] = p;
  }
  __syncthreads();

  if (V == 0 && tid < CC) {  // s_t = r_t + sum_i phat k^2 (eq. kla-box-gain)
    float s = s_k2[tid];
#pragma unroll
    for (int w = 1; w < DK / 32; ++w) s += s_k2[w * CC + tid];
    s += s_r[tid];
    s_is[tid] = fminf(kKkUp / s, FLT_MAX);
    if (SAVE) a.stok[(size_t)bh * a.Tp + c * CC + tid] = s;
  }
  // T' = Kbar Kk'^T (threads 0..63), A'_qk = Qbar Kk'^T (64..127): 32 x 32, 4 x 4 a thread.
  const int lane = tid & 31, w2 = (tid >> 5) & 1, ga = lane >> 2, gb = (lane & 3) + 4 * w2;
  float acc[4][4];
  zero<4>(acc);
  tile_mm<DK, 4, true>(acc, (tid < 64 ? sK : sQ) + ga * LD, 8 * LD, sKk + 4 * gb * LD, LD);
  if (V == 0) __syncthreads();  // s_is
#pragma unroll
  for (int m = 0; m < 4; ++m) {
    const int r = ga + 8 * m;
    float x[4];
#pragma unroll
    for (int n = 0; n < 4; ++n) {
      const int s = 4 * gb + n;
      x[n] = (s < r || (s == r && tid >= 64)) ? acc[m][n] * (V == 0 ? s_is[s] : 1.f) : 0.f;
    }
    if (tid < 64) st4(sT + r * LC + 4 * gb, x);
    else st4(a.Aqk + (base * CC + r) * CC + 4 * gb, x);
  }
  __syncthreads();
  cp_wait<0>();  // V (the barriers of the solve make every thread's copies visible)
  inverse32(sT, sA, sX);

  // W = A Kbar and U = A V (32 x dk, 32 x dv; 16 columns a warp), then Qbar, K_tail
  for (int e = tid; e < 2 * (DK + dv); e += PT) {
    const int col = 16 * (e >> 5) + 4 * (e & 3);
    const bool isW = col < DK;
    zero<4>(acc);
    if (isW) tile_mm<CC, 4, false>(acc, sA + ga * LC, 8 * LC, sK + col, LD);
    else tile_mm<CC, 4, false, DT>(acc, sA + ga * LC, 8 * LC, sV + col - DK, lv);
#pragma unroll
    for (int m = 0; m < 4; ++m) {
      const int r = ga + 8 * m;
      if (isW) st4(a.W + (base * CC + r) * DK + col, acc[m]);
      else st4(a.U + (base * CC + r) * dv + col - DK, acc[m]);
    }
  }
  for (int e = tid; e < CC * (DK / 4); e += PT) {
    const int t = e / (DK / 4), i4 = 4 * (e % (DK / 4));
    float x[4], y[4], g4[4];
    ld4<float>(sQ + t * LD, i4, x);
    st4(a.Qb + (base * CC + t) * DK + i4, x);
    ld4<float>(sKk + t * LD, i4, y);
    ld4<float>(s_gC, i4, g4);
#pragma unroll
    for (int u = 0; u < 4; ++u) y[u] = g4[u] * (V == 0 ? y[u] * s_is[t] : y[u]);
    st4(a.Kt + (base * CC + t) * DK + i4, y);
  }
  if (SAVE) {
    for (int e = tid; e < CC * (CC / 4); e += PT) {
      float x[4];
      ld4<float>(sA + (e >> 3) * LC, 4 * (e & 7), x);
      st4(a.Ainv + base * CC * CC + 4 * e, x);
    }
  }
}

// ---------------------------------------------------------------------------
// The inter-chunk pass: a chain over the chunks, one CTA per (sequence, value columns), the next
// chunk's factors in flight.  A thread keeps its rows of S in registers and forms 8 x 4 tiles of
// [W; Qbar] S.  With one warp per scheduler it is bound by latency and shared-memory loads (ncu,
// B8 H16 T2048 d = 64: 55 % of the issue slots, 52 % of the shared-memory cycles): 267 us for
// 64 chunks, 790 before.  The sums are split in halves and a chunk's part is added to S at once, so that
// they round no more than a token loop's would (261 us in one chain, S and dS off by up to 1.5 times as much).

template <int DK, int CW, int TM, int SAVE>
__global__ void __launch_bounds__(StateCfg<DK, CW, TM>::NTH) k_state_fwd(Args a) {
  using Cfg = StateCfg<DK, CW, TM>;
  constexpr int LD = Cfg::LD, LS = Cfg::LS, GA = Cfg::GA, RS = Cfg::RS, TH = TM / 2;
  extern __shared__ __align__(16) float sm[];
  float *sS = sm + 2 * Cfg::FLOATS, *sR = sS + DK * LS;
  const int ns = a.dv / CW, bh = (int)(blockIdx.x / (unsigned)ns), j0 = (int)(blockIdx.x % (unsigned)ns) * CW;
  const int tid = KDN_TID, b = bh / a.H, h = bh % a.H, dv = a.dv;
  const int col = 4 * (tid % (CW / 4)), ga = tid / (CW / 4), i0 = RS * ga;
  const size_t sbase = ((size_t)bh * DK + i0) * dv + j0 + col;
  float S[RS][4];  // this thread's rows of the memory, mirrored in sS
#pragma unroll
  for (int m = 0; m < RS; ++m) {
#pragma unroll
    for (int n = 0; n < 4; ++n) S[m][n] = 0.f;
    if (a.S0) ld4<float>(a.S0 + sbase + (size_t)m * dv, 0, S[m]);
    st4(sS + (i0 + m) * LS + col, S[m]);
  }
  issue_chunk_factors<Cfg, DK, CW>(a, bh, 0, sm, j0, false);
  cp_commit();
  for (int c = 0; c < a.NC; ++c) {
    const float *buf = sm + (c & 1) * Cfg::FLOATS;
    cp_wait<0>();
    __syncthreads();  // chunk c has landed; chunk c - 1 is finished by every thread
    if (c + 1 < a.NC) issue_chunk_factors<Cfg, DK, CW>(a, bh, c + 1, sm + ((c + 1) & 1) * Cfg::FLOATS, j0, false);
    cp_commit();
    const float *sKt = buf + 2 * CC * LD, *sAqk = sKt + CC * LD, *sgC = sAqk + CC * LC, *sU = sgC + DK;
    const size_t base = (size_t)bh * a.NC + c;
    if (SAVE) {
#pragma unroll
      for (int m = 0; m < RS; ++m) st4(a.Sin + (base * DK + i0 + m) * dv + j0 + col, S[m]);
    }
    float acc[TM][4];
    zero<TM>(acc);
    tile_mm2<DK, TM>(acc, buf + ga * LD, GA * LD, sS + col, LS);
    // R = U - W S_in
#pragma unroll
    for (int m = 0; m < TH; ++m) {
      const int r = ga + GA * m;
      float u[4];
      ld4<float>(sU + r * LS, col, u);
#pragma unroll
      for (int n = 0; n < 4; ++n) u[n] -= acc[m][n];
      st4(sR + r * LS + col, u);
      if (SAVE) st4(a.R + (base * CC + r) * dv + j0 + col, u);
    }
    __syncthreads();
    // O = Qbar S_in + A_qk R
    if (a.o) {
      float t[TH][4];
      zero<TH>(t);
      tile_mm<CC, TH, false>(t, sAqk + ga * LC, GA * LC, sR + col, LS);
#pragma unroll
      for (int m = 0; m < TH; ++m) {
        const int tt = c * CC + ga + GA * m;
#pragma unroll
        for (int n = 0; n < 4; ++n) t[m][n] += acc[TH + m][n];
        if (tt < a.T) sto4(a.odt, a.o, tok_index(a, b, tt, h) * dv + j0 + col, t[m]);
      }
    }
    // S_out = diag(gamma_C) S_in + K_tail^T R: the chunk's part first, so that S is rounded once
    float inc[2][RS][4];
#pragma unroll
    for (int hf = 0; hf < 2; ++hf) {
      zero<RS>(inc[hf]);
      tile_mm_t<CC / 2, RS>(inc[hf], sKt + hf * (CC / 2) * LD + i0, LD, sR + hf * (CC / 2) * LS + col, LS);
    }
#pragma unroll
    for (int m = 0; m < RS; ++m) {
      const float g = sgC[i0 + m];
#pragma unroll
      for (int n = 0; n < 4; ++n) S[m][n] = fmaf(g, S[m][n], inc[0][m][n] + inc[1][m][n]);
      st4(sS + (i0 + m) * LS + col, S[m]);
    }
  }
  if (a.ST) {
#pragma unroll
    for (int m = 0; m < RS; ++m) st4(a.ST + sbase + (size_t)m * dv, S[m]);
  }
}

// ---------------------------------------------------------------------------
// Launchers

template <int DK, int CW, int TM, int SAVE>
bool state_fwd(const Args &a, cudaStream_t s) {
  using Cfg = StateCfg<DK, CW, TM>;
  return launch(k_state_fwd<DK, CW, TM, SAVE>, (size_t)a.B * a.H * (a.dv / CW), Cfg::NTH, Cfg::SMEM, s, a);
}
template <int V, typename DT, int DK, int SAVE>
kdn_status_t fwd_impl(const Args &a, cudaStream_t s) {
  const size_t BH = (size_t)a.B * a.H, n = BH * a.NC;
  constexpr int per = 128 / (DK / 4);
  bool ok = V == 0 ? launch(k_gain_comp_diag<DT, DK>, (n + per - 1) / per, 128, 0, s, a)
                   : launch(k_gain_comp_iso<DT, DK>, (n + 3) / 4, 128, 0, s, a);
  ok = ok && launch(k_gain_scan, (BH * a.P + 127) / 128, 128, 0, s, a);
  ok = ok && launch(k_chunk_prep<V, DT, DK, SAVE>, n, PT, prep_smem_bytes<DT, DK>(a.dv), s, a);
  switch (state_cols(a)) {
    case 64: ok = ok && state_fwd<DK, 64, 8, SAVE>(a, s); break;
    case 32: ok = ok && state_fwd<DK, 32, 4, SAVE>(a, s); break;
    default: ok = ok && state_fwd<DK, 16, 2, SAVE>(a, s);
  }
  return ok ? KDN_OK : KDN_ERR_CUDA;
}

template <int V, typename DT>
kdn_status_t fwd_dk(const Args &a, cudaStream_t s, bool save) {
  switch (a.dk) {
    case 32: return save ? fwd_impl<V, DT, 32, 1>(a, s) : fwd_impl<V, DT, 32, 0>(a, s);
    case 64: return save ? fwd_impl<V, DT, 64, 1>(a, s) : fwd_impl<V, DT, 64, 0>(a, s);
    case 128: return save ? fwd_impl<V, DT, 128, 1>(a, s) : fwd_impl<V, DT, 128, 0>(a, s);
  }
  return KDN_ERR_UNSUPPORTED;
}

}  // namespace

int chunked_chunk_len() { return CC; }

int chunked_fwd_launches(const Args &) { return 4; }

kdn_status_t launch_chunked_fwd(const Args &a, cudaStream_t s, bool save) {
  if (a.variant == 0)
    return a.dtype == KDN_BF16 ? fwd_dk<0, __nv_bfloat16>(a, s, save) : fwd_dk<0, float>(a, s, save);
  return a.dtype == KDN_BF16 ? fwd_dk<1, __nv_bfloat16>(a, s, save) : fwd_dk<1, float>(a, s, save);
}

}  // namespace kdn
