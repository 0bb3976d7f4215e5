// kdn_wy_fwd.cu -- chunked forward of the Diagonal KDN in compact-WY form
// (App. F.2, eq. chunk-memory-wy / chunk-memory-output-state) for bfloat16
// activations, d_k = d_v = 128 and chunks of C = 64 tokens, on the tcgen05
// tensor cores of sm_103a.
//
// One CTA (16 warps) owns one (batch, head) and walks its chunks in order; the
// 128 x 128 float32 memory S stays in tensor memory for the whole sequence,
// every activation tile is read once by TMA and o is written once.  Per chunk,
// with G_t = sum_{u<=t} g_u the cumulative log-decay inside the chunk (per
// channel) and gamma_t = exp(G_t):
//
//   gain     warps 0-3, one thread per key channel, run the uncertainty
//            recursion of Prop. 3 over the 64 tokens (eq. diag-cov-update,
//            eq. prefix-diag-uncertainty).  Each thread writes
//              Kk'_t = phat_t k_t exp(c - G_t)          (tf32, MMA-T operand)
//              K'_t  = phat_t k_t exp(G_C - G_t)        (fp16, tensor memory)
//            where c = G_C / 2 is a per-channel reference in the middle of
//            the chunk's decay range.
//   prepare  warps 4-11, one thread per (4 channels, 8 tokens), form
//              Kbar_t = k_t exp(G_t - c), Qbar_t = tau q_t exp(G_t - c)  (tf32)
//              -Kbar_t = -gamma_t k_t, Qbar_t = tau gamma_t q_t        (fp16)
//   MMA-T    [Kbar; Qbar] Kk'^T (tf32) = [T'; A'_qk].  The ratios
//            exp(G_t - G_s) of App. F.2 are exact products of the two
//            referenced factors, each within exp(+-|G_C| / 2).
//            s_t = r_t + sum_i phat_t,i k_t,i^2 (the denominator of the gain,
//            eq. kla-box-gain) is r_t plus the diagonal of T'.
//   MMA-KS   [-Kbar; Qbar] S_in = [-Kbar S_in; Qbar S_in]  (fp16), on the tensor
//            cores while the CUDA cores solve
//   solve    with L = diag(s) + strict_lower(T'), A = (I + T)^-1 = diag(s) L^-1
//            (T = strict_lower(T') diag(1/s)) on CUDA cores in fp32: diagonal blocks on two
//            warps beside Y = V - Kbar S_in on six, the 32 x 32 products without the zero
//            quarter of their triangular factor.
//   MMA-R    R = U - W S_in = A (V - Kbar S_in)  (fp16; W = A Kbar, U = A V of
//            eq. chunk-memory-wy are only formed for the backward's context)
//   MMA-O    O = Qbar S_in + A'_qk R'          with R' = diag(1/s) R
//   MMA-S2   S_out = diag(gamma_C) S_in + K'^T R'   (K' in tensor memory)
// so that A'_qk R' = A_qk R and K'^T R' = K_tail^T R of eq.
// chunk-memory-output-state, with A_qk = lower(A'_qk) diag(1/s).  Every MMA
// accumulates in float32 in tensor memory.
//
// The chunk is a chain of dependent stages inside one CTA, and with logit gates the gain (run
// one chunk ahead on its own warps) is as long as the rest: the kernel is bound by
// that latency, not by HBM or shared-memory throughput.  B8 H16 T4096: 545 us (646 with the
// solve's diagonal blocks and Y on the same warps, and MMAs issued under a divergent branch),
// with the context 633 us (730; its copies go out one per warp, and A_qk is written
// beside the -W product).  Few sequences: k_wy_flow (below).
// Every per-element pass
// still reads and writes 8 or 16 bytes per shared-memory instruction wherever the
// layout allows (the gain's per-channel recursion is the exception), and the
// next chunk's TMA operations are issued from a thread outside the MMA issuer's
// warp while every main warp waits for MMA-T.
//
// Range: the referenced factors stay finite while the chunk's cumulative
// log-decay G_C >= -160 in every channel (average alpha >= 0.082 over 64
// tokens).  A chunk below that (flagged by the gain warps, for every channel
// at once) runs in range mode: the main warps form T' and A'_qk on the CUDA
// cores from exp(G_t - G_s), s <= t, which never exceeds 1, in place of MMA-T;
// gamma_t and K' are then formed from G_t directly.  The context-saving
// instantiation keeps the referenced form (the fused backward it feeds divides
// by gamma and reports exp(G_C) < 1e-36 as KDN_ERR_RANGE).
//
// Logit gates (LG): g, omega, r hold the logits x, y, z of the layer's
// parameterisation (Sec. 5): log alpha = -softplus(-x), omega = softplus(y),
// r = r_min + softplus(z), formed in float32.  The gain forms log alpha once per
// element and keeps it in its column of the Kk' tile until the recursion
// overwrites it; the prepare pass forms its own.  The tokens past T are identity
// updates: their rows of the g and omega tiles are set to logits whose
// activations are exactly alpha = 1 and omega = 0, so no pass masks elements.
//
// Every wait on an mbarrier is bounded; on timeout the kernel records
// KDN_ERR_TIMEOUT in the status word, waits (bounded) for its copies in flight,
// frees its tensor memory and returns.
#include <algorithm>
#include <type_traits>

#include "kdn_internal.cuh"
#include "kdn_sm103.cuh"
#include "kdn_fused_common.cuh"

namespace kdn {
namespace {

using namespace sm103;
using namespace fused;

constexpr int WT = 512;  // threads
constexpr int CM = 64;   // chunk length
constexpr int D = 128;   // d_k = d_v
constexpr uint32_t kWait = 1u << 25;
constexpr uint32_t kDrain = 1u << 14;  // bounded waits of the failure path
constexpr float kLog2e = 1.4426950408889634f;
constexpr float kLn2 = 0.6931471805599453f;
constexpr float kMinHalfG = -80.f;  // c = G_C / 2 below this: out of range
constexpr int kPrepThreads = 256;   // warps 4-11: the preparing pass
constexpr int kMain = 384;          // warps 4-15: everything but the gain
constexpr int kBarMain = 2, kBarGain = 3;  // named barriers (0 = __syncthreads)
constexpr int kTmaThread = 224;  // warp 7, lane 0: issues each chunk's next-chunk TMA operations

// shared-memory map (bytes from the 1024-aligned base)
constexpr int LT = 68;          // row stride (floats) of the fp32 T and A tiles
constexpr int O_RK = 0;        // raw k  [64 t][128 i] bf16, two 64-channel slabs   16 KB
constexpr int O_RG = 16384;    // raw g                                          16 KB
constexpr int O_RW = 32768;    // raw omega                                      16 KB
constexpr int O_V = 49152;     // V (TMA bf16), then Y fp16, then R' fp16 [64 s][128 j]  16 KB
constexpr int O_TA = 65536;    // tf32 [Kbar; Qbar] [128][128], four 32-channel slabs 64 KB
constexpr int O_TB = 133120;   // tf32 Kk' [64][128], four slabs                   32 KB
constexpr int O_Q = 165888;    // q (TMA, one chunk ahead; the preparing pass)    16 KB
constexpr int O_AS1 = 182272;  // fp16 [-Kbar; Qbar] [128][128], two slabs (MMA-KS A) 32 KB
constexpr int O_SMALL = 215040;
// after MMA-T has read the tf32 tiles (T and A run 2 KB past the tf32 tile)
constexpr int O_S16 = O_TA;                      // fp16 S_in [128 i][128 j], two slabs (MMA-KS B)
constexpr int O_SWT = O_TA + 32768;              // fp32 T' [64][LT]
constexpr int O_SWA = O_SWT + 64 * LT * 4;       // fp32 L^-1 [64][LT]
static_assert(O_SWA + 64 * LT * 4 <= O_TB, "T and A tiles overlap the Kk' tile");
constexpr int O_AWU = O_SWT;           // fp16 [A; .] [128][64] (MMA-R A), over T' after the solve
// small arrays (floats); r and mu / r per token for two chunks (the gain works one chunk ahead)
constexpr int SM_R = 0, SM_MUR = 128, SM_S = 256, SM_IS = 320, SM_C = 384, SM_GC = 512,
              SM_PART = 640, SM_OOR = 640 + 8 * 128, SM_FLOATS = SM_OOR + 16;
constexpr int O_BAR = O_SMALL + SM_FLOATS * 4;
constexpr int O_SX = O_BAR + 64;       // scratch of the solve: 2 x 256 floats
constexpr int O_SY = O_SX + 2048;      //                       32 x 32 floats
constexpr int SMEM_BYTES = O_SY + 4096 + 1024;
static_assert(SMEM_BYTES <= 232448, "shared memory per CTA");

// tensor-memory columns (512 allocated)
constexpr uint32_t TC_S = 0, TC_D1 = 128, TC_KT = 192, TC_W = 256, TC_U = 384;

__device__ __forceinline__ float ex2f(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
__device__ __forceinline__ float rcpf(float x) {
  float y;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
__device__ __forceinline__ float lg2f(float x) {
  float y;
  asm("lg2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
// softplus(x) = max(x, 0) + log(1 + exp(-|x|)), from the two approximate base-2
// operations with subnormals flushed (exactly 0 below x = -88)
__device__ __forceinline__ float softplus_w(float x) {
  return fmaxf(x, 0.f) + kLn2 * lg2f(1.f + ex2f(-fabsf(x) * kLog2e));
}
// round to tf32 (nearest, ties away): the tensor core reads the top 19 bits
__device__ __forceinline__ float tf32r(float x) {
  uint32_t u;
  asm("cvt.rna.tf32.f32 %0, %1;" : "=r"(u) : "f"(x));
  return __uint_as_float(u);
}
// byte offset of fp32 element (row, col) of a 128-byte-swizzled tile with 32
// elements per row
__device__ __forceinline__ uint32_t sw32_off(uint32_t row, uint32_t col) {
  return row * 128u + ((((col >> 2) ^ (row & 7u)) << 4) | ((col & 3u) << 2));
}
__device__ __forceinline__ void bar_sync(int id, int n) {
  asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(n) : "memory");
}
// generic-proxy accesses before, async-proxy (bulk copy) accesses after, for every state space
__device__ __forceinline__ void fence_proxy_async_all() { asm volatile("fence.proxy.async;" ::: "memory"); }
__device__ __forceinline__ void bar_arrive(int id, int n) {
  asm volatile("bar.arrive %0, %1;" ::"r"(id), "r"(n) : "memory");
}
// named barrier that also returns the OR of a predicate over its n threads
__device__ __forceinline__ bool bar_or(int id, int n, bool p) {
  uint32_t r;
  asm volatile(
      "{\n .reg .pred pi, po;\n setp.ne.u32 pi, %1, 0;\n barrier.cta.red.or.pred po, %2, %3, pi;\n"
      " selp.u32 %0, 1, 0, po;\n}"
      : "=r"(r)
      : "r"((uint32_t)p), "r"(id), "r"(n)
      : "memory");
  return r != 0;
}
__host__ __device__ constexpr uint32_t idesc_tf32(int M, int N) {
  return (1u << 4) | (2u << 7) | (2u << 10) | ((uint32_t)(N >> 3) << 17) | ((uint32_t)(M >> 4) << 24);
}
__device__ __forceinline__ void umma_tf32(uint32_t lead, uint32_t d, uint64_t a, uint64_t b,
                                          uint32_t idesc, uint32_t acc) {
  asm volatile(
      "{\n .reg .pred p, q;\n setp.ne.b32 p, %4, 0;\n setp.ne.b32 q, %5, 0;\n"
      " @q tcgen05.mma.cta_group::1.kind::tf32 [%0], %1, %2, %3, p;\n}\n" ::"r"(d),
      "l"(a), "l"(b), "r"(idesc), "r"(acc), "r"(lead)
      : "memory");
}
// A operand in tensor memory: lane = row, 32-bit column c holds the 16-bit
// elements 2c (low half) and 2c + 1 of that row
__device__ __forceinline__ void umma_f16_tA(uint32_t lead, uint32_t d, uint32_t a_tmem, uint64_t b,
                                            uint32_t idesc, uint32_t acc) {
  asm volatile(
      "{\n .reg .pred p, q;\n setp.ne.b32 p, %4, 0;\n setp.ne.b32 q, %5, 0;\n"
      " @q tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n}\n" ::"r"(d),
      "r"(a_tmem), "l"(b), "r"(idesc), "r"(acc), "r"(lead)
      : "memory");
}
__device__ __forceinline__ void tmem_st4u(uint32_t taddr, const uint32_t *v) {
  asm volatile("tcgen05.st.sync.aligned.32x32b.x4.b32 [%0], {%1, %2, %3, %4};" ::"r"(taddr),
               "r"(v[0]), "r"(v[1]), "r"(v[2]), "r"(v[3])
               : "memory");
}
// four bf16 (8 bytes) -> floats
__device__ __forceinline__ void unpack_bf4(uint2 u, float *v) {
  v[0] = __uint_as_float(u.x << 16);
  v[1] = __uint_as_float(u.x & 0xffff0000u);
  v[2] = __uint_as_float(u.y << 16);
  v[3] = __uint_as_float(u.y & 0xffff0000u);
}
__device__ __forceinline__ uint2 pack_h4(float a0, float a1, float a2, float a3) {
  uint2 u;
  __half2 h0 = __floats2half2_rn(a0, a1), h1 = __floats2half2_rn(a2, a3);
  u.x = *reinterpret_cast<uint32_t *>(&h0);
  u.y = *reinterpret_cast<uint32_t *>(&h1);
  return u;
}
// byte offset of the 4 bf16 / fp16 channels i0..i0+3 (i0 % 4 == 0) of row t
// in a 128-byte-swizzled [t][64] slab
__device__ __forceinline__ uint32_t sw128_off4(uint32_t t, uint32_t i0) {
  return t * 128u + (((((i0 & 63u) >> 3) ^ (t & 7u)) << 4) | ((i0 & 7u) << 1));
}

// X = L^-1 for the lower triangular 64 x 64 fp32 L = diag(s) + strict_lower(T')
// held in sT (row stride LT; only the lower triangle is read), with
// s_t = r_t + T'_tt, into sA (its strict upper triangle zero), by 16 x 16
// blocks: the diagonal blocks D_I = L_II^-1 by forward substitution (one thread
// per column), then the 32 x 32 halves
//   X_10 = -D_1 L_10 D_0,  X_32 = -D_3 L_32 D_2,
// and the lower-left quarter X_21 = -X22 L21 X11 (X11, X22 the 32 x 32
// diagonal halves), each output thread forming four adjacent columns from
// 16-byte loads.  s_t and 1 / s_t go to s_s, s_is.  Called by the kMain
// threads tid = 0 .. kMain - 1 of warps 4-15 (named-barrier synchronisation).
template <class Side>
__device__ __forceinline__ void wy_inverse(int tid, const float *sT, float *sA, float *sX, float *sY,
                                           const float *s_r, float *s_s, float *s_is,
                                           unsigned char *awu, Side side) {
  const int w = tid >> 5;  // main warp 0 .. 11 (lane quarter w & 3)
  if (w == 2 || w == 3) {
    const int st = tid - 64;
    // column c of D_I: x_r = (delta_rc - sum_{m<r} L_rm x_m) / L_rr.  Lane c also forms row c's
    // s_t and its reciprocal, handed round by shuffles; rows are loaded two steps ahead
    const int o = 16 * (st >> 4), c = st & 15;
    const float *tb = sT + o * (LT + 1);
    const float sc = s_r[o + c] + tb[c * (LT + 1)];  // s_t = r_t + sum_i phat k^2 (eq. kla-box-gain)
    const float ic = rcpf(sc);
    s_s[o + c] = sc;
    s_is[o + c] = ic;
    float x[16], row[3][16];
    auto load = [&](int r) {
#pragma unroll
      for (int j = 0; j < 4; ++j)
        if (4 * j < r) {
          const float4 t4 = *reinterpret_cast<const float4 *>(tb + r * LT + 4 * j);
          float *d = row[r % 3] + 4 * j;
          d[0] = t4.x; d[1] = t4.y; d[2] = t4.z; d[3] = t4.w;
        }
    };
    load(1);
    load(2);
#pragma unroll
    for (int r = 0; r < 16; ++r) {
      if (r + 2 < 16 && r > 0) load(r + 2);
      const float inv = __shfl_sync(0xffffffffu, ic, r, 16);
      float acc0 = (r == c) ? 1.f : 0.f, acc1 = 0.f;
#pragma unroll
      for (int m = 0; m < 15; ++m) {
        if (m < r) {
          if (m & 1) acc1 = fmaf(-row[r % 3][m], x[m], acc1);
          else acc0 = fmaf(-row[r % 3][m], x[m], acc0);
        }
      }
      x[r] = (acc0 + acc1) * inv;  // x[r] = 0 for r < c
    }
    float *ab = sA + o * (LT + 1) + c;
#pragma unroll
    for (int r = 0; r < 16; ++r) ab[r * LT] = x[r];
  } else if ((w & 3) < 2) {
    side();  // lane quarters 0, 1
  } else {
    // zero the upper right 16 x 16 blocks of X11 and X22: 2 blocks x 16 rows x 4 float4
    const int z = 32 * (w == 6 ? 0 : w == 7 ? 1 : w == 10 ? 2 : 3) + (tid & 31);
    const int o = 32 * (z >> 6), rr = (z >> 2) & 15, q4 = z & 3;
    *reinterpret_cast<float4 *>(sA + (o + rr) * LT + o + 16 + 4 * q4) = make_float4(0.f, 0.f, 0.f, 0.f);
  }
  bar_sync(kBarMain, kMain);
  // X_10, X_32: one thread per (block, row, 4 columns)
  const int blk = tid >> 6, r2 = (tid >> 2) & 15, cq2 = 4 * (tid & 3);
  const int C0 = 32 * blk, R0 = C0 + 16;
  if (tid < 128) {
    const float *tp = sT + (R0 + r2) * LT + C0;
    float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const float4 t4 = *reinterpret_cast<const float4 *>(tp + 4 * j);
      const float tv[4] = {t4.x, t4.y, t4.z, t4.w};
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const float4 a4 = *reinterpret_cast<const float4 *>(sA + (C0 + 4 * j + u) * LT + C0 + cq2);
        acc.x = fmaf(tv[u], a4.x, acc.x);
        acc.y = fmaf(tv[u], a4.y, acc.y);
        acc.z = fmaf(tv[u], a4.z, acc.z);
        acc.w = fmaf(tv[u], a4.w, acc.w);
      }
    }
    *reinterpret_cast<float4 *>(sX + blk * 256 + r2 * 16 + cq2) = acc;
  }
  bar_sync(kBarMain, kMain);
  if (tid < 128) {
    const float *dp = sA + (R0 + r2) * LT + R0;
    float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const float4 d4 = *reinterpret_cast<const float4 *>(dp + 4 * j);
      const float dv[4] = {d4.x, d4.y, d4.z, d4.w};
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const float4 x4 = *reinterpret_cast<const float4 *>(sX + blk * 256 + (4 * j + u) * 16 + cq2);
        acc.x = fmaf(dv[u], x4.x, acc.x);
        acc.y = fmaf(dv[u], x4.y, acc.y);
        acc.z = fmaf(dv[u], x4.z, acc.z);
        acc.w = fmaf(dv[u], x4.w, acc.w);
      }
    }
    *reinterpret_cast<float4 *>(sA + (R0 + r2) * LT + C0 + cq2) = make_float4(-acc.x, -acc.y, -acc.z, -acc.w);
  }
  bar_sync(kBarMain, kMain);
  // Y = L21 X11 (32 x 32 x 32): one thread per (row, 4 columns), warps 0..3 the left columns,
  // 4..7 the right ones, which need k >= 16 only (X11's upper right quarter is zero)
  if (tid < 256) {
    const int r3 = 8 * (w & 3) + ((tid & 31) >> 2), cq3 = 16 * (w >> 2) + 4 * (tid & 3);
    const float *tp = sT + (32 + r3) * LT;
    float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      if (j < 4 && w >= 4) continue;
      const float4 t4 = *reinterpret_cast<const float4 *>(tp + 4 * j);
      const float tv[4] = {t4.x, t4.y, t4.z, t4.w};
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const float4 a4 = *reinterpret_cast<const float4 *>(sA + (4 * j + u) * LT + cq3);
        acc.x = fmaf(tv[u], a4.x, acc.x);
        acc.y = fmaf(tv[u], a4.y, acc.y);
        acc.z = fmaf(tv[u], a4.z, acc.z);
        acc.w = fmaf(tv[u], a4.w, acc.w);
      }
    }
    *reinterpret_cast<float4 *>(sY + r3 * 32 + cq3) = acc;
  }
  bar_sync(kBarMain, kMain);
  // T' is dead from here on: [A; .] fp16 [128 t][64 s] (A = diag(s) L^-1) is written over it.
  // X_21 = -X22 Y by threads 0..255 (rows 0..15 of X22 end at k = 15), straight to fp16;
  // threads 256..383 convert the rest.
  if (tid < 256) {
    const int r3 = tid >> 3, cq3 = 4 * (tid & 7);
    const float *dp = sA + (32 + r3) * LT + 32;
    float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      if (j >= 4 && w < 4) continue;
      const float4 d4 = *reinterpret_cast<const float4 *>(dp + 4 * j);
      const float dv[4] = {d4.x, d4.y, d4.z, d4.w};
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const float4 y4 = *reinterpret_cast<const float4 *>(sY + (4 * j + u) * 32 + cq3);
        acc.x = fmaf(dv[u], y4.x, acc.x);
        acc.y = fmaf(dv[u], y4.y, acc.y);
        acc.z = fmaf(dv[u], y4.z, acc.z);
        acc.w = fmaf(dv[u], y4.w, acc.w);
      }
    }
    const int r = 32 + r3;
    const float sr = -s_s[r];
    *reinterpret_cast<uint2 *>(awu + chunk_off(r, cq3 >> 3) + 2 * (cq3 & 4)) =
        pack_h4(sr * acc.x, sr * acc.y, sr * acc.z, sr * acc.w);
  } else {
    // rows 0..31 (8 column chunks), rows 32..63 columns 32..63 (4 chunks).  (Rows 64..127 of
    // [A; .] keep what is there: they only reach accumulator rows that nobody reads.)
    for (int e = tid - 256; e < 384; e += 128) {
      const int r = e < 256 ? e >> 3 : 32 + ((e - 256) >> 2), cc = e < 256 ? e & 7 : 4 + (e & 3);
      float v[8];
      const float sr = s_s[r];
      const float4 a0 = *reinterpret_cast<const float4 *>(sA + r * LT + 8 * cc);
      const float4 a1 = *reinterpret_cast<const float4 *>(sA + r * LT + 8 * cc + 4);
      const float av[8] = {a0.x, a0.y, a0.z, a0.w, a1.x, a1.y, a1.z, a1.w};
#pragma unroll
      for (int j = 0; j < 8; ++j) v[j] = (8 * cc + j <= r) ? sr * av[j] : 0.f;
      sm16(awu, chunk_off(r, cc)) = pack_h8(v);
    }
  }
}

// fp32 G_t of the range mode: [64 t][128 i], 512-byte rows, 16-byte groups of four
// channels XOR-swizzled by the row
__device__ __forceinline__ uint32_t g_off(int t, int i4) {
  return (uint32_t)t * 512u + ((uint32_t)(i4 ^ (t & 31)) << 4);
}

// Range mode: a chunk whose cumulative log-decay leaves the range of the
// referenced factors (G_C < -160 in some channel) forms
//   T'_ts   = sum_i k_t,i phat_s,i k_s,i exp(G_t,i - G_s,i)
//   A'qk_ts = tau sum_i q_t,i phat_s,i k_s,i exp(G_t,i - G_s,i)      (s <= t)
// from the cumulative log-decay differences themselves (App. F.2): every ratio
// exp(G_t - G_s), s <= t, lies in (0, 1].  Inputs: raw k, q (bf16 tiles), G (fp32,
// g_off layout) and phat k (fp32 in the layout of the Kk' tile).  Outputs: T' into
// sT and A'_qk into sA (fp32 [64][LT]), zero above the diagonal.  One thread per
// (row t, group of four columns); rows t and 63 - t together have 17 groups.
__device__ __noinline__ void direct_products(int tid, const unsigned char *rk, const unsigned char *rq,
                                                const unsigned char *gbuf, const unsigned char *tb,
                                                float tau, float *sT, float *sA) {
  for (int e = tid; e < 32 * 17; e += kMain) {
    const int pr = e / 17, j = e - 17 * pr, n0 = (pr >> 2) + 1;
    const int t = j < n0 ? pr : 63 - pr;
    const int s0 = 4 * (j < n0 ? j : j - n0);
    float aT[4] = {0.f, 0.f, 0.f, 0.f}, aQ[4] = {0.f, 0.f, 0.f, 0.f};
    for (int i4 = 0; i4 < 32; ++i4) {
      const int i0 = 4 * i4;
      const uint32_t sl8 = (uint32_t)(i0 >> 6) * 8192u;
      float kv[4], qv[4];
      unpack_bf4(*reinterpret_cast<const uint2 *>(rk + sl8 + sw128_off4(t, i0)), kv);
      unpack_bf4(*reinterpret_cast<const uint2 *>(rq + sl8 + sw128_off4(t, i0)), qv);
      const float4 gt = *reinterpret_cast<const float4 *>(gbuf + g_off(t, i4));
      const unsigned char *pkb = tb + (i0 >> 5) * 8192;
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const int sidx = s0 + u;
        const float4 gs = *reinterpret_cast<const float4 *>(gbuf + g_off(sidx, i4));
        const float4 pk = *reinterpret_cast<const float4 *>(pkb + sw32_off(sidx, i0 & 31));
        // columns above the diagonal are clamped to finite values and masked below
        const float e0 = ex2f(fminf(gt.x - gs.x, 0.f) * kLog2e) * pk.x;
        const float e1 = ex2f(fminf(gt.y - gs.y, 0.f) * kLog2e) * pk.y;
        const float e2 = ex2f(fminf(gt.z - gs.z, 0.f) * kLog2e) * pk.z;
        const float e3 = ex2f(fminf(gt.w - gs.w, 0.f) * kLog2e) * pk.w;
        aT[u] = fmaf(kv[0], e0, fmaf(kv[1], e1, fmaf(kv[2], e2, fmaf(kv[3], e3, aT[u]))));
        aQ[u] = fmaf(qv[0], e0, fmaf(qv[1], e1, fmaf(qv[2], e2, fmaf(qv[3], e3, aQ[u]))));
      }
    }
    *reinterpret_cast<float4 *>(sT + t * LT + s0) =
        make_float4(s0 <= t ? aT[0] : 0.f, s0 + 1 <= t ? aT[1] : 0.f, s0 + 2 <= t ? aT[2] : 0.f,
                    s0 + 3 <= t ? aT[3] : 0.f);
    *reinterpret_cast<float4 *>(sA + t * LT + s0) =
        make_float4(s0 <= t ? tau * aQ[0] : 0.f, s0 + 1 <= t ? tau * aQ[1] : 0.f,
                    s0 + 2 <= t ? tau * aQ[2] : 0.f, s0 + 3 <= t ? tau * aQ[3] : 0.f);
  }
  for (int e = tid; e < 64 * 16; e += kMain) {
    const int t = e >> 4, s0 = 4 * (e & 15);
    if (s0 > t) {
      *reinterpret_cast<float4 *>(sT + t * LT + s0) = make_float4(0.f, 0.f, 0.f, 0.f);
      *reinterpret_cast<float4 *>(sA + t * LT + s0) = make_float4(0.f, 0.f, 0.f, 0.f);
    }
  }
}

struct WyParams {
  Args a;
  unsigned char *save_S;  // SV: [BH][NC] context records of the backward
  float *save_p;          // SV: [BH][NC][128] uncertainty carry entering each chunk
  // CH: records of the per-chunk operands (SV: in the context records), what enters every chunk
  unsigned char *pre;
  size_t prec;
  float *pin;             // [BH][NC][128], preset to kUnset
  unsigned *flag;         // per chunk, fstride apart, zeroed: warps that have written their part of its record
  size_t fstride;
  // k_wy_flow: the chunks c0 .. c0 + nc - 1 of every sequence, and the states around them (null: the
  // zero memory, the unit uncertainty; not written)
  int c0, nc;
  const float *S_in, *p_in;
  float *S_out, *p_out;
};

// The uncertainty entering a chunk is handed over as the 4-byte value itself, in place of a
// pattern no result has (a NaN other than the one that arithmetic gives).
constexpr unsigned kUnset = 0xffffffffu;
constexpr uint32_t kFlowWait = 1u << 22;  // polls
__device__ __forceinline__ bool is_unset(float p) { return __float_as_uint(p) == kUnset; }
__device__ __forceinline__ float pin_peek(const float *q) {
  unsigned v;
  asm volatile("ld.relaxed.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(q) : "memory");
  return __uint_as_float(v);
}
__device__ __forceinline__ bool pin_get(const float *q, float *p) {
  for (uint32_t n = 0; n < kFlowWait; ++n) {
    *p = pin_peek(q);
    if (!is_unset(*p)) return true;
    if (n > 64) __nanosleep(32);
  }
  return false;
}
__device__ __forceinline__ void pin_put(float *q, float p) {
  const unsigned v = is_unset(p) ? 0x7fffffffu : __float_as_uint(p);
  asm volatile("st.relaxed.gpu.global.u32 [%0], %1;" ::"l"(q), "r"(v) : "memory");
}
// One count per warp once its stores to a record are visible; a reader waits for all of them.
constexpr unsigned kFlowWarps = WT / 32;
__device__ __forceinline__ void publish(unsigned *flag) {
  __threadfence();
  __syncwarp();
  if ((threadIdx.x & 31) == 0) asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(flag) : "memory");
}
__device__ __forceinline__ bool flow_wait(const unsigned *flag) {
  for (uint32_t n = 0; n < kFlowWait; ++n) {
    unsigned v;
    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(flag) : "memory");
    if (v >= kFlowWarps) return true;
    if (n > 64) __nanosleep(32);
  }
  return false;
}

// Per-chunk operands that k_wy_flow's chunk part leaves for its memory part, in a record of their
// own or (SV) in the context record: [-Kbar; Qbar] fp16 32 KB, K'^T fp16 [128 i][64 s] 16 KB, A
// fp16 8 KB, A'_qk fp16 8 KB, gamma_C [128], s_t [64].  In the context the first two and A'_qk lie where
// S_in, Y and R go, which the memory part writes once it has read them.
constexpr size_t kPreBytes = 66560;
template <int SV>
struct Pre {
  static constexpr int KQ = SV ? kCtxS : 0, Kt = SV ? kCtxY : 32768, A = SV ? kCtxA : 49152;
  static constexpr int Aq = SV ? kCtxR : 57344, gC = SV ? kCtxGa + 63 * D * 4 : 65536, s = SV ? kCtxTok : 66048;
};

// SV: besides o, S_T and p_T (each written when its pointer is non-null), keep
// the chunked backward's context: per chunk the fp16 tiles S_in, R, -W, A_qk,
// A = (I + T)^-1 and Y = V - Kbar S_in in the 128-byte-swizzled layout of the
// fused backward (all but A_qk staged in shared memory and bulk-copied),
// phat and gamma in float32 [64 t][128 i], s_t per token, and the uncertainty
// entering the chunk.  The arithmetic is the same with and without it.

// CH: the part of this work that needs no memory S, for the chunks block, block + nblocks, ..
// of all sequences, its results left in records for wy_state; the uncertainty entering
// each chunk comes from wy_gain.  The same instructions, so the same bits.
template <int SV, int LG, int CH>  // LG: g, omega, r hold the logits x, y, z of the gates
__device__ __forceinline__ void wy_body(const CUtensorMap &mk, const CUtensorMap &mg, const CUtensorMap &mw,
                                        const CUtensorMap &mv, const CUtensorMap &mq, const WyParams &P,
                                        const int block, const int nblocks) {
  const Args &a = P.a;
  extern __shared__ unsigned char smraw[];
  unsigned char *sm =
      reinterpret_cast<unsigned char *>((reinterpret_cast<uintptr_t>(smraw) + 1023) & ~uintptr_t(1023));
  unsigned char *rk = sm + O_RK, *rg = sm + O_RG, *rw = sm + O_RW, *vr = sm + O_V, *rq = sm + O_Q;
  unsigned char *ta = sm + O_TA, *tb = sm + O_TB, *as1 = sm + O_AS1;
  unsigned char *s16 = sm + O_S16, *awu = sm + O_AWU;
  float *sT = reinterpret_cast<float *>(sm + O_SWT), *sA = reinterpret_cast<float *>(sm + O_SWA);
  unsigned char *wst = sm + O_SWA;  // context: -W fp16 staged over L^-1 after the solve
  float *sX = reinterpret_cast<float *>(sm + O_SX), *sY = reinterpret_cast<float *>(sm + O_SY);
  float *sf = reinterpret_cast<float *>(sm + O_SMALL);
  float *s_r = sf + SM_R, *s_mur = sf + SM_MUR, *s_s = sf + SM_S, *s_is = sf + SM_IS;
  float *s_c = sf + SM_C, *s_gC = sf + SM_GC, *s_part = sf + SM_PART;
  // per chunk (slot c & 1): some channel's decay left the range of the referenced factors
  int *s_oor = reinterpret_cast<int *>(sf + SM_OOR);
  uint64_t *bars = reinterpret_cast<uint64_t *>(sm + O_BAR);
  uint64_t *bar_raw = bars, *bar_v = bars + 1, *bar_mma = bars + 2, *bar_q = bars + 3;
  uint64_t *bar_t = bars + 4;  // MMA-T completions (one a chunk)
  uint64_t *bar_w = bars + 5;  // MMA-W completions (context mode only, one a chunk)
  uint32_t *s_tbase = reinterpret_cast<uint32_t *>(bars + 6);

  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int wq = warp & 3, wg = warp >> 2;  // TMEM lane quarter, column group
  const int bh = block;  // (not CH)
  const int NCs = CH ? P.nc : (a.T + CM - 1) / CM, BH = a.B * a.H;
  // chunks of this CTA, counted by `c` below; ct, b, h: a chunk's place in its sequence
  const int NC = CH ? (NCs * BH - block + nblocks - 1) / nblocks : NCs;
  struct Job { int ct, b, h; size_t rc; };
  auto job = [&](int c) {
    Job o;
    const int j = CH ? block + c * nblocks : 0, q = CH ? j % BH : bh;
    o.ct = CH ? j / BH : c;
    o.b = q / a.H;
    o.h = q % a.H;
    o.rc = (size_t)q * NCs + o.ct;
    if (CH) o.ct += P.c0;
    return o;
  };
  const bool issuer = tid == 128;  // copies; the MMAs: its whole warp with an elected lane
  const int warp_u = __shfl_sync(0xffffffffu, warp, 0);
  const uint32_t lane_base = (uint32_t)(32 * wq) << 16;

  if (issuer) {
    mbar_init(bar_raw, 1);
    mbar_init(bar_v, 1);
    mbar_init(bar_mma, 1);
    mbar_init(bar_q, 1);
    mbar_init(bar_t, 1);
    mbar_init(bar_w, 1);
    fence_mbar_init();
    prefetch_tmap(&mk);
    prefetch_tmap(&mg);
    prefetch_tmap(&mw);
    prefetch_tmap(&mv);
    prefetch_tmap(&mq);
  }
  if (warp == 0) {
    tmem_alloc(s_tbase, 512);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tbase = *s_tbase;
  const uint32_t TS = tbase + TC_S, TD1 = tbase + TC_D1, TKT = tbase + TC_KT, TW = tbase + TC_W,
                 TU = tbase + TC_U;

  // k, g, omega of chunk c (the gain and the preparing pass), q of chunk c (the
  // preparing pass), V of chunk c (once MMA-O / MMA-S2 of chunk c - 1 has read R')
  auto issue_raw = [&](const Job &o) {
    mbar_expect_tx(bar_raw, 49152);
    for (int s = 0; s < 2; ++s) {
      tma_load_4d(rk + s * 8192, &mk, bar_raw, 64 * s, o.h, o.ct * CM, o.b);
      tma_load_4d(rg + s * 8192, &mg, bar_raw, 64 * s, o.h, o.ct * CM, o.b);
      tma_load_4d(rw + s * 8192, &mw, bar_raw, 64 * s, o.h, o.ct * CM, o.b);
    }
  };
  auto issue_q = [&](const Job &o) {
    mbar_expect_tx(bar_q, 16384);
    for (int s = 0; s < 2; ++s) tma_load_4d(rq + s * 8192, &mq, bar_q, 64 * s, o.h, o.ct * CM, o.b);
  };
  auto issue_v = [&](const Job &o) {
    mbar_expect_tx(bar_v, 16384);
    for (int s = 0; s < 2; ++s) tma_load_4d(vr + s * 8192, &mv, bar_v, 64 * s, o.h, o.ct * CM, o.b);
  };
  auto prefetch = [&](const Job &o) {  // k, g, omega, q into L2
    for (int s = 0; s < 2; ++s) {
      tma_prefetch_4d(&mk, 64 * s, o.h, o.ct * CM, o.b);
      tma_prefetch_4d(&mg, 64 * s, o.h, o.ct * CM, o.b);
      tma_prefetch_4d(&mw, 64 * s, o.h, o.ct * CM, o.b);
      tma_prefetch_4d(&mq, 64 * s, o.h, o.ct * CM, o.b);
    }
  };
  if (issuer && NC > 0) {
    issue_raw(job(0));
    issue_q(job(0));
    if (!CH) issue_v(job(0));
    if (NC > 1) prefetch(job(1));
  }

  // initial memory S_0 -> TMEM (row = key channel i, column = value j)
  if constexpr (!CH) {
    const int i = 32 * wq + lane;
    for (int c0 = 0; c0 < 32; c0 += 16) {
      float v[16];
      const int j0 = 32 * wg + c0;
      if (a.S0) {
        const float4 *src = reinterpret_cast<const float4 *>(a.S0 + ((size_t)bh * D + i) * D + j0);
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          const float4 x = src[u];
          v[4 * u] = x.x; v[4 * u + 1] = x.y; v[4 * u + 2] = x.z; v[4 * u + 3] = x.w;
        }
      } else {
#pragma unroll
        for (int u = 0; u < 16; ++u) v[u] = 0.f;
      }
      tmem_st16(TS + lane_base + j0, v);
    }
    tmem_st_wait();
  }

  // roles: warps 0-3 run the gain one chunk ahead; warps 4-15 (the main warps)
  // prepare the operands (warps 4-11), store o (warps 14, 15), and run every
  // tensor-core and solve stage, synchronised among themselves by named barriers
  const bool gain = tid < 128;
  const bool prep = tid >= 128 && tid < 128 + kPrepThreads;
  const int mt = tid - 128;           // main thread 0 .. kMain - 1
  const int wgm = (warp >> 2) - 1;    // main warps: 0, 1, 2 within a lane quarter
  float p = 1.f;                      // gain threads: uncertainty carry of channel tid
  if (!CH && gain && a.p0) p = a.p0[(size_t)bh * D + tid];
  // gain threads tid < 64: the r input of the next chunk's token tid, converted when it is
  // used (a conversion here would wait for the load)
  __nv_bfloat16 znext = __float2bfloat16_rn(0.f);
  float pnext = 1.f;  // CH: the uncertainty entering the next chunk
  auto load_r = [&](int c) {
    if (c >= NC) return;
    const Job o = job(c);
    if (tid < CM) znext = static_cast<const __nv_bfloat16 *>(a.r)[tok_index(a, o.b, min(o.ct * CM + tid, a.T - 1), o.h)];
    if (CH && gain) pnext = pin_peek(P.pin + o.rc * D + tid);
  };
  load_r(0);

  uint32_t mph = 0;  // main threads: completions of bar_mma observed (three per chunk:
                     // MMA-KS, MMA-R, MMA-O / MMA-S2)
  auto mma_wait_main = [&]() -> bool {
    const bool r = mbar_wait(bar_mma, mph & 1, kWait);
    ++mph;
    return r;
  };
  const uint32_t id_T = idesc_tf32(128, 64);
  const uint32_t id_16 = idesc_f16(128, 128, 0, 1);  // A K-major, B MN-major

  // ---- the gain of chunk c (warps 0-3): r and mu / r of its tokens into buffer
  //      c & 1, the recursion over its 64 tokens.  Its Kk' tile may be written
  //      once MMA-T of chunk c - 1 has read the previous one.
  auto gain_chunk = [&](int c) -> bool {
    const int i = tid, sb = c & 1;
    const Job o = job(c);
    const int left = a.T - o.ct * CM;  // tokens of the sequence from this chunk on
    bool g_in = true;
    if (CH) {
      if (is_unset(pnext)) g_in = pin_get(P.pin + o.rc * D + i, &pnext);
      p = pnext;
    }
    float *sr = s_r + 64 * sb, *smur = s_mur + 64 * sb;
    if (tid < CM) {
      const bool live = tid < left;
      const float z = live ? __bfloat162float(znext) : 0.f;
      const float r = !live ? 1.f : LG ? a.rmin + softplus_w(z) : z;  // r = r_min + softplus(z) (Sec. 5)
      sr[tid] = r;
      smur[tid] = a.mu / r;
    }
    load_r(c + 1);
    bar_sync(kBarGain, 128);
    bool g_ok = mbar_wait(bar_raw, c & 1, kWait) && g_in;
    const unsigned char *pg = rg + (i >> 6) * 8192, *pw = rw + (i >> 6) * 8192, *pk = rk + (i >> 6) * 8192;
    const int cl = i & 63;
    // element (t, i) of a raw slab: row t, 128-byte swizzle
    auto raw = [&](const unsigned char *base, int t) {
      return __bfloat162float(*reinterpret_cast<const __nv_bfloat16 *>(base + sw128_off(t, cl)));
    };
    // log alpha and omega from the tile's values
    auto lga = [&](float x) { return LG ? -softplus_w(-x) : x; };
    auto omg = [&](float y) { return LG ? softplus_w(y) : y; };
    // logit gates: the tokens past T must be identity updates (alpha = 1, omega = 0).
    // Their rows of the g and omega tiles, zero-filled by TMA, get the logits +-1e30,
    // whose activations are exactly those (softplus(-1e30) = 0), so that no pass
    // masks its elements; the preparing pass reads the same rows
    if (LG && left < CM) {
      const __nv_bfloat16 big = __float2bfloat16_rn(1e30f), nbig = __float2bfloat16_rn(-1e30f);
      for (int t = left; t < CM; ++t) {
        *reinterpret_cast<__nv_bfloat16 *>(rg + (i >> 6) * 8192 + sw128_off(t, cl)) = big;
        *reinterpret_cast<__nv_bfloat16 *>(rw + (i >> 6) * 8192 + sw128_off(t, cl)) = nbig;
      }
    }
    unsigned char *pb = tb + (i >> 5) * 8192;
    const int cb = i & 31;
    // logit gates: log alpha is formed once per element here and kept (fp32) in this
    // channel's column of the Kk' tile, which the loop below overwrites token by token
    // after reading it; the tile is free once MMA-T of chunk c - 1 has read it
    if (LG && c > 0) g_ok = mbar_wait(bar_t, (c - 1) & 1, kWait) && g_ok;
    auto lga_t = [&](int t) {  // log alpha of token t in the loop
      return LG ? *reinterpret_cast<const float *>(pb + sw32_off(t, cb)) : lga(raw(pg, t));
    };
    // G_C, and the sums of the chunk's eight 8-token segments for the preparing pass
    // (which reads them at the next chunk boundary; it is done with the previous chunk's)
    // (logit gates: 16 tokens at a time, their loads ahead of the stores of log alpha,
    // which the compiler must otherwise keep in order with the next loads)
    float GC = 0.f;
    if constexpr (!LG) {
#pragma unroll
      for (int sg = 0; sg < 8; ++sg) {
        const int t = 8 * sg;
        const float ss = ((raw(pg, t) + raw(pg, t + 1)) + (raw(pg, t + 2) + raw(pg, t + 3))) +
                         ((raw(pg, t + 4) + raw(pg, t + 5)) + (raw(pg, t + 6) + raw(pg, t + 7)));
        s_part[sg * D + i] = ss;
        GC += ss;
      }
    } else {
#pragma unroll
      for (int s2 = 0; s2 < 4; ++s2) {
        float x[16];
#pragma unroll
        for (int j = 0; j < 16; ++j) x[j] = lga(raw(pg, 16 * s2 + j));
#pragma unroll
        for (int h2 = 0; h2 < 2; ++h2) {
          const float *y = x + 8 * h2;
          const float ss = ((y[0] + y[1]) + (y[2] + y[3])) + ((y[4] + y[5]) + (y[6] + y[7]));
          s_part[(2 * s2 + h2) * D + i] = ss;
          GC += ss;
        }
#pragma unroll
        for (int j = 0; j < 16; ++j) *reinterpret_cast<float *>(pb + sw32_off(16 * s2 + j, cb)) = x[j];
      }
    }
    const float cref = 0.5f * GC;
    s_c[i] = cref;
    // out of the referenced factors' range in some channel: this chunk forms T' and A'_qk
    // from exp(G_t - G_s) directly
    // (the training forward keeps the referenced form: its context feeds a backward
    // that needs exp(G_C) >= 1e-36, and such chunks are reported instead)
    const bool oor = !SV && bar_or(kBarGain, 128, cref < kMinHalfG);
    if (tid == 0) s_oor[sb] = oor ? 1 : 0;
    float Gt = 0.f;  // G_t of this channel (range mode)
    unsigned char *gctx = SV ? P.save_S + o.rc * kCtxBytes : nullptr;
    unsigned char *gpre = CH ? P.pre + o.rc * P.prec : gctx;
    if (SV && !CH) P.save_p[o.rc * D + i] = p;
    float *cph = SV ? reinterpret_cast<float *>(gctx + kCtxPh) + i : nullptr;
    float f = ex2f(cref * kLog2e);                // exp(c - G_t), G_{-1} = 0
    const float E2 = ex2f((GC - cref) * kLog2e);  // exp(G_C - c)
    const uint32_t tkt = TKT + (uint32_t)((c & 1) * 32);
    float gb[8], wb[8], kb8[8], mb[8];
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      gb[j] = lga_t(j);
      wb[j] = omg(raw(pw, j));
      kb8[j] = raw(pk, j);
    }
    {
      const float4 m0 = *reinterpret_cast<const float4 *>(smur), m1 = *reinterpret_cast<const float4 *>(smur + 4);
      mb[0] = m0.x; mb[1] = m0.y; mb[2] = m0.z; mb[3] = m0.w; mb[4] = m1.x; mb[5] = m1.y; mb[6] = m1.z; mb[7] = m1.w;
    }
    if (!LG && c > 0) g_ok = mbar_wait(bar_t, (c - 1) & 1, kWait) && g_ok;  // Kk' of chunk c - 1 has been read
    // the chunk in blocks of 8 tokens; the next block's inputs are loaded
    // before the current block's outputs are stored
    if (oor) {
      // range mode (rare): Kk' is replaced by phat k itself, and K' is formed from G_t
      // directly; a compact loop without the prefetching of the referenced mode
#pragma unroll 1
      for (int blk = 0; blk < 8; ++blk) {
        uint32_t kt[4];
#pragma unroll
        for (int j = 0; j < 8; ++j) {
          const int t = 8 * blk + j;
          const float lg = lga_t(t), kk = raw(pk, t);
          const float al = ex2f(lg * kLog2e);
          const float ph = fmaf(al * al, p, omg(raw(pw, t)));
          const float den = fmaf(kk * kk * smur[t], ph, 1.f);
          p = ph * rcpf(den);
          Gt += lg;
          const float pkv = ph * kk;
          if (SV) cph[t * D] = ph;
          *reinterpret_cast<float *>(pb + sw32_off(t, cb)) = pkv;
          const uint32_t hb =
              (uint32_t)__half_as_ushort(__float2half_rn(pkv * ex2f((GC - Gt) * kLog2e)));
          if ((j & 1) == 0) kt[j >> 1] = hb;
          else kt[j >> 1] |= hb << 16;
        }
        if (CH) *reinterpret_cast<uint4 *>(gpre + Pre<SV>::Kt + chunk_off(i, blk)) = make_uint4(kt[0], kt[1], kt[2], kt[3]);
        else tmem_st4u(tkt + lane_base + (uint32_t)(4 * blk), kt);
      }
    } else {
#pragma unroll
      for (int blk = 0; blk < 8; ++blk) {
        float gn[8], wn[8], kn[8], mn[8];
        if (blk < 7) {
#pragma unroll
          for (int j = 0; j < 8; ++j) {
            const int t = 8 * (blk + 1) + j;
            gn[j] = lga_t(t);
            wn[j] = omg(raw(pw, t));
            kn[j] = raw(pk, t);
          }
          const float4 m0 = *reinterpret_cast<const float4 *>(smur + 8 * (blk + 1));
          const float4 m1 = *reinterpret_cast<const float4 *>(smur + 8 * (blk + 1) + 4);
          mn[0] = m0.x; mn[1] = m0.y; mn[2] = m0.z; mn[3] = m0.w; mn[4] = m1.x; mn[5] = m1.y; mn[6] = m1.z; mn[7] = m1.w;
        }
        uint32_t kt[4];
#pragma unroll
        for (int j = 0; j < 8; ++j) {
          const int t = 8 * blk + j;
          const float al = ex2f(gb[j] * kLog2e), a2 = al * al;
          const float ph = fmaf(a2, p, wb[j]);               // eq. diag-covariance-prediction
          const float u = kb8[j] * kb8[j] * mb[j];
          const float den = fmaf(u, ph, 1.f);
          const float x = rcpf(al * den);
          p = ph * (x * al);                                  // eq. prefix-diag-uncertainty
          f *= x * den;                                       // / alpha_t
          const float pkv = ph * kb8[j];
          if (SV) cph[t * D] = ph;
          *reinterpret_cast<float *>(pb + sw32_off(t, cb)) = tf32r(pkv * f);
          const uint32_t hb = (uint32_t)__half_as_ushort(__float2half_rn(pkv * (f * E2)));
          if ((j & 1) == 0) kt[j >> 1] = hb;
          else kt[j >> 1] |= hb << 16;
        }
        if (!CH) tmem_st4u(tkt + lane_base + (uint32_t)(4 * blk), kt);
        if (CH)
          *reinterpret_cast<uint4 *>(gpre + Pre<SV>::Kt + chunk_off(i, blk)) = make_uint4(kt[0], kt[1], kt[2], kt[3]);
        if (blk < 7) {
#pragma unroll
          for (int j = 0; j < 8; ++j) {
            gb[j] = gn[j];
            wb[j] = wn[j];
            kb8[j] = kn[j];
            mb[j] = mn[j];
          }
        }
      }
    }
    tmem_st_wait();
    fence_proxy_async();
    if (CH) publish(P.flag + o.rc * P.fstride);  // K'^T
    return g_ok;
  };

  bool mine = true;    // this thread's waits so far; combined at the CTA-wide barriers
  bool failed = false;
  if (gain && NC > 0) mine = gain_chunk(0);

  for (int c = 0; c < NC; ++c) {
    const uint32_t tkt = TKT + (uint32_t)((c & 1) * 32);
    const Job o = job(c);
    unsigned char *ctx = SV ? P.save_S + o.rc * kCtxBytes : nullptr;
    unsigned char *pre = CH ? P.pre + o.rc * P.prec : ctx;
    if ((SV || CH) && lane == 0) bulk_wait_read();  // the previous chunk's context tiles have left shared memory
    // ---- [0] the previous chunk's MMA-O / MMA-S2 must be done before V is brought
    //          into its R' buffer; the gain of this chunk is done (its warps arrive here)
    if (!gain) mine = mbar_wait(bar_raw, c & 1, kWait) && mine;
    if (!CH && issuer && c > 0) {
      mine = mma_wait_main() && mine;  // MMA-O / MMA-S2 of chunk c - 1
      if (mine) issue_v(o);
    } else if (!gain && c > 0) {
      ++mph;
    }
    tc_fence_before();
    if (!__syncthreads_and(mine)) {
      failed = true;
      break;
    }
    tc_fence_after();

    // ---- [1] operand preparation (warps 4-11) and the previous chunk's output
    //          (warps 14, 15); the gain of this chunk is already done
    if (prep) {
      const int pi = mt;
      const int i0 = 4 * (pi & 31), seg = pi >> 5, t0 = 8 * seg;
      const uint32_t sl8 = (uint32_t)(i0 >> 6) * 8192u;  // 64-channel slab of a [t][64] 16-bit tile
      // the chunk's g for this thread's 8 tokens and 4 channels (8 bytes a token)
      uint2 gq[8];
      const bool oor = !SV && s_oor[c & 1] != 0;
      // (logit gates: the rows past T hold logits whose log alpha is exactly 0)
      auto unpack_lga = [&](uint2 u, float *gv) {
        unpack_bf4(u, gv);
        if (LG) {
#pragma unroll
          for (int w = 0; w < 4; ++w) gv[w] = -softplus_w(-gv[w]);
        }
      };
#pragma unroll
      for (int j = 0; j < 8; ++j) gq[j] = *reinterpret_cast<const uint2 *>(rg + sl8 + sw128_off4(t0 + j, i0));
      // G at the start of this thread's segment from the segment sums the gain formed
      float cr[4], G[4] = {0.f, 0.f, 0.f, 0.f}, Ec[4], gm[4];
      {
        const float4 c4 = *reinterpret_cast<const float4 *>(s_c + i0);
        cr[0] = c4.x; cr[1] = c4.y; cr[2] = c4.z; cr[3] = c4.w;
      }
      for (int s2 = 0; s2 < seg; ++s2) {
        const float4 p4 = *reinterpret_cast<const float4 *>(s_part + s2 * D + i0);
        G[0] += p4.x; G[1] += p4.y; G[2] += p4.z; G[3] += p4.w;
      }
#pragma unroll
      for (int u = 0; u < 4; ++u) Ec[u] = ex2f(cr[u] * kLog2e);
      mine = mbar_wait(bar_q, c & 1, kWait) && mine;
      unsigned char *pa = ta + (i0 >> 5) * 16384, *pqh = as1 + (i0 >> 6) * 16384;
      const int cc = i0 & 31;
      auto prep_loop = [&](auto range_mode) {
        constexpr bool RM = decltype(range_mode)::value;
#pragma unroll
        for (int j = 0; j < 8; ++j) {
          const int t = t0 + j;
          float gv[4], kv[4], qv[4], e[4];
          unpack_lga(gq[j], gv);
          unpack_bf4(*reinterpret_cast<const uint2 *>(rk + sl8 + sw128_off4(t, i0)), kv);
          unpack_bf4(*reinterpret_cast<const uint2 *>(rq + sl8 + sw128_off4(t, i0)), qv);
          if constexpr (RM) {  // G_t itself for the direct products; gamma_t = exp(G_t) (may underflow)
#pragma unroll
            for (int u = 0; u < 4; ++u) {
              G[u] += gv[u];
              gm[u] = ex2f(G[u] * kLog2e);
              qv[u] *= a.tau;
            }
            *reinterpret_cast<float4 *>(ta + g_off(t, i0 >> 2)) = make_float4(G[0], G[1], G[2], G[3]);
          } else {
#pragma unroll
            for (int u = 0; u < 4; ++u) {
              G[u] += gv[u];
              e[u] = ex2f((G[u] - cr[u]) * kLog2e);
              gm[u] = e[u] * Ec[u];
              qv[u] *= a.tau;
            }
            *reinterpret_cast<float4 *>(pa + sw32_off(t, cc)) =
                make_float4(tf32r(e[0] * kv[0]), tf32r(e[1] * kv[1]), tf32r(e[2] * kv[2]), tf32r(e[3] * kv[3]));
            *reinterpret_cast<float4 *>(pa + sw32_off(64 + t, cc)) =
                make_float4(tf32r(e[0] * qv[0]), tf32r(e[1] * qv[1]), tf32r(e[2] * qv[2]), tf32r(e[3] * qv[3]));
          }
          *reinterpret_cast<uint2 *>(pqh + sw128_off4(t, i0)) =
              pack_h4(-gm[0] * kv[0], -gm[1] * kv[1], -gm[2] * kv[2], -gm[3] * kv[3]);
          *reinterpret_cast<uint2 *>(pqh + sw128_off4(64 + t, i0)) =
              pack_h4(gm[0] * qv[0], gm[1] * qv[1], gm[2] * qv[2], gm[3] * qv[3]);
          if (SV)
            *reinterpret_cast<float4 *>(reinterpret_cast<float *>(ctx + kCtxGa) + t * D + i0) =
                make_float4(gm[0], gm[1], gm[2], gm[3]);
        }
      };
      if (oor) prep_loop(std::true_type{});
      else prep_loop(std::false_type{});
      if (seg == 7) {
        *reinterpret_cast<float4 *>(s_gC + i0) = make_float4(gm[0], gm[1], gm[2], gm[3]);
        // the fused backward divides by the saved gamma: it needs gamma_C >= 1e-36
        if (SV)
          for (int u = 0; u < 4; ++u) check_gamma_range(gm[u], a.status);
      }
    } else if (!CH && !gain && wq >= 2 && wgm == 2 && c > 0 && a.o) {  // warps 14, 15: O of chunk c - 1
      const int t = 32 * (wq - 2) + lane, tt = (c - 1) * CM + t;
      for (int j0 = 0; j0 < D; j0 += 16) {
        float v[16];
        tmem_ld16(TU + lane_base + j0, v);
        if (tt < a.T) {
          const size_t base = tok_index(a, o.b, tt, o.h) * D + j0;
          if (a.odt == KDN_BF16) {
            uint4 *dst = reinterpret_cast<uint4 *>(static_cast<__nv_bfloat16 *>(a.o) + base);
            dst[0] = pack_bf8(v);
            dst[1] = pack_bf8(v + 8);
          } else {
            float4 *dst = reinterpret_cast<float4 *>(static_cast<float *>(a.o) + base);
#pragma unroll
            for (int u = 0; u < 4; ++u) dst[u] = make_float4(v[4 * u], v[4 * u + 1], v[4 * u + 2], v[4 * u + 3]);
          }
        }
      }
    }
    fence_proxy_async();
    tc_fence_before();
    if (!__syncthreads_and(mine)) {
      failed = true;
      break;
    }

    // ---- [2] MMA-T; the next chunk's k, g, omega and q.  In range mode the main
    //          warps form T' and A'_qk on the CUDA cores instead, and the issuer
    //          completes the MMA-T barrier's phase by hand once they are done.
    const bool oor = !SV && s_oor[c & 1] != 0;
    auto issue_next = [&]() {
      if (c + 1 < NC) {
        const Job n = job(c + 1);
        issue_raw(n);
        issue_q(n);
        if (!CH)
          for (int s = 0; s < 2; ++s) tma_prefetch_4d(&mv, 64 * s, n.h, n.ct * CM, n.b);
      }
      if (c + 2 < NC) prefetch(job(c + 2));  // into L2: its tiles are loaded during chunk c + 1
    };
    if (warp_u == 4 && !oor) {
      tc_fence_after();
      const uint32_t lead = elect_one();
      const uint64_t A0 = sw128_desc(smem_u32(ta), 16, 1024), B0 = sw128_desc(smem_u32(tb), 16, 1024);
#pragma unroll
      for (int kk = 0; kk < 16; ++kk)
        umma_tf32(lead, TD1, step(A0, (kk >> 2) * 16384 + (kk & 3) * 32),
                  step(B0, (kk >> 2) * 8192 + (kk & 3) * 32), id_T, kk > 0);
      commit_if(lead, bar_t);
    }
    // the next chunk's tiles (the raw tiles are free: the preparing pass is done), from a
    // main thread outside the MMA issuer's warp: its ~20 TMA operations then overlap
    // MMA-T, for which every main warp waits anyway
    if (tid == kTmaThread && !oor) issue_next();
    if (gain) {
      // the next chunk's gain, overlapping this chunk's remaining stages
      if (c + 1 < NC) mine = gain_chunk(c + 1) && mine;
      continue;
    }
    if (oor) {
      direct_products(mt, rk, rq, ta, tb, a.tau, sT, sA);
      bar_sync(kBarMain, kMain);
      if (issuer) {  // the raw tiles and phat k have been read
        mbar_arrive(bar_t);
        issue_next();
      }
    }
    mine = mbar_wait(bar_t, c & 1, kWait) && mine;
    tc_fence_after();

    // ---- [3] T' (with its diagonal) out of TMEM; A'_qk -> fp16 pairs in place (the
    //          A operand of MMA-O); S_in -> fp16; V -> fp16
    if (wq < 2 && !oor) {  // T' rows 0..63, lower triangle with the diagonal -> fp32 tile
      const int t = 32 * wq + lane;
      for (int g = wgm; g < 4; g += 3) {
        const int s0 = 16 * g;
        float v[16];
        tmem_ld16(TD1 + lane_base + s0, v);
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          float4 o;
          o.x = (s0 + 4 * u + 0 <= t) ? v[4 * u + 0] : 0.f;
          o.y = (s0 + 4 * u + 1 <= t) ? v[4 * u + 1] : 0.f;
          o.z = (s0 + 4 * u + 2 <= t) ? v[4 * u + 2] : 0.f;
          o.w = (s0 + 4 * u + 3 <= t) ? v[4 * u + 3] : 0.f;
          *reinterpret_cast<float4 *>(sT + t * LT + s0 + 4 * u) = o;
        }
      }
    } else if (wgm == 0 && wq >= 2) {
      // A'_qk rows 64..127, lower triangle: columns 16g .. 16g + 15 -> fp16 pairs in
      // columns 8g .. 8g + 7 (each column is read before it is overwritten)
      const int t = 32 * (wq - 2) + lane;
      for (int g = 0; g < 4; ++g) {
        float v[16], hv[8];
        if (oor) {
#pragma unroll
          for (int u = 0; u < 4; ++u) {
            const float4 x4 = *reinterpret_cast<const float4 *>(sA + t * LT + 16 * g + 4 * u);
            v[4 * u] = x4.x; v[4 * u + 1] = x4.y; v[4 * u + 2] = x4.z; v[4 * u + 3] = x4.w;
          }
        } else {
          tmem_ld16(TD1 + lane_base + 16 * g, v);
        }
#pragma unroll
        for (int j = 0; j < 8; ++j) {
          const __half2 h2 = __floats2half2_rn((16 * g + 2 * j <= t) ? v[2 * j] : 0.f,
                                               (16 * g + 2 * j + 1 <= t) ? v[2 * j + 1] : 0.f);
          hv[j] = __uint_as_float(*reinterpret_cast<const uint32_t *>(&h2));
        }
        if (CH) {
#pragma unroll
          for (int w = 0; w < 2; ++w)
            *reinterpret_cast<float4 *>(pre + Pre<SV>::Aq + chunk_off(t, 2 * g + w)) =
                make_float4(hv[4 * w], hv[4 * w + 1], hv[4 * w + 2], hv[4 * w + 3]);
        }
        if (!CH || SV) tmem_st8(TD1 + lane_base + 8 * g, hv);
      }
    }
    if (CH && !SV && mt < D) reinterpret_cast<float *>(pre + Pre<SV>::gC)[mt] = s_gC[mt];
    if constexpr (!CH) {  // S_in -> fp16 (MN-major B of MMA-KS); diag(gamma_C) S_in back to TMEM
      const int i = 32 * wq + lane;
      const float gC = s_gC[i];
      for (int g = wgm; g < 8; g += 3) {
        float v[16];
        const int j0 = 16 * g, sl = j0 >> 6, cc0 = (j0 & 63) >> 3;
        tmem_ld16(TS + lane_base + j0, v);
        sm16(s16, sl * 16384 + chunk_off(i, cc0)) = pack_h8(v);
        sm16(s16, sl * 16384 + chunk_off(i, cc0 + 1)) = pack_h8(v + 8);
#pragma unroll
        for (int u = 0; u < 16; ++u) v[u] *= gC;
        tmem_st16(TS + lane_base + j0, v);
      }
    }
    tmem_st_wait();
    fence_proxy_async();
    tc_fence_before();
    bar_sync(kBarMain, kMain);
    tc_fence_after();
    // MMA-KS: TU = [-Kbar; Qbar] S_in (fp16), while the CUDA cores solve
    if (!CH && warp_u == 4) {
      const uint32_t lead = elect_one();
      const uint64_t A1 = sw128_desc(smem_u32(as1), 16, 1024), B1 = sw128_desc(smem_u32(s16), 16384, 1024);
#pragma unroll
      for (int kk = 0; kk < 8; ++kk)
        umma_if(lead, TU, step(A1, (kk >> 2) * 16384 + (kk & 3) * 32), step(B1, kk * 2048), id_16, kk > 0);
      commit_if(lead, bar_mma);
    }
    // (the copies of the context tiles are issued one per warp, by warps with nothing else to
    // do at that point: each costs its warp a few hundred cycles)
    if (CH && lane == 0 && (warp == 11 || warp == 14)) {
      bulk_s2g(pre + Pre<SV>::KQ + (warp == 14) * 16384, as1 + (warp == 14) * 16384, 16384);
      bulk_commit();
    } else if (!CH && SV && lane == 0) {
      if (warp == 10) bulk_s2g(ctx + kCtxS, s16, 32768);
      bulk_commit();
    }

    // ---- [4] A = (I + T)^-1 = diag(s) L^-1 with L = diag(s) + strict_lower(T')
    //          (T = strict_lower(T') diag(1/s)), then [A; .] fp16 over T';
    //          Y = V - Kbar S_in (rows 0..63 of TU plus V) -> fp16 in place over V, by warps
    //          4, 5, 8, 9, 12, 13 while warps 6, 7 solve the diagonal blocks
    {
      auto y_side = [&]() {
        if (CH) return;
        const bool ks_ok = mma_wait_main();  // MMA-KS
        const bool v_ok = mbar_wait(bar_v, c & 1, kWait);
        mine = ks_ok && v_ok && mine;
        tc_fence_after();
        const int t = 32 * wq + lane;
        for (int g = wgm; g < 8; g += 3) {
          float v[16], vv[16];
          const int j0 = 16 * g, sl = j0 >> 6, cc0 = (j0 & 63) >> 3;
          tmem_ld16(TU + lane_base + j0, v);
          const uint32_t o0 = sl * 8192 + chunk_off(t, cc0), o1 = sl * 8192 + chunk_off(t, cc0 + 1);
          unpack_bf8(sm16(vr, o0), vv);
          unpack_bf8(sm16(vr, o1), vv + 8);
#pragma unroll
          for (int u = 0; u < 16; ++u) v[u] += vv[u];
          sm16(vr, o0) = pack_h8(v);
          sm16(vr, o1) = pack_h8(v + 8);
        }
      };
      wy_inverse(mt, sT, sA, sX, sY, s_r + 64 * (c & 1), s_s, s_is, awu, y_side);
      if (!CH && wq >= 2) ++mph;  // MMA-KS, observed by the Y warps
    }
    fence_proxy_async();
    tc_fence_before();
    bar_sync(kBarMain, kMain);

    // ---- [5] (context only) -W = A (-Kbar) into TW, then to the context
    if (CH && !SV) {
      if (lane == 0 && warp == 14) {
        bulk_s2g(pre + Pre<SV>::A, awu, 8192);
        bulk_commit();
      }
      if (mt < CM) reinterpret_cast<float *>(pre + Pre<SV>::s)[mt] = s_s[mt];
    }
    if (SV) {
      if (lane == 0 && warp >= 14) {
        if (warp == 14) bulk_s2g(ctx + kCtxA, awu, 8192);
        else if (!CH) bulk_s2g(ctx + kCtxY, vr, 16384);  // Y, before R' is written over it
        bulk_commit();
      }
      if (warp_u == 4) {
        tc_fence_after();
        const uint32_t lead = elect_one();
        const uint64_t AW = sw128_desc(smem_u32(awu), 16, 1024), KN = sw128_desc(smem_u32(as1), 16384, 1024);
#pragma unroll
        for (int kk = 0; kk < 4; ++kk)  // B = rows 0..63 of [-Kbar; Qbar], MN-major
          umma_if(lead, TW, step(AW, kk * 32), step(KN, kk * 2048), id_16, kk > 0);
        commit_if(lead, bar_w);  // its own barrier: MMA-KS may not have been observed yet
      }
    }
    // ---- [6] (context only) -W out of TMEM; A_qk and s_t
    if (SV) {  // -W of the context (rows 0..63 of TW), once MMA-W has completed
      if (wq >= 2 && wgm < 2) {  // A_qk = lower(A'_qk) diag(1/s) into the context, columns 32 wgm ..
        const int t = 32 * (wq - 2) + lane;
        float pv[16];
        tmem_ld16(TD1 + lane_base + 16 * wgm, pv);
#pragma unroll
        for (int q4 = 0; q4 < 4; ++q4) {
          const int cc = 4 * wgm + q4;
          float v8[8];
#pragma unroll
          for (int j = 0; j < 4; ++j) {
            const uint32_t bits = __float_as_uint(pv[4 * q4 + j]);
            const float2 f2 = __half22float2(*reinterpret_cast<const __half2 *>(&bits));
            v8[2 * j] = f2.x * s_is[8 * cc + 2 * j];
            v8[2 * j + 1] = f2.y * s_is[8 * cc + 2 * j + 1];
          }
          *reinterpret_cast<uint4 *>(ctx + kCtxAqk + chunk_off(t, cc)) = pack_h8(v8);
        }
      } else if (wq >= 2) {
        const int t = 32 * (wq - 2) + lane;
        reinterpret_cast<float *>(ctx + kCtxTok)[t] = s_s[t];
      }
      mine = mbar_wait(bar_w, c & 1, kWait) && mine;
      tc_fence_after();
      if (wq < 2) {  // into the fp32 L^-1 tile, dead since the solve, for one bulk copy
        const int t = 32 * wq + lane;
        for (int g = wgm; g < 8; g += 3) {
          float v[16];
          const int j0 = 16 * g, sl = j0 >> 6, cc0 = (j0 & 63) >> 3;
          tmem_ld16(TW + lane_base + j0, v);
          sm16(wst, sl * 8192 + chunk_off(t, cc0)) = pack_h8(v);
          sm16(wst, sl * 8192 + chunk_off(t, cc0 + 1)) = pack_h8(v + 8);
        }
      }
      if (lane == 0 && warp >= 14) bulk_wait_read();  // [A; .] and Y may be written over in [8]
      fence_proxy_async();
      tc_fence_before();
      bar_sync(kBarMain, kMain);  // TW is free for MMA-R
      if (tid == 32 * 10) {
        bulk_s2g(ctx + kCtxW, wst, 16384);
        bulk_commit();
      }
    }

    if (CH) {  // the rest needs the memory
      if (lane == 0) bulk_wait_all();  // (the records' bulk copies have been written)
      publish(P.flag + o.rc * P.fstride);
      continue;
    }
    // ---- [7] MMA-R: TW = [A; .] Y = [R; 0]  (fp16)
    if (warp_u == 4) {
      tc_fence_after();
      const uint32_t lead = elect_one();
      const uint64_t AW = sw128_desc(smem_u32(awu), 16, 1024), VR = sw128_desc(smem_u32(vr), 8192, 1024);
#pragma unroll
      for (int kk = 0; kk < 4; ++kk) umma_if(lead, TW, step(AW, kk * 32), step(VR, kk * 2048), id_16, kk > 0);
      commit_if(lead, bar_mma);
    }
    mine = mma_wait_main() && mine;
    tc_fence_after();

    // ---- [8] R' = diag(1/s) R -> fp16 [t][j] (MN-major B), over Y
    if (wq < 2) {
      const int t = 32 * wq + lane;
      const float ist = s_is[t];
      for (int g = wgm; g < 8; g += 3) {
        float v[16];
        const int j0 = 16 * g, sl = j0 >> 6, cc0 = (j0 & 63) >> 3;
        tmem_ld16(TW + lane_base + j0, v);
        if (SV) {  // R for the context, staged over [A; .] (MMA-R has read it) for one bulk copy
          sm16(awu, sl * 8192 + chunk_off(t, cc0)) = pack_h8(v);
          sm16(awu, sl * 8192 + chunk_off(t, cc0 + 1)) = pack_h8(v + 8);
        }
#pragma unroll
        for (int u = 0; u < 16; ++u) v[u] *= ist;
        sm16(vr, sl * 8192 + chunk_off(t, cc0)) = pack_h8(v);
        sm16(vr, sl * 8192 + chunk_off(t, cc0 + 1)) = pack_h8(v + 8);
      }
    }
    fence_proxy_async();
    tc_fence_before();
    bar_sync(kBarMain, kMain);

    // ---- [9] MMA-O (rows 64..127 of TU += A'_qk R', A'_qk in TMEM) and
    //          MMA-S2 (S += K'^T R', K' in TMEM)
    if (SV && tid == 32 * 11) {
      bulk_s2g(ctx + kCtxR, awu, 16384);
      bulk_commit();
    }
    if (warp_u == 4) {
      tc_fence_after();
      const uint32_t lead = elect_one();
      const uint64_t VR = sw128_desc(smem_u32(vr), 8192, 1024);
#pragma unroll
      for (int kk = 0; kk < 4; ++kk) {
        const uint64_t bd = step(VR, kk * 2048);
        umma_f16_tA(lead, TU, TD1 + (uint32_t)(kk * 8), bd, id_16, 1);
        umma_f16_tA(lead, TS, tkt + (uint32_t)(kk * 8), bd, id_16, 1);
      }
      commit_if(lead, bar_mma);
    }
  }

  if (!CH && !failed && NC > 0) {
    if (!gain) mine = mma_wait_main() && mine;  // MMA-O / MMA-S2 of the last chunk
    tc_fence_before();
    failed = !__syncthreads_and(mine);
    tc_fence_after();
  }
  if (!CH && !failed) {
    const Job o = job(NC - 1);
    if (!gain && wq >= 2 && NC > 0 && a.o) {  // O of the last chunk
      const int t = 32 * (wq - 2) + lane, tt = (NC - 1) * CM + t;
      for (int g = wgm; g < 8; g += 3) {
        float v[16];
        const int j0 = 16 * g;
        tmem_ld16(TU + lane_base + j0, v);
        if (tt < a.T) {
          const size_t base = tok_index(a, o.b, tt, o.h) * D + j0;
          if (a.odt == KDN_BF16) {
            uint4 *dst = reinterpret_cast<uint4 *>(static_cast<__nv_bfloat16 *>(a.o) + base);
            dst[0] = pack_bf8(v);
            dst[1] = pack_bf8(v + 8);
          } else {
            float4 *dst = reinterpret_cast<float4 *>(static_cast<float *>(a.o) + base);
#pragma unroll
            for (int u = 0; u < 4; ++u) dst[u] = make_float4(v[4 * u], v[4 * u + 1], v[4 * u + 2], v[4 * u + 3]);
          }
        }
      }
    }
    if (!gain && a.ST) {
      const int i = 32 * wq + lane;
      for (int g = wgm; g < 8; g += 3) {
        float v[16];
        const int j0 = 16 * g;
        tmem_ld16(TS + lane_base + j0, v);
        float4 *dst = reinterpret_cast<float4 *>(a.ST + ((size_t)bh * D + i) * D + j0);
#pragma unroll
        for (int u = 0; u < 4; ++u) dst[u] = make_float4(v[4 * u], v[4 * u + 1], v[4 * u + 2], v[4 * u + 3]);
      }
    }
    if (a.pT && gain) a.pT[(size_t)bh * D + tid] = p;
  } else if (failed) {
    if (tid == 0) atomicExch(a.status, (unsigned)KDN_ERR_TIMEOUT);
    // copies and MMAs in flight land before the CTA's memory goes away
    // (short bounds: a copy or MMA that was issued lands within microseconds,
    // and a phase that was never armed must not hold the call for long)
    if (issuer) {
      for (int k = 0; k < 6; ++k) {
        mbar_wait(bars + k, 0, kDrain);
        mbar_wait(bars + k, 1, kDrain);
      }
    }
  }
  if ((SV || CH) && lane == 0) bulk_wait_all();
  tc_fence_before();
  __syncthreads();
  if (warp == 0) tmem_dealloc(tbase, 512);
}

template <int SV, int LG>
__global__ void __launch_bounds__(WT, 1)
    k_wy_fwd(const __grid_constant__ CUtensorMap mk, const __grid_constant__ CUtensorMap mg,
             const __grid_constant__ CUtensorMap mw, const __grid_constant__ CUtensorMap mv,
             const __grid_constant__ CUtensorMap mq, const WyParams P) {
  wy_body<SV, LG, 0>(mk, mg, mw, mv, mq, P, (int)blockIdx.x, (int)gridDim.x);
}

// ---------------------------------------------------------------------------
// wy_gain: the uncertainty entering every chunk, one CTA per sequence: nothing but the serial
// chain of p, with the operations of gain_chunk.  Warps 4..15 form alpha, omega and mu k^2 / r
// half a chunk ahead of warps 0..3, whose loop is the chain alone (~45 cycles a token).  With
// the inputs loaded by the chain's own threads 16 tokens ahead it took 13 K cycles a chunk,
// this way 5 K (with the range test 6.5 K).
constexpr int kBarFull = 1, kBarEmpty = 3, kBarProd = 5;  // (full, empty: + half of the chunk)
constexpr int kProd = WT - 128;
constexpr int SG_RAW = 49152, SG_X = 2 * SG_RAW, SG_HALF = 3 * 32 * D * 4, SG_SS = SG_X + 2 * SG_HALF;
constexpr int SG_MR = SG_SS + 16 * D * 4, SG_BAR = SG_MR + 2 * CM * 4, SG_SMEM = SG_BAR + 64 + 1024;
static_assert(SG_SMEM <= 232448, "shared memory");

template <int SV, int LG>
__device__ __forceinline__ void wy_gain(const CUtensorMap &mk, const CUtensorMap &mg, const CUtensorMap &mw,
                                        const WyParams &P, const int bh) {
  const Args &a = P.a;
  extern __shared__ unsigned char smraw[];
  unsigned char *sm =
      reinterpret_cast<unsigned char *>((reinterpret_cast<uintptr_t>(smraw) + 1023) & ~uintptr_t(1023));
  float *s_ss = reinterpret_cast<float *>(sm + SG_SS), *s_mr = reinterpret_cast<float *>(sm + SG_MR);
  uint64_t *bars = reinterpret_cast<uint64_t *>(sm + SG_BAR);
  int *s_oor = reinterpret_cast<int *>(bars + 2);
  const int tid = threadIdx.x, b = bh / a.H, h = bh % a.H, NC = P.nc;
  auto alpha = [&](int half) { return reinterpret_cast<float *>(sm + SG_X + half * SG_HALF); };  // then omega, u
  if (tid == 0) {
    mbar_init(bars, 1);
    mbar_init(bars + 1, 1);
    fence_mbar_init();
  }
  __syncthreads();
  if (tid < D) {  // ---- the chain
    float p = P.p_in ? P.p_in[(size_t)bh * D + tid] : 1.f;
    for (int c = 0; c < NC; ++c) {
      pin_put(P.pin + ((size_t)bh * NC + c) * D + tid, p);
#pragma unroll 1
      for (int half = 0; half < 2; ++half) {
        bar_sync(kBarFull + half, WT);
        const float *xa = alpha(half) + tid, *xw = xa + 32 * D, *xu = xw + 32 * D;
        if (!SV && s_oor[c & 1]) {  // range mode (see gain_chunk)
#pragma unroll 8
          for (int t = 0; t < 32; ++t) {
            const float al = xa[t * D], ph = fmaf(al * al, p, xw[t * D]);
            p = ph * rcpf(fmaf(xu[t * D], ph, 1.f));
          }
        } else {
#pragma unroll
          for (int t = 0; t < 32; ++t) {
            const float al = xa[t * D], ph = fmaf(al * al, p, xw[t * D]);
            const float x = rcpf(al * fmaf(xu[t * D], ph, 1.f));
            p = ph * (x * al);
          }
        }
        if (c + 1 < NC) bar_arrive(kBarEmpty + half, WT);
      }
    }
    if (P.p_out) P.p_out[(size_t)bh * D + tid] = p;
  } else {  // ---- its inputs
    const int pt = tid - D;
    auto issue = [&](int c) {
      unsigned char *d = sm + (c & 1) * SG_RAW;
      mbar_expect_tx(bars + (c & 1), SG_RAW);
      const int t = (P.c0 + c) * CM;
      for (int s = 0; s < 2; ++s) {
        tma_load_4d(d + s * 8192, &mk, bars + (c & 1), 64 * s, h, t, b);
        tma_load_4d(d + 16384 + s * 8192, &mg, bars + (c & 1), 64 * s, h, t, b);
        tma_load_4d(d + 32768 + s * 8192, &mw, bars + (c & 1), 64 * s, h, t, b);
      }
    };
    __nv_bfloat16 znext = __float2bfloat16_rn(0.f);
    auto load_r = [&](int c) {
      if (pt < CM && c < NC)
        znext = static_cast<const __nv_bfloat16 *>(a.r)[tok_index(a, b, min((P.c0 + c) * CM + pt, a.T - 1), h)];
    };
    auto lga = [&](float x) { return LG ? -softplus_w(-x) : x; };
    if (pt == 0) {
      issue(0);
      if (NC > 1) issue(1);
    }
    load_r(0);
    bool ok = true;
    for (int c = 0; c < NC; ++c) {
      const int left = a.T - (P.c0 + c) * CM;  // tokens past T: alpha 1, omega 0, u 0
      float *mr = s_mr + (c & 1) * CM;
      if (pt < CM) {
        const float z = __bfloat162float(znext), r = LG ? a.rmin + softplus_w(z) : z;
        mr[pt] = pt < left ? a.mu / r : 0.f;
      }
      load_r(c + 1);
      ok = mbar_wait(bars + (c & 1), (c >> 1) & 1, kWait) && ok;
      const unsigned char *d = sm + (c & 1) * SG_RAW;
      auto raw = [&](int which, int t, int i) {  // channels i, i + 1 of token t
        return __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162 *>(d + which * 16384 + (i >> 6) * 8192 +
                                                                            sw128_off(t, i & 63)));
      };
      if (SV) {
        bar_sync(kBarProd, kProd);
      } else {  // does a channel leave the referenced range?  G_C summed in gain_chunk's order
        for (int e = pt; e < 16 * (D / 2); e += kProd) {  // four tokens of two channels
          const int i = 2 * (e & 63), t = 4 * (e >> 6);
          float2 x[4];
#pragma unroll
          for (int j = 0; j < 4; ++j) {
            const float2 y = raw(1, t + j, i);
            x[j] = t + j < left ? make_float2(lga(y.x), lga(y.y)) : make_float2(0.f, 0.f);
          }
          *reinterpret_cast<float2 *>(s_ss + (e >> 6) * D + i) =
              make_float2((x[0].x + x[1].x) + (x[2].x + x[3].x), (x[0].y + x[1].y) + (x[2].y + x[3].y));
        }
        bar_sync(kBarProd, kProd);
        float GC = 0.f;
        if (pt < D)
          for (int sg = 0; sg < 8; ++sg) GC += s_ss[2 * sg * D + pt] + s_ss[(2 * sg + 1) * D + pt];
        const bool oor = bar_or(kBarProd, kProd, pt < D && 0.5f * GC < kMinHalfG);
        if (pt == 0) s_oor[c & 1] = oor ? 1 : 0;
      }
#pragma unroll 1
      for (int half = 0; half < 2; ++half) {
        if (c > 0) bar_sync(kBarEmpty + half, WT);
        float *xa = alpha(half), *xw = xa + 32 * D, *xu = xw + 32 * D;
        for (int e = pt; e < 16 * (D / 2); e += kProd) {  // two tokens of two channels
          const int i = 2 * (e & 63), t0 = 2 * (e >> 6);
#pragma unroll
          for (int j = 0; j < 2; ++j) {
            const int t = 32 * half + t0 + j, o = (t0 + j) * D + i;
            const bool live = t < left;
            const float2 k = raw(0, t, i), x = raw(1, t, i), y = raw(2, t, i);
            const float m = mr[t];
            float2 al = make_float2(ex2f(lga(x.x) * kLog2e), ex2f(lga(x.y) * kLog2e));
            float2 w = LG ? make_float2(softplus_w(y.x), softplus_w(y.y)) : y;
            if (!live) {
              al = make_float2(1.f, 1.f);
              w = make_float2(0.f, 0.f);
            }
            *reinterpret_cast<float2 *>(xa + o) = al;
            *reinterpret_cast<float2 *>(xw + o) = w;
            *reinterpret_cast<float2 *>(xu + o) = make_float2(k.x * k.x * m, k.y * k.y * m);
          }
        }
        bar_arrive(kBarFull + half, WT);
      }
      bar_sync(kBarProd, kProd);  // the raw tiles have been read
      if (pt == 0 && c + 2 < NC) issue(c + 2);
    }
    if (!ok) atomicExch(a.status, (unsigned)KDN_ERR_TIMEOUT);
  }
}

// ---------------------------------------------------------------------------
// wy_state: the memory over the chunks of one sequence, from the records of the chunk part:
//   TU = [-Kbar; Qbar] S;  Y = V + TU;  R = A Y;  R' = R / s;  O = TU + A'_qk R';
//   S = gamma_C S + K'^T R'.
// One CTA per sequence; warp w: TMEM lanes 32 (w % 4) .., columns by w / 4.  A chunk's
// operands (80 KB) are double-buffered bulk copies; O is stored beside the next chunk's first
// product (TU has two buffers).  Bound by the chain of its three products and their
// conversions, ~6 K cycles a chunk.
constexpr int SB_KQ = 0, SB_KT = 32768, SB_AA = 49152, SB_V = 65536, SB_SC = 81920, SB_BUF = 82944;
constexpr int SO_S16 = 2 * SB_BUF, SO_R = SO_S16 + 32768, SO_BARS = SO_R + 16384, ST_SMEM = SO_BARS + 64 + 1024;
static_assert(SB_BUF % 1024 == 0 && ST_SMEM <= 232448, "shared memory");

template <int SV>
__device__ __forceinline__ void wy_state(const CUtensorMap &mv, const WyParams &P, const int bh) {
  using R = Pre<SV>;
  const Args &a = P.a;
  extern __shared__ unsigned char smraw[];
  unsigned char *sm =
      reinterpret_cast<unsigned char *>((reinterpret_cast<uintptr_t>(smraw) + 1023) & ~uintptr_t(1023));
  unsigned char *s16 = sm + SO_S16, *rst = sm + SO_R;
  uint64_t *bars = reinterpret_cast<uint64_t *>(sm + SO_BARS);
  uint64_t *bar_ld = bars, *bar_mma = bars + 2, *bar_o = bars + 3;
  uint32_t *s_tbase = reinterpret_cast<uint32_t *>(bars + 4);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, wq = warp & 3, wg = warp >> 2;
  const int b = bh / a.H, h = bh % a.H, NC = P.nc;
  const int warp_u = __shfl_sync(0xffffffffu, warp, 0);
  const uint32_t lane_base = (uint32_t)(32 * wq) << 16;
  bool ok = true;
  if (tid == 0) {
    mbar_init(bar_ld, 8);
    mbar_init(bar_ld + 1, 8);
    mbar_init(bar_mma, 1);
    mbar_init(bar_o, 1);
    fence_mbar_init();
    prefetch_tmap(&mv);
  }
  if (warp == 0) {
    tmem_alloc(s_tbase, 512);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t TS = *s_tbase, TW = TS + 128, TUb = TS + 256;
  auto record = [&](int c) { return P.pre + ((size_t)bh * NC + c) * P.prec; };
  auto issue = [&](int c) {  // lane 0 of warps 8..15
    const unsigned char *rec = record(c);
    unsigned char *d = sm + (c & 1) * SB_BUF;
    uint64_t *bar = bar_ld + (c & 1);
    if (lane == 0 && warp >= 8) {  // (a record that never comes is read as it is: the call fails)
      ok = flow_wait(P.flag + ((size_t)bh * NC + c) * P.fstride) && ok;
      fence_proxy_async_all();
    }
    switch (lane == 0 ? warp : -1) {
      case 8: mbar_expect_tx(bar, 16384); bulk_g2s(d + SB_KQ, rec + R::KQ, 16384, bar); break;
      case 9: mbar_expect_tx(bar, 16384); bulk_g2s(d + SB_KQ + 16384, rec + R::KQ + 16384, 16384, bar); break;
      case 10: mbar_expect_tx(bar, 16384); bulk_g2s(d + SB_KT, rec + R::Kt, 16384, bar); break;
      case 11: mbar_expect_tx(bar, 8192); bulk_g2s(d + SB_AA, rec + R::A, 8192, bar); break;
      case 12: mbar_expect_tx(bar, 8192); bulk_g2s(d + SB_AA + 8192, rec + R::Aq, 8192, bar); break;
      case 13: mbar_expect_tx(bar, 8192); tma_load_4d(d + SB_V, &mv, bar, 0, h, (P.c0 + c) * CM, b); break;
      case 14: mbar_expect_tx(bar, 8192); tma_load_4d(d + SB_V + 8192, &mv, bar, 64, h, (P.c0 + c) * CM, b); break;
      case 15:
        mbar_expect_tx(bar, 768);
        bulk_g2s(d + SB_SC, rec + R::gC, 512, bar);
        bulk_g2s(d + SB_SC + 512, rec + R::s, 256, bar);
        break;
    }
  };
  issue(0);
  const int i = 32 * wq + lane, j0 = 32 * wg;  // this thread's row and first column of S
  for (int c0 = 0; c0 < 32; c0 += 16) {
    float v[16];
    if (P.S_in) {
      const float4 *src = reinterpret_cast<const float4 *>(P.S_in + ((size_t)bh * D + i) * D + j0 + c0);
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const float4 x = src[u];
        v[4 * u] = x.x; v[4 * u + 1] = x.y; v[4 * u + 2] = x.z; v[4 * u + 3] = x.w;
      }
    } else {
#pragma unroll
      for (int u = 0; u < 16; ++u) v[u] = 0.f;
    }
    tmem_st16(TS + lane_base + j0 + c0, v);
  }
  tmem_st_wait();
  auto store_o = [&](int c) {  // O of chunk c: rows 64..127 of its TU, 32 columns a thread
    const int t = 32 * (wq - 2) + lane, tt = (P.c0 + c) * CM + t;
    for (int c0 = 0; c0 < 32; c0 += 16) {
      float v[16];
      tmem_ld16(TUb + (c & 1) * 128 + lane_base + j0 + c0, v);
      if (tt < a.T) {
        const size_t base = tok_index(a, b, tt, h) * D + j0 + c0;
        if (a.odt == KDN_BF16) {
          uint4 *dst = reinterpret_cast<uint4 *>(static_cast<__nv_bfloat16 *>(a.o) + base);
          dst[0] = pack_bf8(v);
          dst[1] = pack_bf8(v + 8);
        } else {
          float4 *dst = reinterpret_cast<float4 *>(static_cast<float *>(a.o) + base);
#pragma unroll
          for (int u = 0; u < 4; ++u) dst[u] = make_float4(v[4 * u], v[4 * u + 1], v[4 * u + 2], v[4 * u + 3]);
        }
      }
    }
  };
  uint32_t mph = 0;
  auto mma_wait = [&]() -> bool {
    const bool r = mbar_wait(bar_mma, mph & 1, kWait);
    ++mph;
    tc_fence_after();
    return r;
  };
  const uint32_t id_16 = idesc_f16(128, 128, 0, 1);  // A K-major, B MN-major
  for (int c = 0; c < NC; ++c) {
    unsigned char *d = sm + (c & 1) * SB_BUF, *vr = d + SB_V;
    unsigned char *ctx = SV ? P.save_S + ((size_t)bh * NC + c) * kCtxBytes : nullptr;
    const float *sc = reinterpret_cast<const float *>(d + SB_SC);
    const uint32_t TU = TUb + (c & 1) * 128;
    // ---- [1] S -> fp16; diag(gamma_C) S back
    ok = mbar_wait(bar_ld + (c & 1), (c >> 1) & 1, kWait) && ok;
    if (c > 0) ok = mma_wait() && ok;  // MMA-S2 of chunk c - 1
    if (SV && lane == 0) bulk_wait_read();  // its S, Y and R tiles have left shared memory
    if (SV) __syncthreads();
    {
      const float gC = sc[i];
#pragma unroll
      for (int c0 = 0; c0 < 32; c0 += 16) {
        float v[16];
        tmem_ld16(TS + lane_base + j0 + c0, v);
        const int sl = j0 >> 6, cc0 = ((j0 & 63) + c0) >> 3;
        sm16(s16, sl * 16384 + chunk_off(i, cc0)) = pack_h8(v);
        sm16(s16, sl * 16384 + chunk_off(i, cc0 + 1)) = pack_h8(v + 8);
#pragma unroll
        for (int u = 0; u < 16; ++u) v[u] *= gC;
        tmem_st16(TS + lane_base + j0 + c0, v);
      }
    }
    tmem_st_wait();
    fence_proxy_async();
    tc_fence_before();
    if (!__syncthreads_and(ok)) {
      ok = false;
      break;
    }
    // ---- [2] MMA-KS; the next chunk's operands; O of chunk c - 1
    if (warp_u == 0) {
      tc_fence_after();
      const uint32_t lead = elect_one();
      const uint64_t A1 = sw128_desc(smem_u32(d + SB_KQ), 16, 1024), B1 = sw128_desc(smem_u32(s16), 16384, 1024);
#pragma unroll
      for (int kk = 0; kk < 8; ++kk)
        umma_if(lead, TU, step(A1, (kk >> 2) * 16384 + (kk & 3) * 32), step(B1, kk * 2048), id_16, kk > 0);
      commit_if(lead, bar_mma);
    }
    if (c > 0) ok = mbar_wait(bar_o, (c - 1) & 1, kWait) && ok;  // MMA-O of chunk c - 1: its buffer is free
    if (c + 1 < NC) issue(c + 1);
    if (SV && tid == 32) {
      bulk_s2g(ctx + kCtxS, s16, 32768);
      bulk_commit();
    }
    if (wq >= 2 && c > 0 && a.o) {
      tc_fence_after();
      store_o(c - 1);
      tc_fence_before();
    }
    ok = mma_wait() && ok;
    // ---- [3] Y = V - Kbar S_in -> fp16 over V
    if (wq < 2) {
      for (int c0 = 0; c0 < 32; c0 += 16) {
        float v[16], vv[16];
        const int jj = j0 + c0, sl = jj >> 6, cc0 = (jj & 63) >> 3;
        tmem_ld16(TU + lane_base + jj, v);
        const uint32_t o0 = sl * 8192 + chunk_off(i, cc0), o1 = sl * 8192 + chunk_off(i, cc0 + 1);
        unpack_bf8(sm16(vr, o0), vv);
        unpack_bf8(sm16(vr, o1), vv + 8);
#pragma unroll
        for (int u = 0; u < 16; ++u) v[u] += vv[u];
        sm16(vr, o0) = pack_h8(v);
        sm16(vr, o1) = pack_h8(v + 8);
      }
    }
    fence_proxy_async();
    tc_fence_before();
    __syncthreads();
    // ---- [4] MMA-R: TW = [A; A'_qk] Y (rows 0..63: R)
    const uint64_t AA = sw128_desc(smem_u32(d + SB_AA), 16, 1024), VR = sw128_desc(smem_u32(vr), 8192, 1024);
    if (warp_u == 0) {
      tc_fence_after();
      const uint32_t lead = elect_one();
#pragma unroll
      for (int kk = 0; kk < 4; ++kk) umma_if(lead, TW, step(AA, kk * 32), step(VR, kk * 2048), id_16, kk > 0);
      commit_if(lead, bar_mma);
    }
    if (SV && tid == 64) {
      bulk_s2g(ctx + kCtxY, vr, 16384);
      bulk_commit();
      bulk_wait_read();  // R' is written over it
    }
    ok = mma_wait() && ok;
    if (SV) __syncthreads();
    // ---- [5] R' = diag(1/s) R -> fp16 over Y
    if (wq < 2) {
      const float ist = rcpf(sc[D + i]);
      for (int c0 = 0; c0 < 32; c0 += 16) {
        float v[16];
        const int jj = j0 + c0, sl = jj >> 6, cc0 = (jj & 63) >> 3;
        const uint32_t o0 = sl * 8192 + chunk_off(i, cc0), o1 = sl * 8192 + chunk_off(i, cc0 + 1);
        tmem_ld16(TW + lane_base + jj, v);
        if (SV) {
          sm16(rst, o0) = pack_h8(v);
          sm16(rst, o1) = pack_h8(v + 8);
        }
#pragma unroll
        for (int u = 0; u < 16; ++u) v[u] *= ist;
        sm16(vr, o0) = pack_h8(v);
        sm16(vr, o1) = pack_h8(v + 8);
      }
    }
    fence_proxy_async();
    tc_fence_before();
    __syncthreads();
    // ---- [6] MMA-S2 (S += K'^T R'), which the next chunk waits for, then MMA-O (rows 64..127
    //          of TU += A'_qk R')
    if (warp_u == 0) {
      tc_fence_after();
      const uint32_t lead = elect_one();
      const uint64_t KT = sw128_desc(smem_u32(d + SB_KT), 16, 1024);
#pragma unroll
      for (int kk = 0; kk < 4; ++kk) umma_if(lead, TS, step(KT, kk * 32), step(VR, kk * 2048), id_16, 1);
      commit_if(lead, bar_mma);
#pragma unroll
      for (int kk = 0; kk < 4; ++kk) umma_if(lead, TU, step(AA, kk * 32), step(VR, kk * 2048), id_16, 1);
      commit_if(lead, bar_o);
    }
    if (SV && tid == 96) {
      bulk_s2g(ctx + kCtxR, rst, 16384);
      bulk_commit();
    }
  }
  if (ok && NC > 0) ok = mma_wait() && mbar_wait(bar_o, (NC - 1) & 1, kWait);
  if (__syncthreads_and(ok)) {
    tc_fence_after();
    if (wq >= 2 && a.o) store_o(NC - 1);
    if (P.S_out) {
      for (int c0 = 0; c0 < 32; c0 += 16) {
        float v[16];
        tmem_ld16(TS + lane_base + j0 + c0, v);
        float4 *dst = reinterpret_cast<float4 *>(P.S_out + ((size_t)bh * D + i) * D + j0 + c0);
#pragma unroll
        for (int u = 0; u < 4; ++u) dst[u] = make_float4(v[4 * u], v[4 * u + 1], v[4 * u + 2], v[4 * u + 3]);
      }
    }
  } else if (tid == 0) {
    atomicExch(a.status, (unsigned)KDN_ERR_TIMEOUT);
    // copies and MMAs in flight land before the CTA's memory goes away
    for (int k = 0; k < 4; ++k) {
      mbar_wait(bars + k, 0, kDrain);
      mbar_wait(bars + k, 1, kDrain);
    }
  }
  if (SV && lane == 0) bulk_wait_all();
  tc_fence_before();
  __syncthreads();
  if (warp == 0) tmem_dealloc(TS, 512);
}

// ---------------------------------------------------------------------------
// k_wy_flow: the three parts at once, one CTA per SM: first the gain's CTAs (one per sequence),
// then the chunk part's, then the memory's (one per sequence).  The parts wait for one another
// (bounded), so the launch is cooperative: it starts once all its CTAs can be resident.  (Places by
// the order of start would do as well, but mix the parts on the two SMs of a TPC, which fetch
// instructions together: B2 H16 T1999 with logit gates 230 us, not 207.)  B1 H16 T777 with
// logit gates 119 us as three launches, 78 us as one (one CTA per sequence: 143 us); training
// forward B2 H16 T1999 302 and 207 us (430).
constexpr int FLOW_SMEM = SMEM_BYTES > SG_SMEM ? (SMEM_BYTES > ST_SMEM ? SMEM_BYTES : ST_SMEM)
                                               : (SG_SMEM > ST_SMEM ? SG_SMEM : ST_SMEM);
template <int SV, int LG>
__global__ void __launch_bounds__(WT, 1)
    k_wy_flow(const __grid_constant__ CUtensorMap mk, const __grid_constant__ CUtensorMap mg,
              const __grid_constant__ CUtensorMap mw, const __grid_constant__ CUtensorMap mv,
              const __grid_constant__ CUtensorMap mq, const WyParams P) {
  const int BH = P.a.B * P.a.H, block = (int)blockIdx.x, workers = (int)gridDim.x - 2 * BH;
  if (block < BH) wy_gain<SV, LG>(mk, mg, mw, P, block);
  else if (block < BH + workers) wy_body<SV, LG, 1>(mk, mg, mw, mv, mq, P, block - BH, workers);
  else wy_state<SV>(mv, P, block - BH - workers);
}

}  // namespace

bool wy_fwd_supported(const Args &a) {
  return a.variant == 0 && (a.gates == KDN_GATES_POST || a.gates == KDN_GATES_LOGITS) &&
         a.dtype == KDN_BF16 && a.dk == D && a.dv == D && a.T > 0 && a.chunk != 32;
}

// Where k_wy_flow finishes sooner than k_wy_fwd, in thousands of cycles as measured: the one
// takes 17 a chunk with one CTA per sequence; k_wy_flow 7 a chunk of a sequence (its memory part)
// or 19 a chunk of all sequences over its workers, whichever is longer, and 45 until the first
// records are there.  Post-activation gates, k_wy_flow and k_wy_fwd in us: B1 H16 T823 75 and
// 118, T2047 141 and 269, T8191 483 and 1046, T65471 3869 and 8172, B2 H16 T2047 168 and 278, B1 H40 T4001 424
// and 540, B24 H1 T257 48 and 55; logit gates: 82 and 146, 151 and 333, 497 and 1315, 3999 and 10284,
// 224 and 353, 580 and 670, 55 and 68.  With 48 sequences
// the one is ahead (B3 H16 T1300 216 and 198, T2047 301 and 298); more sequences than 56 leave too few workers.
// Fewer than 96 chunks in all are left to the one kernel (tens of us either way).
// A workspace holds the records of kSlice chunks of all sequences (136 MB); longer sequences take
// several launches, which hand the state on in float32 (the same results), each with its 45.
constexpr long long kSlice = 2048;
int wy_slices(const Args &a) {
  const long long bh = (long long)a.B * a.H, nc = (a.T + CM - 1) / CM, per = kSlice / bh;
  return (int)((nc + per - 1) / per);
}
static long long wy_slice_chunks(const Args &a) {
  const long long nc = (a.T + CM - 1) / CM, ns = wy_slices(a);
  return (nc + ns - 1) / ns;
}
bool wy_split_sizes(const Args &a) {
  if (!wy_fwd_supported(a)) return false;
  const long long bh = (long long)a.B * a.H, nc = (a.T + CM - 1) / CM;
  if (bh * nc < 96 || bh > 56) return false;
  const long long workers = kSms - 2 * bh, sc = wy_slice_chunks(a);
  return wy_slices(a) * (std::max(sc * 7, (bh * sc + workers - 1) / workers * 19) + 45) < nc * 17;
}

size_t wy_split_workspace_bytes(const Args &a) {
  if (!wy_split_sizes(a)) return 0;
  const size_t bh = (size_t)a.B * a.H;
  return bh * wy_slice_chunks(a) * (kPreBytes + D * sizeof(float) + sizeof(unsigned)) +
         (wy_slices(a) > 1 ? bh * (D * D + D) * sizeof(float) + 256 : 0);
}

namespace {
template <int SV, int LG>
kdn_status_t launch_wy(WyParams &W, bool split, char *ws, cudaStream_t s) {
  const Args &a = W.a;
  CUtensorMap mk, mg, mw, mv, mq;
  if (!make_map(&mk, a.k, a) || !make_map(&mg, a.g, a) || !make_map(&mw, a.omega, a) ||
      !make_map(&mv, a.v, a) || !make_map(&mq, a.q, a))
    return KDN_ERR_CUDA;
  const int bh = a.B * a.H, NC = (a.T + CM - 1) / CM;
  const auto attr = cudaFuncAttributeMaxDynamicSharedMemorySize;
  auto one = [&]() {
    if (cudaFuncSetAttribute(k_wy_fwd<SV, LG>, attr, SMEM_BYTES) != cudaSuccess) return KDN_ERR_CUDA;
    k_wy_fwd<SV, LG><<<bh, WT, SMEM_BYTES, s>>>(mk, mg, mw, mv, mq, W);
    return cudaGetLastError() == cudaSuccess ? KDN_OK : KDN_ERR_CUDA;
  };
  if (!split) return one();
  if (cudaFuncSetAttribute(k_wy_flow<SV, LG>, attr, FLOW_SMEM) != cudaSuccess) return KDN_ERR_CUDA;
  const int per = SV ? NC : (int)wy_slice_chunks(a);  // (the context has room for every chunk)
  float *Sc = nullptr, *pc = nullptr;                 // the state between two slices
  if (!SV) {
    const size_t n = (size_t)bh * per;
    W.pre = reinterpret_cast<unsigned char *>(ws);
    W.prec = kPreBytes;
    W.pin = reinterpret_cast<float *>(ws + n * kPreBytes);
    W.flag = reinterpret_cast<unsigned *>(W.pin + n * D);
    W.fstride = 1;
    const uintptr_t end = reinterpret_cast<uintptr_t>(W.flag + n);
    Sc = reinterpret_cast<float *>((end + 255) & ~uintptr_t(255));
    pc = Sc + (size_t)bh * D * D;
  }
  for (W.c0 = 0; W.c0 < NC; W.c0 += per) {
    const bool first = W.c0 == 0, last = W.c0 + per >= NC;
    W.nc = last ? NC - W.c0 : per;
    W.S_in = first ? a.S0 : Sc;
    W.p_in = first ? a.p0 : pc;
    W.S_out = last ? a.ST : Sc;
    W.p_out = last ? a.pT : pc;
    const size_t n = (size_t)bh * W.nc;
    if (cudaMemsetAsync(W.pin, 0xff, n * D * sizeof(float), s) != cudaSuccess ||
        (SV ? cudaMemset2DAsync(W.flag, kCtxBytes, 0, sizeof(unsigned), n, s)
            : cudaMemsetAsync(W.flag, 0, n * sizeof(unsigned), s)) != cudaSuccess)
      return KDN_ERR_CUDA;
    cudaLaunchAttribute coop;
    coop.id = cudaLaunchAttributeCooperative;
    coop.val.cooperative = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = kSms;
    cfg.blockDim = WT;
    cfg.dynamicSmemBytes = FLOW_SMEM;
    cfg.stream = s;
    cfg.attrs = &coop;
    cfg.numAttrs = 1;
    const cudaError_t e =
        cudaLaunchKernelEx(&cfg, k_wy_flow<SV, LG>, mk, mg, mw, mv, mq, static_cast<const WyParams>(W));
    if (e == cudaErrorCooperativeLaunchTooLarge && first) {  // (fewer SMs than a whole GPU's are ours)
      cudaGetLastError();
      return one();
    }
    if (e != cudaSuccess) return KDN_ERR_CUDA;
  }
  return KDN_OK;
}
}  // namespace

// ws: room for wy_split_workspace_bytes() (null: the one kernel, unless the context has the room)
kdn_status_t launch_wy_fwd(const Args &a, cudaStream_t s, unsigned char *save_S, float *save_p, char *ws) {
  if (!wy_fwd_supported(a) || (!save_S) != (!save_p)) return KDN_ERR_UNSUPPORTED;
  WyParams P{};
  P.a = a;
  P.save_S = save_S;
  P.save_p = save_p;
  const bool split = wy_split_sizes(a) && (save_S || ws);
  if (split && save_S) {
    P.pre = save_S;
    P.prec = kCtxBytes;
    P.pin = save_p;
    P.flag = reinterpret_cast<unsigned *>(save_S + kCtxTok + 3 * CM * sizeof(float));  // (no value there)
    P.fstride = kCtxBytes / sizeof(unsigned);
  }
  if (a.gates == KDN_GATES_LOGITS)
    return save_S ? launch_wy<1, 1>(P, split, ws, s) : launch_wy<0, 1>(P, split, ws, s);
  return save_S ? launch_wy<1, 0>(P, split, ws, s) : launch_wy<0, 0>(P, split, ws, s);
}

}  // namespace kdn
