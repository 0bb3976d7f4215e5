// kdn_split_bwd.cu -- backward of the Diagonal KDN (bfloat16 activations, d_k = d_v =
// 128, 64-token chunks) in two steps, so that only what is sequential over chunks
// runs sequentially:
//   k_bwd_state   one CTA per (batch, head) carries the memory cotangent dS (128 x 128
//                 fp32 in tensor memory) backwards over the chunks:
//                   dR   = A_qk^T dO + K_tail dS
//                   dS_in = diag(gamma_C) dS + Qbar^T dO - W^T dR
//                 and leaves dS and dR of every chunk in 16 bits (its operands K_tail and
//                 Qbar are formed before, in parallel over chunks, by k_bwd_tiles);
//   k_bwd_chunk   every other adjoint of a chunk, in parallel over (chunk, batch, head):
//                 persistent CTAs take chunks in reverse time order.  The uncertainty
//                 cotangent dp is the one value that still runs backwards: a chunk awaits dp_out
//                 ahead of its last pass and hands on at once the dp_in that the pass will end with.
// The one-kernel sweep (kdn_fused_bwd.cu) spends ~40 K cycles on a chunk, nearly all of it
// on work that needs no other chunk, with one CTA per (batch, head): 128 CTAs at most
// busy on 152 SMs, 32 at B2 H16.  Here the serial part is ~6 K cycles a chunk.
//
// Scratch per chunk and head: dS fp16 (32 KB), dR as an fp16 pair (32 KB; K_tail and Qbar
// before), and ~4 KB of small values.  It lies in the gradient buffers
// themselves: a chunk's rows of dq, dk, dv, dg hold its tiles and its rows of
// domega the small values until k_bwd_chunk, which is the only one to read them, writes the
// chunk's gradients there.  The partial last chunk of a ragged length has too few rows there: its
// 80 KB lie in the workspace.
//
// It serves bf16 gradients without state gradients (see split_bwd_supported).  The gradients are
// those of the one-kernel sweep bit for bit: the same operand tiles (fp16 tiles, hi/lo
// bf16 pairs where Gamma-scaled operands meet, fp16 pairs for dR in A^T dR), products and sums
// in the same order, fp32 accumulators, dS fp32 across chunks, cotangents scaled by the same
// power of two.
//
// Every wait is bounded; on timeout KDN_ERR_TIMEOUT goes to the status word.
#include <algorithm>

#include "kdn_internal.cuh"
#include "kdn_sm103.cuh"
#include "kdn_bwd_common.cuh"

namespace kdn {
namespace {

using namespace sm103;
using namespace fused;

constexpr int BT = 512, CM = 64, D = 128, KB = 1024;
constexpr uint32_t kWaitIters = 1u << 25;
constexpr uint32_t kDpWait = 1u << 22;  // polls for the uncertainty cotangent of the next chunk

// Where a chunk's small values lie: rows of 256 bytes, one per token of the chunk.
// Rows 0..7: dgamma_C's dS part [4][128]; 8..11: dp [128] as (value, tag) pairs; 12: lambda;
// 13: the r inputs z_t [64].
// The partial last chunk of a ragged length (its tiles' rows are not tokens) has rows of its own.
struct Scratch {
  unsigned char *small;  // domega
  unsigned char *tail;   // [5][B][64][H][128] 16-bit: the last chunk's tiles and small values (null: none)
  int last;              // chunk that lies there
};
__device__ __forceinline__ unsigned char *small_row(const Scratch &s, const Args &a, int b, int h, int c, int n) {
  const bool tl = s.tail && c == s.last;
  return (tl ? s.tail : s.small) +
         ((tl ? ((size_t)4 * a.B + b) * CM + n : (size_t)b * a.T + c * CM + n) * a.H + h) * (2 * D);
}
// Box of scratch tile k (0, 1: dS, 2, 3: dR; m: the gradient buffer of whole chunks) of a chunk.
struct Box { const CUtensorMap *m; int t, b; };
__device__ __forceinline__ Box box_at(const Scratch &s, const Args &a, const CUtensorMap &m, const CUtensorMap &mt,
                                      int k, int b, int c) {
  return s.tail && c == s.last ? Box{&mt, 0, k * a.B + b} : Box{&m, c * CM, b};
}
__device__ __forceinline__ void box_load(void *dst, const Box &x, uint64_t *bar, int col, int h) {
  tma_load_4d(dst, x.m, bar, col, h, x.t, x.b);
}
__device__ __forceinline__ void box_store(const Box &x, const void *src, int col, int h) {
  tma_store_4d(x.m, src, col, h, x.t, x.b);
}
__device__ __forceinline__ float *small_dgc(const Scratch &s, const Args &a, int b, int h, int c, int i) {
  return reinterpret_cast<float *>(small_row(s, a, b, h, c, i >> 6)) + (i & 63);
}
// (value, tag) slot of channel i's dp
__device__ __forceinline__ uint64_t *small_slot(const Scratch &s, const Args &a, int b, int h, int c, int i) {
  return reinterpret_cast<uint64_t *>(small_row(s, a, b, h, c, 8 + (i >> 5))) + (i & 31);
}
__device__ __forceinline__ float *small_lam(const Scratch &s, const Args &a, int b, int h, int c) {
  return reinterpret_cast<float *>(small_row(s, a, b, h, c, 12));
}
__device__ __forceinline__ float *small_z(const Scratch &s, const Args &a, int b, int h, int c) {
  return reinterpret_cast<float *>(small_row(s, a, b, h, c, 13));
}
// A slot is one 64-bit number, tag above value, stored and loaded by one scalar relaxed access
// (a vector access is two in no set order): value and tag come together and need no other ordering.
__device__ __forceinline__ void slot_put(uint64_t *p, float v) {
  asm volatile("st.relaxed.gpu.global.u64 [%0], %1;" ::"l"(p), "l"(((uint64_t)1 << 32) | __float_as_uint(v)) : "memory");
}
__device__ __forceinline__ uint64_t slot_peek(const uint64_t *p) {
  uint64_t v;
  asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
  return v;
}
// x: what an earlier look at the slot found
__device__ __forceinline__ bool slot_get(const uint64_t *p, uint64_t x, float *v) {
  for (uint32_t i = 0; i < kDpWait; ++i) {
    if (x >> 32) {
      *v = __uint_as_float((uint32_t)x);
      return true;
    }
    if (i > 64) __nanosleep(32);
    x = slot_peek(p);
  }
  return false;
}
// one TMEM column: lane l of the warp gets or sets column taddr.col of lane taddr.lane + l
__device__ __forceinline__ float tmem_ld1(uint32_t taddr) {
  uint32_t r;
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x1.b32 {%0}, [%1];" : "=r"(r) : "r"(taddr) : "memory");
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
  return __uint_as_float(r);
}
__device__ __forceinline__ void tmem_st1(uint32_t taddr, float v) {
  asm volatile("tcgen05.st.sync.aligned.32x32b.x1.b32 [%0], {%1};" ::"r"(taddr), "r"(__float_as_uint(v)) : "memory");
}
// 16-byte asynchronous global -> shared copy past L1, and its completion
__device__ __forceinline__ void cp16(void *dst, const void *src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(smem_u32(dst)), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_wait() {
  asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}

struct SplitParams {
  Args a;
  Scratch s;
  unsigned *ticket;  // zeroed before k_bwd_chunk
};

// ---------------------------------------------------------------------------
// k_bwd_tiles.  One CTA per 64 channels of a chunk: K_tail^T [i][s] and Qbar^T [i][t] in fp16 from
// the context's phat, gamma and s_t, in the operations of the one-kernel sweep (the context does not
// hold them: K_tail needs s_t, which the forward knows only after the gain has moved on).  Left where
// the chunk's dR goes, which k_bwd_state writes once it has read them.  Bound by HBM: 96 KB read and
// 32 KB written per chunk, 154 us at B8 H16 T4096 (6.9 TB/s).  A thread takes two channels of eight
// tokens, all loads ahead; with one CTA of 512 threads a chunk, 16 tokens a thread, it took 218.
constexpr int TT = 256, TILE_SMEM = 16 * KB + 1024;

__global__ void __launch_bounds__(TT, 4)
    k_bwd_tiles(const __grid_constant__ CUtensorMap m2, const __grid_constant__ CUtensorMap m3,
                const __grid_constant__ CUtensorMap mt, const SplitParams P) {
  const Args &a = P.a;
  extern __shared__ unsigned char smraw[];
  __shared__ float s_si[CM];
  unsigned char *sm =
      reinterpret_cast<unsigned char *>((reinterpret_cast<uintptr_t>(smraw) + 1023) & ~uintptr_t(1023));
  const int tid = threadIdx.x, half = (int)(blockIdx.x & 1u), r0 = 2 * (tid & 31), ci = 64 * half + r0;
  const int t0 = 8 * (tid >> 5), job = (int)(blockIdx.x >> 1);
  const int NC = (a.T + CM - 1) / CM, c = job % NC, bh = job / NC, b = bh / a.H, h = bh % a.H;
  const unsigned char *rec = a.fSin + (size_t)job * kCtxBytes;
  const float *cph = reinterpret_cast<const float *>(rec + kCtxPh) + t0 * D + ci;
  const float *cga = reinterpret_cast<const float *>(rec + kCtxGa) + ci;
  float2 ph[8], ga[8];
  __nv_bfloat162 kk[8], qv[8];
#pragma unroll
  for (int j = 0; j < 8; ++j) {
    ph[j] = *reinterpret_cast<const float2 *>(cph + j * D);
    ga[j] = *reinterpret_cast<const float2 *>(cga + (t0 + j) * D);
    const size_t e = tok_index(a, b, min(c * CM + t0 + j, a.T - 1), h) * D + ci;
    kk[j] = *reinterpret_cast<const __nv_bfloat162 *>(static_cast<const __nv_bfloat16 *>(a.k) + e);
    qv[j] = *reinterpret_cast<const __nv_bfloat162 *>(static_cast<const __nv_bfloat16 *>(a.q) + e);
  }
  const float2 gC = *reinterpret_cast<const float2 *>(cga + (CM - 1) * D);
  if (tid < CM) {
    s_si[tid] = 1.f / reinterpret_cast<const float *>(rec + kCtxTok)[tid];
    const int t = c * CM + tid;
    if (half == 0)
      small_z(P.s, a, b, h, c)[tid] =
          t < a.T ? __bfloat162float(static_cast<const __nv_bfloat16 *>(a.r)[tok_index(a, b, t, h)]) : 0.f;
  }
  __syncthreads();
  float kt[2][8], qb[2][8];
#pragma unroll
  for (int j = 0; j < 8; ++j) {
    const bool live = c * CM + t0 + j < a.T;
    const float si = s_si[t0 + j];
    const float2 k = live ? __bfloat1622float2(kk[j]) : make_float2(0.f, 0.f);
    const float2 q = live ? __bfloat1622float2(qv[j]) : make_float2(0.f, 0.f);
    kt[0][j] = gC.x * __fdividef(ph[j].x * si * k.x, ga[j].x);
    kt[1][j] = gC.y * __fdividef(ph[j].y * si * k.y, ga[j].y);
    qb[0][j] = a.tau * ga[j].x * q.x;
    qb[1][j] = a.tau * ga[j].y * q.y;
  }
#pragma unroll
  for (int r = 0; r < 2; ++r) {
    const uint32_t off = chunk_off(r0 + r, t0 >> 3);
    sm16(sm, off) = pack_h8(kt[r]);
    sm16(sm + 8 * KB, off) = pack_h8(qb[r]);
  }
  fence_proxy_async();
  __syncthreads();
  if (tid == 0 || tid == 32) {  // 64 rows of each: one box, at channel 64 half of the scratch tile
    box_store(tid == 0 ? box_at(P.s, a, m2, mt, 2, b, c) : box_at(P.s, a, m3, mt, 3, b, c), sm + (tid >> 5) * 8 * KB,
              64 * half, h);
    bulk_commit();
    bulk_wait_all();
  }
}

// ---------------------------------------------------------------------------
// k_bwd_state.  Bound by HBM: 104 KB read and 64 KB written per chunk, 247 us at B8 H16 T4096
// (5.7 TB/s); with few sequences by its chain, ~6 K cycles a chunk (98 us at B2 H16 T1999).
// 16 warps; warp w holds TMEM lanes 32 (w % 4) .. + 31 and value columns
// 32 (w / 4) .. + 31 of dS.  Per chunk: dS -> fp16 tile; MMA dR; dR -> fp16 hi + lo;
// MMA dS.  A_qk, K_tail and dO are double-buffered bulk copies; Qbar, W (needed
// last) and S_in (for dgamma_C, needed first) are loaded again as soon as they have been read.
constexpr int SB_AQ = 0, SB_KT = 8 * KB, SB_DO = 24 * KB, SB_BUF = 40 * KB;
constexpr int SO_QB = 2 * SB_BUF, SO_WN = SO_QB + 16 * KB, SO_SIN = SO_WN + 16 * KB;
constexpr int SO_DSH = SO_SIN + 32 * KB, SO_DRH = SO_DSH + 32 * KB, SO_DRL = SO_DRH + 16 * KB;
constexpr int SO_PART = SO_DRL + 16 * KB, SO_SC = SO_PART + 256;
constexpr int SO_BAR = SO_SC + 2 * 512, STATE_SMEM = SO_BAR + 64 + 1024;  // SC: gamma_C [128], two buffers
static_assert(STATE_SMEM <= 232448, "shared memory");

__global__ void __launch_bounds__(BT, 1)
    k_bwd_state(const __grid_constant__ CUtensorMap mdo, const __grid_constant__ CUtensorMap m0,
                const __grid_constant__ CUtensorMap m1, const __grid_constant__ CUtensorMap m2,
                const __grid_constant__ CUtensorMap m3, const __grid_constant__ CUtensorMap mt,
                const SplitParams P) {
  const Args &a = P.a;
  extern __shared__ unsigned char smraw[];
  unsigned char *sm =
      reinterpret_cast<unsigned char *>((reinterpret_cast<uintptr_t>(smraw) + 1023) & ~uintptr_t(1023));
  unsigned char *dsh = sm + SO_DSH, *drh = sm + SO_DRH, *drl = sm + SO_DRL;
  float *s_part = reinterpret_cast<float *>(sm + SO_PART), *s_misc = s_part + 32;
  uint64_t *bars = reinterpret_cast<uint64_t *>(sm + SO_BAR);
  uint64_t *bar_full = bars, *bar_r = bars + 2, *bar_s = bars + 3, *bar_w = bars + 4, *bar_i = bars + 5;
  uint32_t *s_tbase = reinterpret_cast<uint32_t *>(bars + 6);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, wq = warp & 3, wg = warp >> 2;
  const int bh = blockIdx.x, b = bh / a.H, h = bh % a.H, NC = (a.T + CM - 1) / CM;
  const int warp_u = __shfl_sync(0xffffffffu, warp, 0);  // warp-uniform: the issue loops stay uniform

  if (tid == 0) {
    mbar_init(bar_full, 5);  // arrivals: one per issuing thread
    mbar_init(bar_full + 1, 5);
    mbar_init(bar_w, 2);
    mbar_init(bar_i, 1);
    mbar_init(bar_r, 1);
    mbar_init(bar_s, 1);
    fence_mbar_init();
    prefetch_tmap(&mdo);
  }
  if (warp == 0) {
    tmem_alloc(s_tbase, 512);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t TS = *s_tbase, TX = TS + 128;
  const uint32_t lane_base = (uint32_t)(32 * wq) << 16;
  auto record = [&](int c) { return a.fSin + ((size_t)bh * NC + c) * kCtxBytes; };
  // The copies are issued one per warp (lane 0): a single thread's run of them would hold
  // up the chain of products.  Warps 1..7 load, 8..11 store dS, 12..15 store dR.
  auto issue = [&](int c, int buf) {  // A_qk, K_tail, dO, gamma_C
    const unsigned char *rec = record(c);
    unsigned char *d = sm + buf * SB_BUF, *sc = sm + SO_SC + buf * 512;
    uint64_t *bar = bar_full + buf;
    switch (lane == 0 ? warp : -1) {
      case 1: mbar_expect_tx(bar, 8192); bulk_g2s(d + SB_AQ, rec + kCtxAqk, 8192, bar); break;
      case 2:
        mbar_expect_tx(bar, 16384);
        for (int s = 0; s < 2; ++s) box_load(d + SB_KT + s * 8192, box_at(P.s, a, m2, mt, 2, b, c), bar, 64 * s, h);
        break;
      case 3: mbar_expect_tx(bar, 8192); tma_load_4d(d + SB_DO, &mdo, bar, 0, h, c * CM, b); break;
      case 4: mbar_expect_tx(bar, 8192); tma_load_4d(d + SB_DO + 8192, &mdo, bar, 64, h, c * CM, b); break;
      case 5: mbar_expect_tx(bar, 512); bulk_g2s(sc, rec + kCtxGa + 63 * D * 4, 512, bar); break;
    }
  };
  auto issue_sin = [&](int c) {
    if (lane == 0 && warp == 6) {
      mbar_expect_tx(bar_i, 32768);
      bulk_g2s(sm + SO_SIN, record(c) + kCtxS, 32768, bar_i);
    }
  };
  auto issue_w = [&](int c) {  // Qbar, -W
    const unsigned char *rec = record(c);
    switch (lane == 0 ? warp : -1) {
      case 6:
        mbar_expect_tx(bar_w, 16384);
        for (int s = 0; s < 2; ++s) box_load(sm + SO_QB + s * 8192, box_at(P.s, a, m3, mt, 3, b, c), bar_w, 64 * s, h);
        break;
      case 7: mbar_expect_tx(bar_w, 16384); bulk_g2s(sm + SO_WN, rec + kCtxW, 16384, bar_w); break;
      case 8:  // the next chunk's, into L2
        if (c > 0) {
          bulk_prefetch_l2(rec - kCtxBytes + kCtxS, 32768);
          bulk_prefetch_l2(rec - kCtxBytes + kCtxW, 16384);
          for (int s = 0; s < 2; ++s) {
            tma_prefetch_4d(&m2, 64 * s, h, (c - 1) * CM, b);
            tma_prefetch_4d(&m3, 64 * s, h, (c - 1) * CM, b);
          }
        }
        break;
    }
  };
  issue_sin(NC - 1);
  issue(NC - 1, 0);

  // cotangent scale lambda = 2^-e with max(|dO|, |dS_T|) * lambda in [1, 2)
  {
    float m = 0.f;
    const unsigned char *dO = static_cast<const unsigned char *>(a.dO);
#pragma unroll 4
    for (int e = tid; e < a.T * 16; e += BT) {
      const uint4 u = *reinterpret_cast<const uint4 *>(dO + (tok_index(a, b, e >> 4, h) * D) * 2 + (e & 15) * 16);
      float v[8];
      unpack_bf8(u, v);
#pragma unroll
      for (int j = 0; j < 8; ++j) m = fmaxf(m, fabsf(v[j]));
    }
    if (a.dST) {
      const float4 *src = reinterpret_cast<const float4 *>(a.dST + (size_t)bh * D * D);
      for (int e = tid; e < D * D / 4; e += BT) {
        const float4 x = src[e];
        m = fmaxf(fmaxf(m, fmaxf(fabsf(x.x), fabsf(x.y))), fmaxf(fabsf(x.z), fabsf(x.w)));
      }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
    if (lane == 0) s_part[warp] = m;
    __syncthreads();
    if (tid == 0) {
      float mm = 0.f;
      for (int w = 0; w < BT / 32; ++w) mm = fmaxf(mm, s_part[w]);
      float lam = 1.f;
      if (mm > 0.f && isfinite(mm)) {
        int e;
        frexpf(mm, &e);  // mm = f 2^e, f in [0.5, 1)
        e = max(e, -100);
        lam = ldexpf(1.f, 1 - e);
      }
      s_misc[0] = lam;
    }
    __syncthreads();
  }
  const float lam = s_misc[0];

  const int i = 32 * wq + lane, j0 = 32 * wg;  // this thread's row and first column of dS
  for (int c0 = 0; c0 < 32; c0 += 16) {
    float v[16];
#pragma unroll
    for (int u = 0; u < 16; ++u) v[u] = 0.f;
    if (a.dST) {
      const float4 *src = reinterpret_cast<const float4 *>(a.dST + ((size_t)bh * D + i) * D + j0 + c0);
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const float4 x = src[u];
        v[4 * u] = lam * x.x; v[4 * u + 1] = lam * x.y; v[4 * u + 2] = lam * x.z; v[4 * u + 3] = lam * x.w;
      }
    }
    tmem_st16(TS + lane_base + j0 + c0, v);
  }
  tmem_st_wait();

  bool ok = true;
  for (int it = 0; it < NC; ++it) {
    const int c = NC - 1 - it, buf = it & 1;
    unsigned char *d = sm + buf * SB_BUF;
    // ---- [1] dS -> fp16 tile; dgamma_C part; dS <- gamma_C dS; lambda dO -> fp16 in place
    ok = mbar_wait(bar_full + buf, (it >> 1) & 1, kWaitIters) && ok;
    ok = mbar_wait(bar_i, it & 1, kWaitIters) && ok;
    if (it > 0) ok = mbar_wait(bar_s, (it - 1) & 1, kWaitIters) && ok;
    issue_w(c);  // (MMA dS of the previous chunk has read the last ones)
    tc_fence_after();
    {
      const float gC = reinterpret_cast<const float *>(sm + SO_SC + buf * 512)[i];
      float dgc = 0.f;
#pragma unroll
      for (int c0 = 0; c0 < 32; c0 += 16) {
        float v[16], s[16];
        tmem_ld16(TS + lane_base + j0 + c0, v);
        const int sl = j0 >> 6, cc0 = ((j0 & 63) + c0) >> 3;
        sm16(dsh, sl * 16384 + chunk_off(i, cc0)) = pack_h8(v);
        sm16(dsh, sl * 16384 + chunk_off(i, cc0 + 1)) = pack_h8(v + 8);
        unpack_h8(sm16(sm + SO_SIN, sl * 16384 + chunk_off(i, cc0)), s);
        unpack_h8(sm16(sm + SO_SIN, sl * 16384 + chunk_off(i, cc0 + 1)), s + 8);
#pragma unroll
        for (int u = 0; u < 16; ++u) {
          dgc = fmaf(v[u], s[u], dgc);
          v[u] *= gC;
        }
        tmem_st16(TS + lane_base + j0 + c0, v);
      }
      *small_dgc(P.s, a, b, h, c, wg * D + i) = dgc;
#pragma unroll
      for (int e = tid; e < 64 * 16; e += BT) {
        const uint32_t off = SB_DO + ((e & 15) >> 3) * 8192 + chunk_off(e >> 4, e & 7);
        float v[8];
        unpack_bf8(sm16(d, off), v);
#pragma unroll
        for (int j = 0; j < 8; ++j) v[j] *= lam;
        sm16(d, off) = pack_h8(v);
      }
    }
    if (lane == 0 && warp >= 12) bulk_wait_read();  // dR of the previous chunk has left its tiles
    tmem_st_wait();
    fence_proxy_async();
    tc_fence_before();
    if (!__syncthreads_and(ok)) {
      ok = false;
      break;
    }
    // ---- [2] MMA: X = (A_qk^T dO + K_tail dS)^T = dR^T, [j][t]
    if (warp_u == 0) {
      tc_fence_after();
      const uint32_t lead = elect_one();
      const uint32_t id11 = idesc_f16(128, 64, 1, 1);
      const uint64_t aq = mdesc(d + SB_AQ, 8192), dov = mdesc(d + SB_DO, 8192), kt = mdesc(d + SB_KT, 8192),
                     ds = mdesc(dsh, 16384);
#pragma unroll
      for (int kk = 0; kk < 4; ++kk) umma_if(lead, TX, step(dov, kk * 2048), step(aq, kk * 2048), id11, kk > 0);
#pragma unroll
      for (int kk = 0; kk < 8; ++kk) umma_if(lead, TX, step(ds, kk * 2048), step(kt, kk * 2048), id11, 1);
      commit_if(lead, bar_r);
    }
    if (c > 0) {
      issue(c - 1, buf ^ 1);
      issue_sin(c - 1);
    }
    if (lane == 0 && warp >= 8 && warp < 12) {  // dS: rows i 0..63 in m0's tiles, 64..127 in m1's
      const int s = warp & 1;
      if (warp < 10) box_store(box_at(P.s, a, m0, mt, 0, b, c), dsh + s * 16384, 64 * s, h);
      else box_store(box_at(P.s, a, m1, mt, 1, b, c), dsh + s * 16384 + 8192, 64 * s, h);
      bulk_commit();
    }
    if (warp >= 4 && warp < 8) {  // the small values of this chunk
      const int ii = tid - 128;
      *small_slot(P.s, a, b, h, c, ii) = 0;
      if (ii == 0) *small_lam(P.s, a, b, h, c) = lam;
    }
    // ---- [3] dR^T -> fp16 hi + lo, [j][t]
    ok = mbar_wait(bar_r, it & 1, kWaitIters) && ok;
    tc_fence_after();
    {
      float x[16];
      tmem_ld16(TX + lane_base + 16 * wg, x);
      uint4 l0, l1;
      sm16(drh, chunk_off(i, 2 * wg)) = split_h8(x, &l0);
      sm16(drh, chunk_off(i, 2 * wg + 1)) = split_h8(x + 8, &l1);
      sm16(drl, chunk_off(i, 2 * wg)) = l0;
      sm16(drl, chunk_off(i, 2 * wg + 1)) = l1;
    }
    if (lane == 0 && warp >= 8 && warp < 12) bulk_wait_read();  // the dS tile has left shared memory
    fence_proxy_async();
    tc_fence_before();
    __syncthreads();
    // ---- [4] MMA: dS += Qbar^T dO - W^T dR
    if (warp_u == 0) {
      ok = mbar_wait(bar_w, it & 1, kWaitIters) && ok;
      tc_fence_after();
      const uint32_t lead = elect_one();
      const uint32_t id01 = idesc_f16(128, 128, 0, 1), id10 = idesc_f16(128, 128, 1, 0);
      const uint64_t qb = kdesc(sm + SO_QB), dov = mdesc(d + SB_DO, 8192), wn = mdesc(sm + SO_WN, 8192),
                     dr = kdesc(drh);
#pragma unroll
      for (int kk = 0; kk < 4; ++kk) {
        umma_if(lead, TS, step(qb, kk * 32), step(dov, kk * 2048), id01, 1);
        umma_if(lead, TS, step(wn, kk * 2048), step(dr, kk * 32), id10, 1);
      }
      commit_if(lead, bar_s);
    }
    if (lane == 0 && warp >= 12) {  // dR^T rows j 0..63, 64..127, over K_tail and Qbar, which have been read
      const int s = warp & 1;
      ok = mbar_wait(bar_w, it & 1, kWaitIters) && ok;
      if (warp < 14) box_store(box_at(P.s, a, m2, mt, 2, b, c), drh + s * 8192, 64 * s, h);
      else box_store(box_at(P.s, a, m3, mt, 3, b, c), drl + s * 8192, 64 * s, h);
      bulk_commit();
    }
  }
  if (ok) ok = mbar_wait(bar_s, (NC - 1) & 1, kWaitIters);
  if (!__syncthreads_and(ok)) {
    if (tid == 0) {
      atomicExch(a.status, (unsigned)KDN_ERR_TIMEOUT);
      // copies and MMAs in flight land before the CTA's memory goes away
      for (int k = 0; k < 6; ++k) {
        mbar_wait(bars + k, 0, 1u << 14);
        mbar_wait(bars + k, 1, 1u << 14);
      }
    }
  }
  if (lane == 0 && warp >= 8) bulk_wait_all();
  tc_fence_before();
  __syncthreads();
  if (warp == 0) tmem_dealloc(TS, 512);
}

// ---------------------------------------------------------------------------
// k_bwd_chunk.  Bound by the chain of a chunk's stages (ncu, B2 H16 T4096: 40 % of the issue
// slots, tensor pipe 8 %; the waits are on tensor-memory reads, barriers and instruction
// fetches): ~32 K cycles a chunk, of which the four tensor-core rounds with their read-outs 13 K
// and the per-channel passes 14 K.  872 us at B8 H16 T4096 (with the tiles and k_bwd_state 1295; the
// one-kernel sweep 1317), 165 us at B2 H16 T1999 logits (285; 668).
// Shared-memory map (bytes from the 1024-aligned base), with the sequence
// of tenants within a chunk; the next chunk's tiles arrive as their buffers fall free.
constexpr int O_RKQ = 0;         // raw k | q, interleaved per 64-channel slab
constexpr int O_SIN = 32 * KB;   // S_in fp16 [i][j] -> Kbar^T hi | Qbar^T hi
constexpr int O_RV = 64 * KB;    // Y fp16 [t][j] -> dW^T bf16 [i][t]
constexpr int O_RDO = 80 * KB;   // raw dO -> lambda dO fp16 -> Qbar^T lo
constexpr int O_AH = 96 * KB;    // A fp16 [t][s]
constexpr int O_AB = 104 * KB;   // gamma, tokens 0..15 -> A bf16 -> (logit gates) omega, channels 0..63
constexpr int O_DT = 112 * KB;   // gamma, tokens 16..31 -> dT bf16
constexpr int O_AQ = 120 * KB;   // gamma, tokens 32..47 -> dA^T fp16 [s][t] -> omega, channels 64..127
constexpr int O_WN = 128 * KB;   // dR^T hi fp16 [j][t] -> Kk^T hi
constexpr int O_KT = 144 * KB;   // dR^T lo fp16 [j][t]
constexpr int O_G = 160 * KB;    // phat -> dS fp16 [i][j] -> dA_qk^T hi | lo, Kk^T lo (then X)
constexpr int O_RH = 192 * KB;   // R fp16 [t][j] -> dv tile
constexpr int O_GA3 = 208 * KB;  // gamma, tokens 48..63
constexpr int BUF_END = 216 * KB;
constexpr int O_DAQ = O_G, O_KKL = O_G + 16 * KB, O_XT = O_G + 24 * KB;
constexpr int OFF_SM = BUF_END;
constexpr int SMALL_FLOATS = 64 * 8 + 512 + 128 * 2 + 32 + 128 + 772;
constexpr int OFF_BAR = OFF_SM + SMALL_FLOATS * 4;
constexpr int CHUNK_SMEM = OFF_BAR + 80 + 1024;
static_assert(CHUNK_SMEM <= 232448, "shared memory");

template <int G>  // G: logit gates
__global__ void __launch_bounds__(BT, 1)
    k_bwd_chunk(const __grid_constant__ CUtensorMap mq, const __grid_constant__ CUtensorMap mk,
                const __grid_constant__ CUtensorMap mdo, const __grid_constant__ CUtensorMap mw,
                const __grid_constant__ CUtensorMap m0, const __grid_constant__ CUtensorMap m1,
                const __grid_constant__ CUtensorMap m2, const __grid_constant__ CUtensorMap m3,
                const __grid_constant__ CUtensorMap mt,
                const SplitParams P) {
  const Args &a = P.a;
  extern __shared__ unsigned char smraw[];
  unsigned char *sm =
      reinterpret_cast<unsigned char *>((reinterpret_cast<uintptr_t>(smraw) + 1023) & ~uintptr_t(1023));
  unsigned char *rkq = sm + O_RKQ, *sin = sm + O_SIN, *rdo = sm + O_RDO;
  float *s_r = reinterpret_cast<float *>(sm + OFF_SM);  // [64] r_t
  float *s_ri = s_r + 64;       // [64] 1 / r_t
  float *s_si = s_ri + 64;      // [64] 1 / s_t
  float *s_ds = s_si + 64;      // [64] ds_t
  float *s_fr = s_ds + 64;      // [64] d r_t / d z_t (1 unless the gates are logits)
  float *s_red = s_fr + 192;    // [4][64] per-warp partial sums over channels (ds_t)
  float *s_red2 = s_red + 256;  // [4][64] (dr_t)
  float *s_gC = s_red2 + 256;   // [128] gamma_C
  float *s_dp = s_gC + 128;     // [128] uncertainty cotangent leaving the chunk
  float *s_misc = s_dp + 128;   // [0] lambda
  int *s_next = reinterpret_cast<int *>(s_misc + 8);
  float *s_pin = s_misc + 32;   // [128] p entering the chunk
  float *n_tok = s_pin + 128;   // next chunk: [2][64] s_t, z_t; [128] p in; [4][128] dgamma_C; lambda
  float *n_pin = n_tok + 128, *n_dgc = n_pin + 128, *n_lam = n_dgc + 512;
  uint64_t *bars = reinterpret_cast<uint64_t *>(sm + OFF_BAR);
  uint64_t *bar_a = bars, *bar_b = bars + 1, *bar_mma = bars + 2, *bar_g = bars + 3, *bar_d = bars + 4,
           *bar_w = bars + 5;
  uint32_t *s_tbase = reinterpret_cast<uint32_t *>(bars + 6);

  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int warp_u = __shfl_sync(0xffffffffu, warp, 0);  // warp-uniform: the issue loops stay uniform
  const int wq = warp & 3, wg = warp >> 2;  // TMEM lane quarter, column group
  const int ci = tid & (D - 1), qq = tid >> 7, t0 = 16 * qq;  // channel view: channel, token quarter
  const int NC = (a.T + CM - 1) / CM, BH = a.B * a.H, njobs = BH * NC;
  const float tau = a.tau, mu = a.mu;

  if (tid == 0) {
    mbar_init(bar_a, 12);  // arrivals: one per issuing thread
    mbar_init(bar_b, 2);
    mbar_init(bar_mma, 2);
    mbar_init(bar_g, 5);
    mbar_init(bar_d, 4);
    mbar_init(bar_w, 2);
    fence_mbar_init();
    prefetch_tmap(&mq);
    prefetch_tmap(&mk);
    prefetch_tmap(&mdo);
  }
  if (warp == 0) {
    tmem_alloc(s_tbase, 512);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tb = *s_tbase;
  const uint32_t TPH = tb, TGM = tb + 64, X0 = tb + 128, X1 = tb + 192, X2 = tb + 256, X3 = tb + 320,
                 X4 = tb + 384, X5 = tb + 448;
  const uint32_t lane_base = (uint32_t)(32 * wq) << 16;

  // Jobs in reverse time order: the chunk whose dp a job awaits has a lower ticket, so it
  // is finished or held by a CTA that waits only for lower tickets still.  One thread
  // takes the next ticket and leaves (job, b, h, c) in shared memory.
  struct Job { int j, b, h, c; const unsigned char *rec; size_t rc; };
  auto take = [&]() {
    const unsigned u = atomicAdd(P.ticket, 1u);  // (unsigned: no job from whatever else the word may hold)
    const int j = u < (unsigned)njobs ? (int)u : njobs, jj = j < njobs ? j : 0, bh = jj % BH;
    s_next[0] = j;
    s_next[1] = bh / a.H;
    s_next[2] = bh % a.H;
    s_next[3] = NC - 1 - jj / BH;
  };
  auto job_at = [&]() {
    Job o;
    o.j = s_next[0];
    o.b = s_next[1];
    o.h = s_next[2];
    o.c = s_next[3];
    o.rc = (size_t)(o.b * a.H + o.h) * NC + o.c;
    o.rec = a.fSin + o.rc * kCtxBytes;
    return o;
  };
  // The copies of a chunk's tiles, spread over lane 0 of the warps: one thread issuing them
  // all (25 operations) held the CTA up for ~6 K cycles a chunk.  Each thread
  // arrives with its own bytes; R comes from the thread that stored dv from its buffer.
  // gamma's tokens 0..15 and 32..47 (logit gates: their buffers hold omega during the passes)
  auto issue_g2 = [&](const Job &o) {
    switch (lane == 0 ? warp : -1) {
      case 14: mbar_expect_tx(bar_g, 8192); bulk_g2s(sm + O_AB, o.rec + kCtxGa, 8192, bar_g); break;
      case 15: mbar_expect_tx(bar_g, 8192); bulk_g2s(sm + O_AQ, o.rec + kCtxGa + 16384, 8192, bar_g); break;
    }
  };
  auto issue_a = [&](const Job &o) {
    const int t = o.c * CM;
    switch (lane == 0 ? warp : -1) {
      case 0: mbar_expect_tx(bar_a, 32768); bulk_g2s(sin, o.rec + kCtxS, 32768, bar_a); break;
      case 1: mbar_expect_tx(bar_a, 16384); bulk_g2s(sm + O_RV, o.rec + kCtxY, 16384, bar_a); break;
      case 2: mbar_expect_tx(bar_a, 8192); bulk_g2s(sm + O_AH, o.rec + kCtxA, 8192, bar_a); break;
      case 3: mbar_expect_tx(bar_a, 8192); box_load(sm + O_WN, box_at(P.s, a, m2, mt, 2, o.b, o.c), bar_a, 0, o.h); break;
      case 4: mbar_expect_tx(bar_a, 8192); box_load(sm + O_WN + 8192, box_at(P.s, a, m2, mt, 2, o.b, o.c), bar_a, 64, o.h); break;
      case 5: mbar_expect_tx(bar_a, 8192); box_load(sm + O_KT, box_at(P.s, a, m3, mt, 3, o.b, o.c), bar_a, 0, o.h); break;
      case 6: mbar_expect_tx(bar_a, 8192); box_load(sm + O_KT + 8192, box_at(P.s, a, m3, mt, 3, o.b, o.c), bar_a, 64, o.h); break;
      case 7:
        bulk_wait_read();  // the dv tile has left the R buffer
        mbar_expect_tx(bar_a, 16384);
        bulk_g2s(sm + O_RH, o.rec + kCtxR, 16384, bar_a);
        break;
      case 8: mbar_expect_tx(bar_b, 8192); tma_load_4d(rdo, &mdo, bar_b, 0, o.h, t, o.b); break;
      case 9: mbar_expect_tx(bar_b, 8192); tma_load_4d(rdo + 8192, &mdo, bar_b, 64, o.h, t, o.b); break;
      case 10: mbar_expect_tx(bar_g, 32768); bulk_g2s(sm + O_G, o.rec + kCtxPh, 32768, bar_g); break;
      case 11: mbar_expect_tx(bar_g, 8192); bulk_g2s(sm + O_DT, o.rec + kCtxGa + 8192, 8192, bar_g); break;
      case 12: mbar_expect_tx(bar_g, 8192); bulk_g2s(sm + O_GA3, o.rec + kCtxGa + 24576, 8192, bar_g); break;
      case 13:  // dS
      case 14: {
        const Box x = warp == 13 ? box_at(P.s, a, m0, mt, 0, o.b, o.c) : box_at(P.s, a, m1, mt, 1, o.b, o.c);
        for (int s = 0; s < 2; ++s) tma_prefetch_4d(x.m, 64 * s, o.h, x.t, x.b);
        break;
      }
      case 15:
        if (G) bulk_prefetch_l2(o.rec + kCtxGa, 24576);
        break;
    }
    if (!G) issue_g2(o);
  };
  auto issue_kq = [&](const Job &o) {
    const int t = o.c * CM;
    switch (lane == 0 ? warp : -1) {
      case 8: mbar_expect_tx(bar_a, 8192); tma_load_4d(rkq, &mk, bar_a, 0, o.h, t, o.b); break;
      case 9: mbar_expect_tx(bar_a, 8192); tma_load_4d(rkq + 8192, &mq, bar_a, 0, o.h, t, o.b); break;
      case 10: mbar_expect_tx(bar_a, 8192); tma_load_4d(rkq + 16384, &mk, bar_a, 64, o.h, t, o.b); break;
      case 11: mbar_expect_tx(bar_a, 8192); tma_load_4d(rkq + 24576, &mq, bar_a, 64, o.h, t, o.b); break;
    }
  };
  // the next job's small values, by asynchronous copies: loads into registers would hold up
  // the next wait on a barrier, and be spilled across the passes
  auto load_small = [&](const Job &o) {
    if (tid < 16) cp16(n_tok + 4 * tid, o.rec + kCtxTok + 16 * tid);
    else if (tid < 32) cp16(n_tok + 4 * tid, small_z(P.s, a, o.b, o.h, o.c) + 4 * (tid - 16));
    else if (tid < 64) cp16(n_pin + 4 * (tid - 32), a.fpin + o.rc * D + 4 * (tid - 32));
    else if (tid < 192) cp16(n_dgc + 4 * (tid - 64), small_dgc(P.s, a, o.b, o.h, o.c, 4 * (tid - 64)));
    else if (tid == 192) cp16(n_lam, small_lam(P.s, a, o.b, o.h, o.c));
  };
  if (tid == 0) take();
  __syncthreads();
  Job on = job_at();
  if (on.j < njobs) {
    issue_a(on);
    issue_kq(on);
    if (G) issue_g2(on);
    load_small(on);
    cp_commit();
    cp_wait<0>();
  }
  __syncthreads();  // (s_next is taken again)
  uint32_t mma_phase = 0;
  bool ok = true;
  auto mma_poll = [&]() -> bool {
    const bool r = mbar_wait(bar_mma, mma_phase & 1, kWaitIters);
    ++mma_phase;
    return r;
  };
  auto raw_k = [&](int t) { return bf(rkq, 16384, t, ci); };
  auto raw_q = [&](int t) { return bf(rkq + 8192, 16384, t, ci); };

  for (int it = 0; on.j < njobs; ++it) {
    const Job o = on;
    const int b = o.b, h = o.h, c = o.c;
    // ---- [1] the chunk's tiles and gains have landed; per-token scalars
    bool mm_ok = mbar_wait(bar_a, it & 1, kWaitIters);
    mm_ok = mbar_wait(bar_g, it & 1, kWaitIters) && mm_ok;
    if (tid < CM) {
      const bool live = c * CM + tid < a.T;
      const float z = n_tok[CM + tid], nr = live ? gate_r(G, a.rmin, z) : 1.f;
      s_r[tid] = nr;
      s_ri[tid] = 1.f / nr;
      s_fr[tid] = live ? dgate_sig(G, z) : 1.f;
      s_si[tid] = 1.f / n_tok[tid];
    }
    if (qq == 1) s_pin[ci] = n_pin[ci];
    const float lam = n_lam[0], invl = 1.f / lam;
    float dgc = n_dgc[tid];  // this thread's part of dgamma_C for channel ci
    // ---- [2] phat and gamma -> TMEM (lane = channel)
    float ph[16], ga[16];
    {
      const unsigned char *gs = sm + (qq < 2 ? O_AB + qq * 8192 : qq == 2 ? O_AQ : O_GA3);
      const float *gp = reinterpret_cast<const float *>(gs) + ci;
      const float *pp = reinterpret_cast<const float *>(sm + O_G) + t0 * D + ci;
#pragma unroll
      for (int j = 0; j < 16; ++j) {
        ga[j] = gp[j * D];
        ph[j] = pp[j * D];
      }
      tmem_st16(TPH + lane_base + t0, ph);
      tmem_st16(TGM + lane_base + t0, ga);
      if (qq == 3) {
        s_gC[ci] = ga[15];
        check_gamma_range(ga[15], a.status);
      }
      tmem_st_wait();
    }
    fence_proxy_async();
    if (!__syncthreads_and(mm_ok)) {
      ok = false;
      break;
    }
    if (lane == 0 && warp >= 12) {  // dS over phat
      const int s = (warp >> 1) & 1;
      mbar_expect_tx(bar_d, 8192);
      if (warp & 1) box_load(sm + O_G + s * 16384 + 8192, box_at(P.s, a, m1, mt, 1, b, c), bar_d, 64 * s, h);
      else box_load(sm + O_G + s * 16384, box_at(P.s, a, m0, mt, 0, b, c), bar_d, 64 * s, h);
    }
    // ---- [3] A -> bf16; lambda dO -> fp16 in place
    {
      float v[8];
      unpack_h8(sm16(sm + O_AH, tid * 16), v);
      sm16(sm + O_AB, tid * 16) = pack_bf8(v);
    }
    mm_ok = mbar_wait(bar_b, it & 1, kWaitIters);
#pragma unroll
    for (int e = tid; e < 64 * 16; e += BT) {
      const uint32_t off = ((e & 15) >> 3) * 8192 + chunk_off(e >> 4, e & 7);
      float v[8];
      unpack_bf8(sm16(rdo, off), v);
#pragma unroll
      for (int j = 0; j < 8; ++j) v[j] *= lam;
      sm16(rdo, off) = pack_h8(v);
    }
    fence_proxy_async();
    tc_fence_before();
    if (!__syncthreads_and(mm_ok)) {
      ok = false;
      break;
    }
    // ---- round 1.  X4 = dA_qk^T (before masking), X1 = -dW^T = (dR S_in^T)^T, X2 = dA^T = (dR Y^T)^T
    //      (dA = dR V^T + dW Kbar^T = dR Y^T, since dW = -dR S_in^T and Y = V - Kbar S_in),
    //      X3 = (dO S_in^T)^T, X5 = dV^T = (A^T dR)^T (dR as hi + lo), X0 = dK_tail^T
    //      (two warps issue)
    if (warp_u == 0) {
      tc_fence_after();
      const uint32_t lead = elect_one();
      const uint32_t id00 = idesc_f16(128, 64, 0, 0), id01 = idesc_f16(128, 64, 0, 1);
      const uint64_t d0 = kdesc(rdo), r0 = mdesc(sm + O_WN, 8192), s0 = kdesc(sin), rr = kdesc(sm + O_RH),
                     y0 = kdesc(sm + O_RV);
#pragma unroll
      for (int kk = 0; kk < 8; ++kk) {
        const uint32_t o8 = (kk >> 2) * 8192 + (kk & 3) * 32, o16 = (kk >> 2) * 16384 + (kk & 3) * 32;
        const uint64_t dov = step(d0, o8), drv = step(r0, kk * 2048), sv = step(s0, o16);
        umma_if(lead, X4, step(rr, o8), dov, id00, kk > 0);
        umma_if(lead, X1, sv, drv, id01, kk > 0);
        umma_if(lead, X2, step(y0, o8), drv, id01, kk > 0);
        umma_if(lead, X3, sv, dov, id00, kk > 0);
      }
      commit_if(lead, bar_mma);
    } else if (warp_u == 4) {
      tc_fence_after();
      const uint32_t lead = elect_one();
      const uint32_t id00 = idesc_f16(128, 64, 0, 0), id01 = idesc_f16(128, 64, 0, 1);
      const uint64_t a0 = mdesc(sm + O_AH, 8192), rh = kdesc(sm + O_WN), rl = kdesc(sm + O_KT),
                     ds = kdesc(sm + O_G), rr = kdesc(sm + O_RH);
#pragma unroll
      for (int kk = 0; kk < 4; ++kk) {
        umma_if(lead, X5, step(rh, kk * 32), step(a0, kk * 2048), id01, kk > 0);
        umma_if(lead, X5, step(rl, kk * 32), step(a0, kk * 2048), id01, 1);
      }
      mm_ok = mbar_wait(bar_d, it & 1, kWaitIters);
#pragma unroll
      for (int kk = 0; kk < 8; ++kk)
        umma_if(lead, X0, step(ds, (kk >> 2) * 16384 + (kk & 3) * 32), step(rr, (kk >> 2) * 8192 + (kk & 3) * 32), id00,
                  kk > 0);
      commit_if(lead, bar_mma);
    } else if (tid == 256) {
      take();  // the next job, known to every thread after the barrier below
    }
    mm_ok = mma_poll() && mm_ok;
    tc_fence_after();
    // ---- dA_qk^T (masked to s <= t) -> hi/lo bf16 [s][t]; dW^T -> bf16; dA^T -> fp16; dV^T -> dv;
    //      X0 <- gamma_C dK_tail^T (start of dKk^T) and its dgamma_C part; the second operand set
    {
      const int j = 32 * wq + lane, tc0 = 16 * wg;
      float v[16];
      tmem_ld16(X1 + lane_base + tc0, v);
#pragma unroll
      for (int u = 0; u < 16; ++u) v[u] = -v[u];
      sm16(sm + O_RV, chunk_off(j, tc0 >> 3)) = pack_bf8(v);
      sm16(sm + O_RV, chunk_off(j, (tc0 >> 3) + 1)) = pack_bf8(v + 8);
      tmem_ld16(X5 + lane_base + tc0, v);
      {  // into the R tile, in the layout of the TMA box
        unsigned char *slab = sm + O_RH + (j >> 6) * 8192;
#pragma unroll
        for (int u = 0; u < 16; ++u)
          *reinterpret_cast<__nv_bfloat16 *>(slab + chunk_off(tc0 + u, (j & 63) >> 3) + 2 * (j & 7)) =
              __float2bfloat16_rn(v[u] * invl);
      }
      if (wq < 2) {
        tmem_ld16(X4 + lane_base + tc0, v);
#pragma unroll
        for (int u = 0; u < 16; ++u)
          if (tc0 + u < j) v[u] = 0.f;
        uint4 lo0, lo1;
        sm16(sm + O_DAQ, chunk_off(j, tc0 >> 3)) = split_bf8(v, &lo0);
        sm16(sm + O_DAQ, chunk_off(j, (tc0 >> 3) + 1)) = split_bf8(v + 8, &lo1);
        sm16(sm + O_DAQ + 8192, chunk_off(j, tc0 >> 3)) = lo0;
        sm16(sm + O_DAQ + 8192, chunk_off(j, (tc0 >> 3) + 1)) = lo1;
        tmem_ld16(X2 + lane_base + tc0, v);
        sm16(sm + O_AQ, chunk_off(j, tc0 >> 3)) = pack_h8(v);
        sm16(sm + O_AQ, chunk_off(j, (tc0 >> 3) + 1)) = pack_h8(v + 8);
      }
    }
    {
      float x[16], v[16];
      tmem_ld16(TPH + lane_base + t0, ph);
      tmem_ld16(TGM + lane_base + t0, ga);
      tmem_ld16(X0 + lane_base + t0, x);
      const float gC = s_gC[ci];
#pragma unroll
      for (int j = 0; j < 16; ++j) {
        const float kk = raw_k(t0 + j);
        v[j] = ga[j] * kk;                                            // Kbar
        ph[j] = __fdividef(ph[j] * s_si[t0 + j] * kk, ga[j]);          // Kk
        dgc += x[j] * ph[j];
        x[j] *= gC;
      }
      tmem_st16(X0 + lane_base + t0, x);
      st_row16_bf(sin, ci, qq, v);                       // Kbar^T hi
      st_row16_split(sm + O_WN, sm + O_KKL, ci, qq, ph);  // Kk^T hi / lo
#pragma unroll
      for (int j = 0; j < 16; ++j) v[j] = tau * ga[j] * raw_q(t0 + j);
      st_row16_split(sin + 16384, rdo, ci, qq, v);  // Qbar^T hi / lo
    }
    tmem_st_wait();
    fence_proxy_async();
    tc_fence_before();
    if (!__syncthreads_and(mm_ok)) {
      ok = false;
      break;
    }
    // ---- round 2.  X3 += (dA_qk Kk)^T, X0 += (dA_qk^T Qbar)^T (hi/lo bf16 pairs), X4 = A^T dA (fp16),
    //      X2 = (A^T dW)^T
    on = job_at();
    if (warp_u == 0) {
      tc_fence_after();
      const uint32_t lead = elect_one();
      const uint32_t id01 = idesc_bf16(128, 64, 0, 1), ih10 = idesc_f16(128, 64, 1, 0);
      const uint64_t a0 = mdesc(sm + O_AH, 8192), da = kdesc(sm + O_AQ), kh0 = kdesc(sm + O_WN),
                     kl0 = kdesc(sm + O_KKL), dh0 = mdesc(sm + O_DAQ, 8192);
#pragma unroll
      for (int kk = 0; kk < 4; ++kk) {
        umma_if(lead, X4, step(a0, kk * 2048), step(da, kk * 32), ih10, kk > 0);
        const uint64_t kh = step(kh0, kk * 32), kl = step(kl0, kk * 32);
        const uint64_t dh = step(dh0, kk * 2048), dl = step(dh0, 8192 + kk * 2048);
        umma_if(lead, X3, kh, dh, id01, 1);
        umma_if(lead, X3, kl, dh, id01, 1);
        umma_if(lead, X3, kh, dl, id01, 1);
      }
      commit_if(lead, bar_mma);
    } else if (warp_u == 4) {
      tc_fence_after();
      const uint32_t lead = elect_one();
      const uint32_t id01 = idesc_bf16(128, 64, 0, 1), id00 = idesc_bf16(128, 64, 0, 0);
      const uint64_t qh0 = kdesc(sin + 16384), ql0 = kdesc(rdo), eh0 = kdesc(sm + O_DAQ), w0 = kdesc(sm + O_RV),
                     ab = mdesc(sm + O_AB, 8192);
#pragma unroll
      for (int kk = 0; kk < 4; ++kk) {
        const uint64_t qh = step(qh0, kk * 32), ql = step(ql0, kk * 32);
        const uint64_t eh = step(eh0, kk * 32), el = step(eh0, 8192 + kk * 32);
        umma_if(lead, X0, qh, eh, id00, 1);
        umma_if(lead, X0, ql, eh, id00, 1);
        umma_if(lead, X0, qh, el, id00, 1);
        umma_if(lead, X2, step(w0, kk * 32), step(ab, kk * 2048), id01, kk > 0);
      }
      commit_if(lead, bar_mma);
    } else if (tid == 224) {
      tma_store_4d(&m2, sm + O_RH, 0, h, c * CM, b);  // (m2: dv itself)
      tma_store_4d(&m2, sm + O_RH + 8192, 64, h, c * CM, b);
      bulk_commit();
    }
    mm_ok = mma_poll();
    tc_fence_after();
    if (wq < 2) {  // X = A^T dA -> fp16 [r][s]
      const int j = 32 * wq + lane, tc0 = 16 * wg;
      float v[16];
      tmem_ld16(X4 + lane_base + tc0, v);
      sm16(sm + O_XT, chunk_off(j, tc0 >> 3)) = pack_h8(v);
      sm16(sm + O_XT, chunk_off(j, (tc0 >> 3) + 1)) = pack_h8(v + 8);
    }
    fence_proxy_async();
    tc_fence_before();
    if (!__syncthreads_and(mm_ok)) {
      ok = false;
      break;
    }
    // ---- round 3.  X1 = X A^T, dT = strict_lower(-A^T dA A^T)
    if (warp_u == 0) {
      tc_fence_after();
      const uint32_t lead = elect_one();
      const uint32_t ih00 = idesc_f16(128, 64, 0, 0);
      for (int kk = 0; kk < 4; ++kk)
        umma_if(lead, X1, kdesc(sm + O_XT + kk * 32), kdesc(sm + O_AH + kk * 32), ih00, kk > 0);
      commit_if(lead, bar_mma);
    } else if (warp_u == 4) {
      commit_if(elect_one(), bar_mma);
    } else if (G && lane == 0 && warp >= 14) {
      // the omega logits for the last pass, over A bf16 and dA^T (read by round 2)
      mbar_expect_tx(bar_w, 8192);
      tma_load_4d(sm + (warp == 14 ? O_AB : O_AQ), &mw, bar_w, warp == 14 ? 0 : 64, h, c * CM, b);
    }
    mm_ok = mma_poll();
    tc_fence_after();
    if (wq < 2) {
      const int r = 32 * wq + lane, tc0 = 16 * wg;
      float v[16];
      tmem_ld16(X1 + lane_base + tc0, v);
#pragma unroll
      for (int u = 0; u < 16; ++u) v[u] = (tc0 + u < r) ? -v[u] : 0.f;
      sm16(sm + O_DT, chunk_off(r, tc0 >> 3)) = pack_bf8(v);
      sm16(sm + O_DT, chunk_off(r, (tc0 >> 3) + 1)) = pack_bf8(v + 8);
    }
    fence_proxy_async();
    tc_fence_before();
    if (!__syncthreads_and(mm_ok)) {
      ok = false;
      break;
    }
    // ---- round 4.  X0 += (dT^T Kbar)^T, X2 += (dT Kk)^T
    if (warp_u == 0) {
      tc_fence_after();
      const uint32_t lead = elect_one();
      const uint32_t id01 = idesc_bf16(128, 64, 0, 1);
      for (int kk = 0; kk < 4; ++kk)
        umma_if(lead, X0, kdesc(sin + kk * 32), mdesc(sm + O_DT + kk * 2048, 8192), id01, 1);
      commit_if(lead, bar_mma);
    } else if (warp_u == 4) {
      tc_fence_after();
      const uint32_t lead = elect_one();
      const uint32_t id00 = idesc_bf16(128, 64, 0, 0);
      for (int kk = 0; kk < 4; ++kk)
        umma_if(lead, X2, kdesc(sm + O_WN + kk * 32), kdesc(sm + O_DT + kk * 32), id00, 1);
      commit_if(lead, bar_mma);
    }
    const float kprev = qq > 0 ? raw_k(t0 - 1) : 0.f;
    mm_ok = mma_poll();
    tc_fence_after();
    fence_proxy_async();
    if (!__syncthreads_and(mm_ok)) {
      ok = false;
      break;
    }
    // every tile but k, q has been read: the next chunk's may land
    if (on.j < njobs) issue_a(on);
    if (on.j < njobs) load_small(on);
    cp_commit();
    // ---- per channel (lane ci, tokens t0..t0+15): back through Gamma and the gain emission,
    //      then the uncertainty recursion backwards in time.  Free TMEM columns hold the
    //      per-(channel, token) intermediates between passes (X2 <- dphat (gain part), X1 <- dk
    //      (memory + gain part), X0 <- alpha, X3 <- 1 / (1 + u phat), X4 <- dG) and, in X5, the
    //      quarters' sums and maps that the four threads of a channel exchange; phat and
    //      gamma are read again from TMEM, eight tokens at a time: few live registers
    {
      const uint32_t XE = X5 + lane_base;  // columns qq: sum of dG; 4 + qq: dgamma_C part;
                                           // 8 + 2 qq ..: A, B of the quarter
      const size_t ostride = (size_t)a.H * D;
      const size_t obase = tok_index(a, b, c * CM + t0, h) * D + ci;
      const int nval = min(16, a.T - (c * CM + t0));
      auto out = [&](void *p, int j, float x) { st_grad<1>(p, obase + (size_t)j * ostride, x); };
      float k16[16];
      // pass A: dq, dG, the ds_t partial sums and the ds-free parts of dphat and dk
      {
        float part[16], tot = 0.f;
#pragma unroll
        for (int h8 = 0; h8 < 2; ++h8) {
          float xq[8], xk[8], xb[8], p8[8], g8[8], c1[8], c2[8], dg[8];
          tmem_ld8(TPH + lane_base + t0 + 8 * h8, p8);
          tmem_ld8(TGM + lane_base + t0 + 8 * h8, g8);
          tmem_ld8(X3 + lane_base + t0 + 8 * h8, xq);
          tmem_ld8(X0 + lane_base + t0 + 8 * h8, xk);
          tmem_ld8(X2 + lane_base + t0 + 8 * h8, xb);
#pragma unroll
          for (int u = 0; u < 8; ++u) {
            const int j = 8 * h8 + u, t = t0 + j;
            const float kk = raw_k(t), qv = raw_q(t), si = s_si[t], g_ = g8[u], ig = __fdividef(1.f, g_);
            const float kap = p8[u] * kk * si;  // kappa_t (eq. kla-box-gain)
            dg[u] = xb[u] * g_ * kk - xk[u] * kap * ig + xq[u] * tau * g_ * qv;
            tot += dg[u];
            const float dkap = xk[u] * ig;
            k16[j] = kk;
            part[j] = dkap * kap;
            c1[u] = dkap * kk * si;
            c2[u] = xb[u] * g_ + dkap * p8[u] * si;
            if (j < nval) out(a.dq, j, tau * g_ * xq[u] * invl);
          }
          tmem_st8(X2 + lane_base + t0 + 8 * h8, c1);
          tmem_st8(X1 + lane_base + t0 + 8 * h8, c2);
          tmem_st8(X4 + lane_base + t0 + 8 * h8, dg);
        }
        tmem_st1(XE + qq, tot);
        tmem_st1(XE + 4 + qq, dgc);
        const float rsum = rs16(part, lane);
        if ((lane & 1) == 0) s_red[wq * 64 + t0 + (lane >> 1)] = rsum;
      }
      tmem_st_wait();
      fence_proxy_async();
      __syncthreads();
      if (on.j < njobs) issue_kq(on);  // raw k, q have been read
      if (tid < CM) s_ds[tid] = -((s_red[tid] + s_red[64 + tid]) + (s_red[128 + tid] + s_red[192 + tid])) * s_si[tid];
      __syncthreads();
      // entry values of this quarter: gamma_{t0-1}, p_{t0-1}
      float ga_prev = 1.f, p_prev = s_pin[ci];
      if (qq > 0) {
        const float pp = tmem_ld1(TPH + lane_base + t0 - 1);
        ga_prev = tmem_ld1(TGM + lane_base + t0 - 1);  // gamma_{t0-1}
        p_prev = __fdividef(pp, 1.f + mu * kprev * kprev * s_ri[t0 - 1] * pp);
      }
      // pass B: per-token coefficients of dp_{t-1} = a_t dp_t + b_t and the quarter's
      //         composition dp_before = A dp_after + B
      {
        float A = 1.f, Bv = 0.f;
#pragma unroll
        for (int h8 = 1; h8 >= 0; --h8) {
          float c1[8], p8[8], g8[8], a2v[8], rdv[8], gp = ga_prev;
          tmem_ld8(TPH + lane_base + t0 + 8 * h8, p8);
          tmem_ld8(TGM + lane_base + t0 + 8 * h8, g8);
          if (h8) gp = tmem_ld1(TGM + lane_base + t0 + 7);
          tmem_ld8(X2 + lane_base + t0 + 8 * h8, c1);
#pragma unroll
          for (int u = 7; u >= 0; --u) {
            const int j = 8 * h8 + u, t = t0 + j;
            const float kk = k16[j];
            const float al = __fdividef(g8[u], u > 0 ? g8[u - 1] : gp), al2 = al * al;
            const float rd = __fdividef(1.f, 1.f + mu * kk * kk * s_ri[t] * p8[u]);
            const float dphl = c1[u] + s_ds[t] * kk * kk;
            const float aj = al2 * rd * rd;
            Bv = aj * Bv + al2 * dphl;
            A = aj * A;
            a2v[u] = al;  // alpha (the last pass squares it again)
            rdv[u] = rd;
            c1[u] = dphl;
          }
          tmem_st8(X0 + lane_base + t0 + 8 * h8, a2v);
          tmem_st8(X3 + lane_base + t0 + 8 * h8, rdv);
          tmem_st8(X2 + lane_base + t0 + 8 * h8, c1);
        }
        tmem_st1(XE + 8 + 2 * qq, A);
        tmem_st1(XE + 9 + 2 * qq, Bv);
      }
      // dp leaving this chunk, if the next chunk's job has handed it on already
      uint64_t early = 0;
      if (tid < D && c < NC - 1) early = slot_peek(small_slot(P.s, a, b, h, c, tid));
      tmem_st_wait();
      tc_fence_before();
      cp_wait<0>();
      mm_ok = true;
      if (G) mm_ok = mbar_wait(bar_w, it & 1, kWaitIters);  // the omega-logit tile has landed
      __syncthreads();
      tc_fence_after();
      float ex[8];  // the quarters' maps of this channel
      tmem_ld8(XE + 8, ex);
      // dp leaving the chunk: from the next chunk's job (thread i: channel i)
      if (tid < D) {
        float dp = 0.f, al0[16], rd0[16], dl0[16];
#pragma unroll
        for (int h8 = 0; h8 < 2; ++h8) {
          tmem_ld8(X0 + lane_base + 8 * h8, al0 + 8 * h8);
          tmem_ld8(X3 + lane_base + 8 * h8, rd0 + 8 * h8);
          tmem_ld8(X2 + lane_base + 8 * h8, dl0 + 8 * h8);
        }
        if (c == NC - 1) {
          if (a.dpT) dp = lam * a.dpT[((size_t)b * a.H + h) * D + tid];
        } else {
          mm_ok = slot_get(small_slot(P.s, a, b, h, c, tid), early, &dp) && mm_ok;
        }
        s_dp[tid] = dp;
        // hand on the dp entering this chunk: pass C's recursion through the first quarter, ahead of the pass
        if (c > 0) {
#pragma unroll
          for (int q2 = 3; q2 > 0; --q2) dp = fmaf(ex[2 * q2], dp, ex[2 * q2 + 1]);
#pragma unroll
          for (int u = 15; u >= 0; --u) {
            const float dph = dp * rd0[u] * rd0[u] + dl0[u];
            dp = al0[u] * al0[u] * dph;
          }
          slot_put(small_slot(P.s, a, b, h, c - 1, tid), dp);
        }
      }
      if (!__syncthreads_and(mm_ok)) {
        ok = false;
        break;
      }
      // pass C: the recursion backwards through this quarter's tokens
      {
        float dp = s_dp[ci];
#pragma unroll
        for (int q2 = 3; q2 > 0; --q2)
          if (q2 > qq) dp = fmaf(ex[2 * q2], dp, ex[2 * q2 + 1]);
        float es[8];  // the quarters' sums of dG, then of dgamma_C
        tmem_ld8(XE, es);
        // dG_63 gains dgamma_C gamma_C; it lies in every suffix
        float run = ((es[4] + es[5]) + (es[6] + es[7])) * s_gC[ci];
#pragma unroll
        for (int q2 = 1; q2 < 4; ++q2)
          if (q2 > qq) run += es[q2];
        float drp[16];
#pragma unroll
        for (int h8 = 1; h8 >= 0; --h8) {
          float a2v[8], dphl[8], c2[8], p8[8], rd8[8], dg[8], pb = p_prev;
          tmem_ld8(TPH + lane_base + t0 + 8 * h8, p8);
          tmem_ld8(X3 + lane_base + t0 + 8 * h8, rd8);
          if (h8) pb = tmem_ld1(TPH + lane_base + t0 + 7) * tmem_ld1(X3 + lane_base + t0 + 7);
          tmem_ld8(X0 + lane_base + t0 + 8 * h8, a2v);
          tmem_ld8(X2 + lane_base + t0 + 8 * h8, dphl);
          tmem_ld8(X1 + lane_base + t0 + 8 * h8, c2);
          tmem_ld8(X4 + lane_base + t0 + 8 * h8, dg);
#pragma unroll
          for (int u = 7; u >= 0; --u) {
            const int j = 8 * h8 + u, t = t0 + j;
            const float kk = k16[j], ds = s_ds[t], ri = s_ri[t];
            const float pt = p8[u] * rd8[u];
            const float pprev = u > 0 ? p8[u - 1] * rd8[u - 1] : pb;
            const float dph = dp * rd8[u] * rd8[u] + dphl[u];
            const float du = -dp * pt * pt;
            const float dkt = c2[u] + 2.f * ds * p8[u] * kk + du * 2.f * mu * kk * ri;
            drp[j] = -du * mu * kk * kk * ri * ri;
            run += dg[u];
            const float al2 = a2v[u] * a2v[u];
            const float dgt = run + 2.f * al2 * pprev * dph;
            if (j < nval) {
              // logit gates: d omega / dy = sigmoid(y), d log alpha / dx = 1 - alpha
              const float fw = G ? sigmoid_f(bf(sm + (ci < 64 ? O_AB : O_AQ), 0, t, ci & 63)) : 1.f;
              const float fg = G ? 1.f - a2v[u] : 1.f;
              out(a.dk_, j, dkt * invl);
              out(a.domega, j, dph * fw * invl);
              out(a.dg, j, dgt * fg * invl);
            }
            dp = al2 * dph;
          }
        }
        const float rs2 = rs16(drp, lane);
        if ((lane & 1) == 0) s_red2[wq * 64 + t0 + (lane >> 1)] = rs2;
      }
      if (G) fence_proxy_async();
      tc_fence_before();
      __syncthreads();
      tc_fence_after();
      if (G && on.j < njobs) issue_g2(on);  // the omega logits have been read
      if (tid < CM) {
        const int tt = c * CM + tid;
        if (tt < a.T) {
          // the part of dr_t through u = mu k^2 / r: -sum_i du mu k^2 / r^2
          const float dru = (s_red2[tid] + s_red2[64 + tid]) + (s_red2[128 + tid] + s_red2[192 + tid]);
          st_grad<1>(a.dr, tok_index(a, b, tt, h), (s_ds[tid] + dru) * (G ? s_fr[tid] : 1.f) * invl);
        }
      }
    }
  }
  if (!ok) {
    if (tid == 0) {
      atomicExch(a.status, (unsigned)KDN_ERR_TIMEOUT);
      // copies and MMAs in flight land before the CTA's memory goes away
      for (int k = 0; k < 6; ++k) {
        mbar_wait(bars + k, 0, 1u << 14);
        mbar_wait(bars + k, 1, 1u << 14);
      }
    }
  }
  if (tid == 224) bulk_wait_all();  // the last chunk's dv stores
  tc_fence_before();
  __syncthreads();
  if (warp == 0) tmem_dealloc(tb, 512);
}

}  // namespace

// Where the two kernels (with k_bwd_tiles) finish sooner than the one-kernel sweep, in tenths of a
// microsecond as measured.  The sweep: 208 a chunk of each wave of sequences.  Here: k_bwd_tiles 0.19 a
// job, k_bwd_state 31 a chunk of a sequence or 0.3 a job (HBM), k_bwd_chunk 162 a round of 152
// jobs, but with few sequences 17 a chunk (the chain of dp), and 280 until its rounds run evenly.
// Two kernels against the sweep, us: B8 H16 T4096 1295 and 1317; B2 H16 T1984 280 and 600, B1 H16 T4096 382 and
// 1213, B64 H1 T512 139 and 171, B40 H5 T512 322 and 353; on the other side B8 H16 T1024 380 and 347, B19 H8 T2048
// 793 and 684, B100 H1 T512 186 and 177, B16 H16 T2048 1345 and 1308.  Fewer than 96 chunks in all are left to the
// sweep (a few tens of us either way).
bool split_bwd_sizes(const Args &a) {
  if (a.variant != 0 || a.chunk == 32 || !fused_fwd_supported(a)) return false;
  const long long bh = (long long)a.B * a.H, nc = (a.T + CM - 1) / CM, jobs = bh * nc;
  if (jobs < 96) return false;
  const long long waves = (bh + kSms - 1) / kSms, rounds = (jobs + kSms - 1) / kSms;
  const long long state = waves * std::max(31 * nc, 3 * std::min<long long>(bh, kSms) * nc / 10);
  const long long chunk = std::max(162 * rounds, 17 * nc + 160) + (rounds > 1 ? 280 : 0);
  return 140 + jobs * 19 / 100 + state + chunk < waves * (208 * nc + 60);
}

// The gradient buffers serve as scratch only where they overlap neither each other nor anything the
// backward reads: the sweep reads each chunk's rows before it writes them, so that a gradient may
// take the place of its input there.
static bool scratch_is_apart(const Args &a) {
  struct Range { uintptr_t p; size_t n; };
  const size_t th = (size_t)a.B * a.T * a.H, bh = (size_t)a.B * a.H, act = th * D * 2;
  auto at = [](const void *p, size_t n) { return Range{reinterpret_cast<uintptr_t>(p), p ? n : 0}; };
  const Range r[] = {at(a.dq, act), at(a.dk_, act), at(a.dv_, act), at(a.dg, act), at(a.domega, act),  // scratch
                     at(a.dr, th * 2), at(a.q, act), at(a.k, act), at(a.v, act), at(a.g, act), at(a.omega, act),
                     at(a.r, th * 2), at(a.dO, act), at(a.dST, bh * D * D * 4), at(a.dpT, bh * D * 4),
                     at(a.fSin, fused_saved_bytes(a)), at(a.status, 256)};
  for (int i = 0; i < 5; ++i)
    for (size_t j = i + 1; j < sizeof r / sizeof *r; ++j)
      if (r[i].p < r[j].p + r[j].n && r[j].p < r[i].p + r[i].n) return false;
  return true;
}

// The calls served: bf16 gradients and none of the initial state or mu, which the two kernels
// do not form.
bool split_bwd_supported(const Args &a) {
  return split_bwd_sizes(a) && a.odt == KDN_BF16 && !a.dS0 && !a.dp0 && !a.dmu && (a.T % CM == 0 || a.split_ws) &&
         scratch_is_apart(a);
}

size_t split_bwd_workspace_bytes(const Args &a) {
  if (!split_bwd_sizes(a) || a.odt != KDN_BF16 || a.T % CM == 0) return 0;
  return (size_t)a.B * a.H * 5 * 16384;
}

kdn_status_t launch_split_bwd(const Args &a, char *ws, cudaStream_t s) {
  SplitParams P;
  P.a = a;
  P.ticket = a.status + 1;
  const int NC = (a.T + CM - 1) / CM;
  P.s.small = static_cast<unsigned char *>(a.domega);
  P.s.tail = a.T % CM ? reinterpret_cast<unsigned char *>(ws) : nullptr;
  P.s.last = NC - 1;
  const void *buf[4] = {a.dq, a.dk_, a.dv_, a.dg};
  CUtensorMap m[4], mq, mk, mdo;
  for (int k = 0; k < 4; ++k)
    if (!make_map(&m[k], buf[k], a)) return KDN_ERR_CUDA;
  CUtensorMap mt = m[0];
  if (P.s.tail) {  // [5 B, 64, H, 128]
    Args t = a;
    t.B = 5 * a.B;
    t.T = CM;
    if (!make_map(&mt, P.s.tail, t)) return KDN_ERR_CUDA;
  }
  if (!make_map(&mq, a.q, a) || !make_map(&mk, a.k, a) || !make_map(&mdo, a.dO, a)) return KDN_ERR_CUDA;
  CUtensorMap mw = mq;  // the omega logits
  if (a.gates && !make_map(&mw, a.omega, a)) return KDN_ERR_CUDA;
  const long long njobs = (long long)a.B * a.H * NC;
  k_bwd_tiles<<<(unsigned)(2 * njobs), TT, TILE_SMEM, s>>>(m[2], m[3], mt, P);
  if (cudaGetLastError() != cudaSuccess) return KDN_ERR_CUDA;
  if (cudaFuncSetAttribute(k_bwd_state, cudaFuncAttributeMaxDynamicSharedMemorySize, STATE_SMEM) != cudaSuccess)
    return KDN_ERR_CUDA;
  k_bwd_state<<<a.B * a.H, BT, STATE_SMEM, s>>>(mdo, m[0], m[1], m[2], m[3], mt, P);
  if (cudaGetLastError() != cudaSuccess) return KDN_ERR_CUDA;
  const auto kern = a.gates ? k_bwd_chunk<1> : k_bwd_chunk<0>;
  if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, CHUNK_SMEM) != cudaSuccess)
    return KDN_ERR_CUDA;
  kern<<<(unsigned)(njobs < kSms ? njobs : kSms), BT, CHUNK_SMEM, s>>>(mq, mk, mdo, mw, m[0], m[1], m[2], m[3],
                                                                       mt, P);
  return cudaGetLastError() == cudaSuccess ? KDN_OK : KDN_ERR_CUDA;
}

}  // namespace kdn
