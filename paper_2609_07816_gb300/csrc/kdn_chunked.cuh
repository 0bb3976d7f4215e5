// kdn_chunked.cuh -- shared by the general chunked forward (kdn_chunked_fwd.cu) and
// backward (kdn_chunked_bwd.cu): register-tiled float32 products and the
// double-buffered factors of the inter-chunk passes.
#pragma once

#include "kdn_internal.cuh"

namespace kdn {
namespace {

constexpr int CC = 32;      // chunk length of these kernels
constexpr int LC = CC + 4;  // row stride (floats) of 32-column tiles: 16-byte rows, and rows
                            // r .. r + 7 start in different groups of four banks

#define KDN_TID (int)threadIdx.x

// Four consecutive elements (i a multiple of 4) as floats.
template <typename DT> __device__ __forceinline__ void ld4(const void *p, size_t i, float *v);
template <> __device__ __forceinline__ void ld4<float>(const void *p, size_t i, float *v) {
  const float4 x = *reinterpret_cast<const float4 *>(static_cast<const float *>(p) + i);
  v[0] = x.x; v[1] = x.y; v[2] = x.z; v[3] = x.w;
}
template <> __device__ __forceinline__ void ld4<__nv_bfloat16>(const void *p, size_t i, float *v) {
  const uint2 u = *reinterpret_cast<const uint2 *>(static_cast<const __nv_bfloat16 *>(p) + i);
  v[0] = __uint_as_float(u.x << 16);
  v[1] = __uint_as_float(u.x & 0xffff0000u);
  v[2] = __uint_as_float(u.y << 16);
  v[3] = __uint_as_float(u.y & 0xffff0000u);
}
__device__ __forceinline__ float4 f4(const float *v) { return make_float4(v[0], v[1], v[2], v[3]); }
__device__ __forceinline__ void st4(float *p, const float *v) { *reinterpret_cast<float4 *>(p) = f4(v); }
// four adjacent outputs in the caller's output dtype
__device__ __forceinline__ void sto4(int odt, void *p, size_t i, const float *v) {
  if (odt == KDN_BF16) {
    const __nv_bfloat162 a = __floats2bfloat162_rn(v[0], v[1]), b = __floats2bfloat162_rn(v[2], v[3]);
    uint2 u;
    u.x = *reinterpret_cast<const uint32_t *>(&a);
    u.y = *reinterpret_cast<const uint32_t *>(&b);
    *reinterpret_cast<uint2 *>(static_cast<__nv_bfloat16 *>(p) + i) = u;
  } else {
    st4(static_cast<float *>(p) + i, v);
  }
}

// acc[m][n] += sum_k A[row m][k] B[k][n].  The thread's rows of A start at A and lie
// `sa` floats apart, k contiguous.  BK: its four columns are rows of a tile with k
// contiguous (ldb apart); else four adjacent columns of a [k][n] tile.
template <int K, int TM, bool BK, typename TB = float>
__device__ __forceinline__ void tile_mm(float (*acc)[4], const float *A, int sa, const TB *B, int ldb) {
#pragma unroll(TM > 2 ? 2 : 4)
  for (int k = 0; k < K; k += 4) {
    float a[TM][4], b[4][4];
#pragma unroll
    for (int m = 0; m < TM; ++m) ld4<float>(A + m * sa, k, a[m]);
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      float x[4];
      ld4<TB>(BK ? B + q * ldb + k : B + (k + q) * ldb, 0, x);
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        if (BK) b[u][q] = x[u];
        else b[q][u] = x[u];
      }
    }
#pragma unroll
    for (int kk = 0; kk < 4; ++kk)
#pragma unroll
      for (int m = 0; m < TM; ++m)
#pragma unroll
        for (int n = 0; n < 4; ++n) acc[m][n] = fmaf(a[m][kk], b[kk][n], acc[m][n]);
  }
}
// acc[m][n] += sum_k A[k][m] B[k][n]: both tiles [k][.], RM adjacent rows m.
template <int K, int RM>
__device__ __forceinline__ void tile_mm_t(float (*acc)[4], const float *A, int lda, const float *B, int ldb) {
#pragma unroll 4
  for (int k = 0; k < K; ++k) {
    float a[RM], b[4];
    if constexpr (RM >= 4) {
#pragma unroll
      for (int m = 0; m < RM; m += 4) ld4<float>(A + k * lda + m, 0, a + m);
    } else if constexpr (RM == 2) {
      const float2 x = *reinterpret_cast<const float2 *>(A + k * lda);
      a[0] = x.x;
      a[1] = x.y;
    } else {
      a[0] = A[k * lda];
    }
    ld4<float>(B + k * ldb, 0, b);
#pragma unroll
    for (int m = 0; m < RM; ++m)
#pragma unroll
      for (int n = 0; n < 4; ++n) acc[m][n] = fmaf(a[m], b[n], acc[m][n]);
  }
}
// The same in two halves of k, each summed by itself (their partial sums round less): the inter-chunk
// passes, whose sums go on through every chunk.
template <int K, int TM>
__device__ __forceinline__ void tile_mm2(float (*acc)[4], const float *A, int sa, const float *B, int ldb) {
  float t[TM][4] = {};
  tile_mm<K / 2, TM, false>(acc, A, sa, B, ldb);
  tile_mm<K / 2, TM, false>(t, A + K / 2, sa, B + K / 2 * ldb, ldb);
#pragma unroll
  for (int m = 0; m < TM; ++m)
#pragma unroll
    for (int n = 0; n < 4; ++n) acc[m][n] += t[m][n];
}
template <int TM> __device__ __forceinline__ void zero(float (*acc)[4]) {
#pragma unroll
  for (int m = 0; m < TM; ++m)
#pragma unroll
    for (int n = 0; n < 4; ++n) acc[m][n] = 0.f;
}

// ---------------------------------------------------------------------------
// Inter-chunk state passes.  The per-chunk factors (W, Qbar, K_tail, A_qk,
// gamma_C and the chunk's U or dO slice) are double-buffered in shared memory
// with cp.async, so chunk c+1 streams in while chunk c is computed.

__device__ __forceinline__ uint32_t smem_addr(const void *p) {
  return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}
// 16-byte global -> shared copy; zero-filled when `valid` is false
__device__ __forceinline__ void cp16(void *dst, const void *src, bool valid = true) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(smem_addr(dst)), "l"(src),
               "r"(valid ? 16 : 0)
               : "memory");
}
__device__ __forceinline__ void cp_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_wait() {
  asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}

// CW value columns per CTA.  [W; Qbar] S_in is a 64 x CW product; TM of its rows and
// four columns a thread: 16 CW / TM threads.  The 32 rows of R and of O are split evenly over
// the threads (rows ga + GA m: the first half of a thread's rows are R's).
template <int DK, int CW, int TM>
struct StateCfg {
  static constexpr int LD = DK + 4, LS = CW + 4, GA = 64 / TM, NTH = GA * CW / 4;
  static constexpr int RS = DK / GA;  // rows of S a thread updates
  // floats per buffer: [W; Qbar], K_tail, A_qk, gamma_C, and a [C][CW] slice (U or raw dO)
  static constexpr int FLOATS = 3 * CC * LD + CC * LC + DK + CC * LS;
  static constexpr size_t SMEM = sizeof(float) * (2 * FLOATS + DK * LS + CC * LS);
};

// Issues the cp.async copies of chunk c's factors into buffer `buf`.
// `slice` is U (forward, fp32) or dO (backward, bytes of the activation dtype).
template <class Cfg, int DK, int CW>
__device__ __forceinline__ void issue_chunk_factors(const Args &a, int bh, int c, float *buf, int j0,
                                                    bool backward) {
  constexpr int NTH = Cfg::NTH, LD = Cfg::LD, LS = Cfg::LS;
  float *sW = buf, *sQ = sW + CC * LD, *sKt = sQ + CC * LD, *sAqk = sKt + CC * LD;
  float *sgC = sAqk + CC * LC, *sSl = sgC + DK;
  const size_t base = (size_t)bh * a.NC + c;
  constexpr int RC = DK / 4;  // 16-byte pieces per factor row
  for (int e = KDN_TID; e < CC * RC; e += NTH) {
    const int r = e / RC, q = e % RC;
    const size_t o = (base * CC + r) * DK + 4 * q;
    cp16(sW + r * LD + 4 * q, a.W + o);
    cp16(sQ + r * LD + 4 * q, a.Qb + o);
    cp16(sKt + r * LD + 4 * q, a.Kt + o);
  }
  for (int e = KDN_TID; e < CC * (CC / 4); e += NTH) {
    const int r = e / (CC / 4), q = e % (CC / 4);
    cp16(sAqk + r * LC + 4 * q, a.Aqk + base * CC * CC + r * CC + 4 * q);
  }
  for (int e = KDN_TID; e < DK / 4; e += NTH) cp16(sgC + 4 * e, a.gC + base * DK + 4 * e);
  if (!backward) {
    for (int e = KDN_TID; e < CC * (CW / 4); e += NTH) {
      const int r = e / (CW / 4), q = e % (CW / 4);
      cp16(sSl + r * LS + 4 * q, a.U + (base * CC + r) * a.dv + j0 + 4 * q);
    }
  } else {
    // raw dO rows of this slice: CW elements of the activation dtype
    const int es = a.dtype == KDN_BF16 ? 2 : 4;
    const int rc = CW * es / 16;
    const int b = bh / a.H, h = bh % a.H;
    for (int e = KDN_TID; e < CC * rc; e += NTH) {
      const int r = e / rc, q = e % rc, tt = c * CC + r;
      const bool valid = tt < a.T;
      const char *src = static_cast<const char *>(a.dO) +
                        ((valid ? tok_index(a, b, tt, h) : 0) * a.dv + j0) * es + 16 * q;
      cp16(reinterpret_cast<char *>(sSl + r * LS) + 16 * q, src, valid);
    }
  }
}

template <typename K>
cudaError_t set_smem(K kernel, size_t bytes) {
  return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
}
template <typename K>
bool launch(K kernel, size_t grid, int threads, size_t smem, cudaStream_t s, const Args &a) {
  if (smem > 48 * 1024 && set_smem(kernel, smem) != cudaSuccess) return false;
  kernel<<<(unsigned)grid, threads, smem, s>>>(a);
  return cudaGetLastError() == cudaSuccess;
}

// Value columns per CTA of the state passes: the widest slice that still gives the
// GPU about one CTA per SM (a narrower slice re-reads the chunk's factors for fewer
// columns, but the pass is a chain over chunks and idle SMs cost more).  With 240 CTAs asked
// for instead of 120 the whole forward takes 638 us, not 616, at B8 H16 T2048 d = 64 bf16 (32
// columns a CTA, not 64) and 648, not 482, at B2 H16 T2048 d = 128 fp32 (16, not 32).
constexpr size_t kStateCtas = 120;
int state_cols(const Args &a) {
  const size_t BH = (size_t)a.B * a.H;
  for (int cw = a.dv < 64 ? a.dv : 64; cw > 16; cw /= 2)
    if (BH * (a.dv / cw) >= kStateCtas) return cw;
  return 16;
}
}  // namespace
}  // namespace kdn
