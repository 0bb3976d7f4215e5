// kdn_fused_bwd.cu -- fused chunked backward of the Diagonal and Isotropic KDN
// for bfloat16 activations with d_k = d_v = 128 and 64-token chunks (App. F),
// on the tcgen05 tensor cores of sm_103a.
//
// The Diagonal KDN with bf16 gradients and no state gradients runs kdn_split_bwd.cu from the
// same context instead, where the sizes gain from it.
//
// Two launches:
//  1. a fused forward in its context-saving mode (the training forward, or the
//     first pass of kdn_*_bwd) stores, per chunk, the 16-bit tiles it formed
//     and multiplied with -- S_in, R, -W, A_qk, A and, for the Diagonal KDN,
//     Y = V - Kbar S_in -- with phat and gamma in fp32, the per-token gain
//     scalars and the uncertainty p entering the chunk;
//  2. k_fused_bwd: one CTA per (batch, head) walks the chunks backwards.  The
//     memory cotangent dS (128 x 128 fp32) stays in tensor memory for the whole
//     sweep; the uncertainty cotangent dp (one value per channel) is carried in
//     shared memory.
// Per chunk (notation of App. F.2: Kbar = Gamma.K, Kk = Kbar^kappa, Qbar = tau
// Gamma.Q, A = (I + T)^-1, W = A Kbar, U = A V, R = U - W S_in, K_tail =
// gamma_C.Kk) the kernel recomputes the forward factors and forms the adjoint of
// O = Qbar S_in + A_qk R,  S_out = diag(gamma_C) S_in + K_tail^T R:
//   dR     = A_qk^T dO + K_tail dS                      (B1)
//   dS_in  = diag(gamma_C) dS + Qbar^T dO - W^T dR      (B2)
//   dA_qk  = lower(dO R^T),  dK_tail = R dS^T           (B3, B4)
//   dW     = -dR S_in^T,     dV = A^T dR                (B5, B7)
//   dQbar  = dO S_in^T + dA_qk Kk                       (B8)
//   dA     = dR V^T + dW Kbar^T,  dT = strict_lower(-A^T dA A^T)   (B6, X, Y)
//            (the Diagonal KDN forms dA = dR Y^T, the same matrix since
//            dW = -dR S_in^T and Y = V - Kbar S_in)
//   dKk    = dA_qk^T Qbar + gamma_C.dK_tail + dT^T Kbar (B9)
//   dKbar  = A^T dW + dT Kk                             (B10)
//   dgamma_C = colsum(dK_tail.Kk) + rowsum(dS.S_in)
// and then, per channel on CUDA cores, the adjoint of the scaling by Gamma and
// of the gain emission (eq. chunk-gain-emission, eq. kla-box-gain /
// iso-kla-box-gain) and of the uncertainty recursion backwards over the chunk's
// tokens: per channel for the Diagonal KDN (eq. diag-covariance-prediction,
// eq. prefix-diag-uncertainty), one scalar per head for the Isotropic KDN
// (eq. iso-kla-box-cov-update, Prop. 5).
//
// Every product runs as a cta_group::1, M = 128 MMA.  Products whose natural
// row count is 64 read 64 further rows of whatever follows the operand in
// shared memory; those accumulator rows are never read.  The matrices with
// 128 rows (channels) are computed transposed, so that channel i is TMEM lane i
// and the per-channel recursions read their operands straight from TMEM.
//
// Precision: the Gamma-scaled operands Kbar, Qbar, Kk and dA_qk (exp(+-G)
// factors) are split into hi + lo bf16 pairs where they meet one another;
// everything else is fp16 (10-bit mantissa).  The cotangents are scaled by a
// power of two lambda (from max|dO| and max|dS_T| of the head) before they
// enter fp16, and every gradient is scaled back by 1/lambda, so the fp16 range
// holds for any magnitude of the incoming cotangents.
//
// Bound by the chain of a chunk's stages on one SM (~40 K cycles diagonal, ~33 K isotropic;
// ~45 % of the issue slots).  Copies are issued one per warp and the per-token inputs arrive by
// bulk copies: one thread's run of TMA operations and loads held at a barrier cost 2-3 K
// cycles a chunk (isotropic B8 H12 T2048: 561 -> 524 us; diagonal B8 H16 T4096: 1317 us).
//
// Every wait on an mbarrier is bounded; on timeout the kernel records
// KDN_ERR_TIMEOUT in the workspace status word and returns.
#include "kdn_internal.cuh"
#include "kdn_sm103.cuh"
#include "kdn_bwd_common.cuh"

namespace kdn {
namespace {

using namespace sm103;
using namespace fused;

constexpr int BT = 512;  // threads (16 warps)
constexpr int CM = 64;   // chunk length
constexpr int D = 128;   // head dim (dk = dv)
constexpr uint32_t kWaitIters = 1u << 25;
constexpr int KB = 1024;

// Shared-memory map (bytes from the 1024-aligned base).  Regions are reused
// across the stages of a chunk; the comments give the sequence of tenants.
constexpr int O_RKQ = 0;         // raw k | q, interleaved per 64-channel slab (whole chunk)
constexpr int O_SIN = 32 * KB;   // S_in fp16 [i][j] (context)  -> Kbar^T hi | Qbar^T hi (second set)
constexpr int O_RV = 64 * KB;    // raw v  -> v fp16 (isotropic); Y (context) -> dW^T bf16 (diagonal)
constexpr int O_RDO = 80 * KB;   // raw dO -> lambda dO fp16 -> Qbar^T lo
constexpr int O_AH = 96 * KB;    // A fp16 [t][s] (context)
constexpr int O_AB = 104 * KB;   // A bf16 [t][s] (from the saved fp16 A)
constexpr int O_DT = 112 * KB;   // dT bf16  -> per-channel scratch of the final stage
constexpr int O_AQ = 120 * KB;   // A_qk fp16 [t][s] (context)
constexpr int O_WN = 128 * KB;   // -W fp16 [t][i] (context)  -> Kk^T hi
constexpr int O_KT = 144 * KB;   // K_tail^T fp16  -> dR^T fp16
constexpr int O_G = 160 * KB;    // dS fp16  -> dA_qk^T | Qbar^T fp16  -> dW^T | Kk^T lo
                                 //   -> dA^T | X  -> dG of the final stage
constexpr int O_RH = 192 * KB;   // R fp16 (context; the next 8 KB are read as padding rows)
                                 //   -> lo part of dR^T fp16
constexpr int BUF_END = 216 * KB;
// derived tenants
constexpr int O_DRT = O_KT, O_KKH2 = O_WN;
constexpr int O_DSH = O_G, O_DAQ = O_G, O_QH = O_G + 16 * KB, O_KKL2 = O_G + 16 * KB;
constexpr int O_DWT = O_G, O_DAT = O_G + 16 * KB, O_XT = O_G + 24 * KB, O_KQH2 = O_SIN;
constexpr int O_QL2 = O_RDO, O_DRTL = O_RH;
// Diagonal KDN: Y (context) in the v buffer, then dW^T; dA^T over A_qk
constexpr int O_DWY = O_RV, O_DAY = O_AQ, O_DVS = O_RH;
// Diagonal KDN: the next chunk's phat and gamma (fp32 [64 t][128 i]) arrive by bulk copies
// into buffers idle from the end of a chunk's last pass to stage [3] of the next: phat over
// the dS tile, gamma's tokens 0..31 over the A bf16 and dT tiles, tokens 32..63 over K_tail
constexpr int O_PHB = O_G, O_GA0 = O_AB, O_GA1 = O_KT;
static_assert(O_AB + 8 * KB == O_DT, "gamma's first half spans the A bf16 and dT tiles");
// small arrays
constexpr int OFF_SM = BUF_END;
constexpr int SMALL_FLOATS = 64 * 18 + 256 * 2 + 128 * 2 + 16;
constexpr int OFF_BAR = OFF_SM + SMALL_FLOATS * 4;
constexpr int OFF_NX = OFF_BAR + 64;  // next chunk's per-token values: [5][64], then gamma [64] (SD)
constexpr int SMEM_BYTES = OFF_NX + 1536 + 1024;  // + alignment slack
static_assert(SMEM_BYTES <= 232448, "shared memory");
static_assert(O_AQ + 8 * KB <= O_WN && O_XT + 8 * KB <= O_RH, "map");

struct BwdParams {
  Args a;
};

// G: the gate inputs are logits (KDN_GATES_LOGITS), a compile-time choice so
// that the post-activation path carries none of the chain-rule code.
// SD: isotropic KDN with one decay per head.  Gamma is then a per-token scalar
// and the products that meet Gamma-scaled operands take it, with beta and tau,
// as fp32 factors on their 64 x 64 partner instead:
//   B8b  (dA_qk Kk)^T   = K^T (dA_qk diag(beta / gamma))^T
//   B9a  (dA_qk^T Qbar)^T = Q^T (diag(tau gamma) dA_qk)
//   B9b  (dT^T Kbar)^T  = K^T (diag(gamma) dT)
//   B10b (dT Kk)^T      = K^T (dT diag(beta / gamma))^T
// with K, Q the raw bf16 tiles (exact operands); the Qbar and Kk tiles of the
// second operand set are not formed.
template <int V, int OBF, int G, int SD>
__global__ void __launch_bounds__(BT, 1)
    k_fused_bwd(const __grid_constant__ CUtensorMap mq, const __grid_constant__ CUtensorMap mk,
                const __grid_constant__ CUtensorMap mv, const __grid_constant__ CUtensorMap mdo,
                const __grid_constant__ CUtensorMap mw, const __grid_constant__ CUtensorMap mdv,
                const BwdParams P) {
  const Args &a = P.a;
  extern __shared__ unsigned char smraw[];
  unsigned char *sm =
      reinterpret_cast<unsigned char *>((reinterpret_cast<uintptr_t>(smraw) + 1023) & ~uintptr_t(1023));
  unsigned char *rkq = sm + O_RKQ, *sin = sm + O_SIN, *rv = sm + O_RV, *rdo = sm + O_RDO;
  float *s_r = reinterpret_cast<float *>(sm + OFF_SM);  // [64] r_t
  float *s_ri = s_r + 64;     // [64] 1 / r_t
  float *s_s = s_ri + 64;     // [64] s_t = r_t + sum_i phat k^2
  float *s_red = s_s + 64;    // [4][64] per-warp partial sums over channels (ds_t)
  float *s_red2 = s_red + 256;  // [4][64] (dr_t)
  float *s_gC = s_red2 + 256;   // [128] gamma_C
  float *s_dp = s_gC + 128;     // [128] uncertainty cotangent carried between chunks
  float *s_si = s_dp + 128;     // [64] 1 / s_t
  float *s_ds = s_si + 64;      // [64] ds_t (cotangent of s_t)
  float *s_fw = s_ds + 64;      // [64] d omega_t / d y_t (iso; 1 unless the gates are logits)
  float *s_gs = s_fw + 64;      // [64] scalar log-decay g_t (iso, one decay per head)
  float *s_n2 = s_gs + 64;      // [64] |k_t|^2 (iso)
  float *s_a = s_n2 + 64;       // [64] a_t = mean alpha^2 (iso)
  float *s_bh = s_a + 64;       // [64] bhat_t (iso)
  float *s_bp = s_bh + 64;      // [64] b_{t-1} (iso)
  float *s_x = s_bp + 64;       // [64] beta_t (iso)
  float *s_dn2 = s_x + 64;      // [64] cotangent of |k_t|^2 (iso)
  float *s_da = s_dn2 + 64;     // [64] cotangent of a_t (iso)
  float *s_misc = s_da + 64;    // [0] lambda, [1..] scratch
  float *s_fr = s_misc + 16;    // [64] d r_t / d z_t (1 unless the gates are logits)
  float *s_dmu = s_fr + 64;     // [64] parts of dL/dmu (lambda-scaled), summed at the end:
                                //      diag one per token slot, iso in [0]
  float *s_gm = s_dmu + 64;     // [64] gamma_t (SD)
  float *s_kf = s_gm + 64;      // [64] beta_t / gamma_t (SD)
  uint64_t *bars = reinterpret_cast<uint64_t *>(sm + OFF_BAR);
  uint64_t *bar_a = bars, *bar_b = bars + 1, *bar_mma = bars + 2;
  // diagonal KDN with logit gates: the chunk's omega logits (tile in O_KT, pass C)
  uint64_t *bar_w = bars + 3;
  constexpr bool WT = V == 0 && G;
  // bf16 gradients: dv leaves by TMA stores of a shared-memory tile
  constexpr bool DVT = OBF;
  uint32_t *s_tbase = reinterpret_cast<uint32_t *>(bars + 4);
  uint64_t *bar_g = bars + 5;  // diagonal KDN: phat and gamma of the chunk

  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int warp_u = __shfl_sync(0xffffffffu, warp, 0);  // warp-uniform: the MMA issue stays uniform
  const int wq = warp & 3, wg = warp >> 2;  // TMEM lane quarter, column group
  const int ci = tid & (D - 1), qq = tid >> 7, t0 = 16 * qq;  // channel view: channel, token quarter
  const int bh = blockIdx.x, b = bh / a.H, h = bh % a.H;
  const int NC = (a.T + CM - 1) / CM;
  const float tau = a.tau, mu = a.mu;
  const bool pcd = (V == 0) || a.pcd;

  if (tid == 0) {  // arrivals: one per issuing thread
    mbar_init(bar_a, V == 0 ? 11 : SD ? 11 : 10);
    mbar_init(bar_b, V == 0 ? 2 : 4);
    mbar_init(bar_mma, 1);
    if (WT) mbar_init(bar_w, 2);
    if (V == 0) mbar_init(bar_g, 3);
    fence_mbar_init();
    prefetch_tmap(&mq);
    prefetch_tmap(&mk);
    prefetch_tmap(&mv);
    prefetch_tmap(&mdo);
    if (WT) prefetch_tmap(&mw);
    if (DVT) prefetch_tmap(&mdv);
  }
  if (warp == 0) {
    tmem_alloc(s_tbase, 512);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tb = *s_tbase;
  const uint32_t TS = tb, TPH = tb + 128, TGM = tb + 192;
  const uint32_t X0 = tb + 256, X1 = tb + 320, X2 = tb + 384, X3 = tb + 448;
  const uint32_t lane_base = (uint32_t)(32 * wq) << 16;

  // loads of chunk c on bar_a: the context record (S_in, R, -W, A_qk, A, the per-token values;
  // issued as soon as their buffers free up) and the raw k, q tiles (issued once the
  // previous chunk is done); bar_b <- dO (isotropic: and v; diagonal KDN: the context's Y in
  // place of v).  The copies are spread over lane 0 of the warps, each arriving with its own
  // bytes: one thread issuing them all holds the whole CTA up.
  float *n_tok = reinterpret_cast<float *>(sm + OFF_NX), *n_gm = n_tok + 5 * CM;
  auto issue_a_ctx = [&](int c) {
    const unsigned char *rec = a.fSin + ((size_t)bh * NC + c) * kCtxBytes;
    switch (lane == 0 ? warp : -1) {
      case 0: mbar_expect_tx(bar_a, 32768); bulk_g2s(sin, rec + kCtxS, 32768, bar_a); break;
      case 1:
        if (DVT) bulk_wait_read();  // the dv tile has left the R buffer (this thread stored it)
        mbar_expect_tx(bar_a, 16384);
        bulk_g2s(sm + O_RH, rec + kCtxR, 16384, bar_a);
        break;
      case 2: mbar_expect_tx(bar_a, 16384); bulk_g2s(sm + O_WN, rec + kCtxW, 16384, bar_a); break;
      case 3: mbar_expect_tx(bar_a, 8192); bulk_g2s(sm + O_AQ, rec + kCtxAqk, 8192, bar_a); break;
      case 4: mbar_expect_tx(bar_a, 8192); bulk_g2s(sm + O_AH, rec + kCtxA, 8192, bar_a); break;
      case 5: mbar_expect_tx(bar_a, 1280); bulk_g2s(n_tok, rec + kCtxTok, 1280, bar_a); break;
      case 6:
        if (V == 0) {
          mbar_expect_tx(bar_a, 16384);
          bulk_g2s(rv, rec + kCtxY, 16384, bar_a);
        } else if (SD) {
          mbar_expect_tx(bar_a, 256);
          bulk_g2s(n_gm, rec + kCtxGa, 256, bar_a);
        }
        break;
    }
  };
  auto issue_a_raw = [&](int c) {
    switch (lane == 0 ? warp : -1) {
      case 7: mbar_expect_tx(bar_a, 8192); tma_load_4d(rkq, &mk, bar_a, 0, h, c * CM, b); break;
      case 8: mbar_expect_tx(bar_a, 8192); tma_load_4d(rkq + 8192, &mq, bar_a, 0, h, c * CM, b); break;
      case 9: mbar_expect_tx(bar_a, 8192); tma_load_4d(rkq + 16384, &mk, bar_a, 64, h, c * CM, b); break;
      case 10: mbar_expect_tx(bar_a, 8192); tma_load_4d(rkq + 24576, &mq, bar_a, 64, h, c * CM, b); break;
    }
  };
  auto issue_b_do = [&](int c) {
    if (lane == 0 && (warp == 11 || warp == 12)) {
      const int s = warp - 11;
      mbar_expect_tx(bar_b, 8192);
      tma_load_4d(rdo + s * 8192, &mdo, bar_b, 64 * s, h, c * CM, b);
    }
  };
  auto issue_b_v = [&](int c) {
    if (lane == 0 && (warp == 13 || warp == 14)) {
      const int s = warp - 13;
      mbar_expect_tx(bar_b, 8192);
      tma_load_4d(rv + s * 8192, &mv, bar_b, 64 * s, h, c * CM, b);
    }
  };
  auto issue_g = [&](int c) {
    const unsigned char *rec = a.fSin + ((size_t)bh * NC + c) * kCtxBytes;
    switch (lane == 0 ? warp : -1) {
      case 2: mbar_expect_tx(bar_g, 32768); bulk_g2s(sm + O_PHB, rec + kCtxPh, 32768, bar_g); break;
      case 3: mbar_expect_tx(bar_g, 16384); bulk_g2s(sm + O_GA0, rec + kCtxGa, 16384, bar_g); break;
      case 4: mbar_expect_tx(bar_g, 16384); bulk_g2s(sm + O_GA1, rec + kCtxGa + 16384, 16384, bar_g); break;
    }
  };
  // this chunk's omega logits for pass C (diagonal KDN with logit gates)
  auto issue_w = [&](int c) {
    if (WT && lane == 0 && (warp == 13 || warp == 14)) {
      const int s = warp - 13;
      mbar_expect_tx(bar_w, 8192);
      tma_load_4d(sm + O_KT + s * 8192, &mw, bar_w, 64 * s, h, c * CM, b);
    }
  };
  auto store_dv = [&](int c) {
    if (DVT && tid == 32) {
      tma_store_4d(&mdv, sm + O_DVS, 0, h, c * CM, b);
      tma_store_4d(&mdv, sm + O_DVS + 8192, 64, h, c * CM, b);
      bulk_commit();
    }
  };
  issue_a_ctx(NC - 1);
  issue_a_raw(NC - 1);
  issue_b_do(NC - 1);
  if (V != 0) issue_b_v(NC - 1);
  if (V == 0) issue_g(NC - 1);

  // ---- cotangent scale lambda = 2^-e with max(|dO|, |dS_T|) * lambda in [1, 2)
  {
    float m = 0.f;
    const unsigned char *dO = static_cast<const unsigned char *>(a.dO);
    for (int e = tid; e < a.T * 16; e += BT) {
      const int t = e >> 4, c16 = e & 15;
      const uint4 u = *reinterpret_cast<const uint4 *>(dO + (tok_index(a, b, t, h) * D) * 2 + c16 * 16);
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
    if (lane == 0) s_red[warp] = m;
    __syncthreads();
    if (tid == 0) {
      float mm = 0.f;
      for (int w = 0; w < BT / 32; ++w) mm = fmaxf(mm, s_red[w]);
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
  const float lam = s_misc[0], invl = 1.f / lam;

  // dS = lambda dS_T -> TMEM (row = key channel i, column = value j); dp = lambda dp_T
  {
    const int i = 32 * wq + lane;
    for (int c0 = 0; c0 < 32; c0 += 16) {
      float v[16];
      const int j0 = 32 * wg + c0;
      if (a.dST) {
        const float4 *src = reinterpret_cast<const float4 *>(a.dST + ((size_t)bh * D + i) * D + j0);
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          const float4 x = src[u];
          v[4 * u] = lam * x.x; v[4 * u + 1] = lam * x.y; v[4 * u + 2] = lam * x.z; v[4 * u + 3] = lam * x.w;
        }
      } else {
#pragma unroll
        for (int u = 0; u < 16; ++u) v[u] = 0.f;
      }
      tmem_st16(TS + lane_base + j0, v);
    }
    tmem_st_wait();
  }
  if (tid < D) {
    const size_t pi = V == 0 ? (size_t)bh * D + tid : (size_t)bh;
    s_dp[tid] = a.dpT ? lam * a.dpT[pi] : 0.f;
  }

  // per-token inputs of the next chunk (r; the scalar decay and omega of the isotropic KDN),
  // prefetched into registers and converted when they are used (a conversion here would
  // wait for the loads)
  __nv_bfloat16 nz = __float2bfloat16_rn(0.f), nx = nz, ny = nz;
  auto load_r = [&](int c) {
    if (tid < CM && c >= 0) {
      const size_t th = tok_index(a, b, min(c * CM + tid, a.T - 1), h);
      nz = static_cast<const __nv_bfloat16 *>(a.r)[th];
      if (V == 1 && !a.pcd) nx = static_cast<const __nv_bfloat16 *>(a.g)[th];
      if (V == 1 && G) ny = static_cast<const __nv_bfloat16 *>(a.omega)[th];
    }
  };
  load_r(NC - 1);

  uint32_t mma_phase = 0;
  bool ok = true;
  // Every thread polls the MMA-completion barrier itself (no CTA barrier between the
  // completion and the TMEM reads); the outcome is combined at the stage's closing barrier,
  // so that every thread leaves the loop at the same point
  auto mma_poll = [&]() -> bool {
    const bool r = mbar_wait(bar_mma, mma_phase & 1, kWaitIters);
    ++mma_phase;
    return r;
  };
  // the thread's tokens t0..t0+15: phat, gamma from TMEM, k from the raw tile
  auto load_ph_ga = [&](float *ph, float *ga) {
    tmem_ld16(TPH + lane_base + t0, ph);
    tmem_ld16(TGM + lane_base + t0, ga);
  };
  // gamma and the gain factor f_t with kappa = f_t k (diag: phat / s_t; iso: beta_t)
  auto load_gain = [&](float *gf, float *ga) {
    tmem_ld16(TGM + lane_base + t0, ga);
    if (V == 0) {
      tmem_ld16(TPH + lane_base + t0, gf);
#pragma unroll
      for (int j = 0; j < 16; ++j) gf[j] *= s_si[t0 + j];
    } else {
#pragma unroll
      for (int j = 0; j < 16; ++j) gf[j] = s_x[t0 + j];
    }
  };
  auto raw_k = [&](int t) { return bf(rkq, 16384, t, ci); };
  auto raw_q = [&](int t) { return bf(rkq + 8192, 16384, t, ci); };

  if (tid < CM) s_dmu[tid] = 0.f;  // ordered before use by the loop's barriers
  for (int it = 0; it < NC && ok; ++it) {
    const int c = NC - 1 - it;
    // ---- [1] per-token scalars; the chunk's gains from the context the forward saved (bulk
    //          copies; isotropic KDN with per-channel decay: global loads); raw tiles
    if (tid < CM) {
      // (with logit gates: and the chain factors sigmoid(z_t), sigmoid(y_t) of r and omega)
      const bool live = c * CM + tid < a.T;
      const float z = __bfloat162float(nz), nr = live ? gate_r(G, a.rmin, z) : 1.f;
      s_r[tid] = nr;
      s_ri[tid] = 1.f / nr;
      s_gs[tid] = V == 1 && !a.pcd && live ? gate_logalpha(G, __bfloat162float(nx)) : 0.f;
      s_fr[tid] = live ? dgate_sig(G, z) : 1.f;
      s_fw[tid] = V == 1 && G && live ? sigmoid_f(__bfloat162float(ny)) : 1.f;
    }
    const unsigned char *rec = a.fSin + ((size_t)bh * NC + c) * kCtxBytes;
    float e16[16], ph16[16];
    if (V != 0 && !SD) {  // gamma [64][128] of the isotropic KDN with per-channel decay
      const float *cga = reinterpret_cast<const float *>(rec + kCtxGa) + t0 * D + ci;
#pragma unroll
      for (int j = 0; j < 16; ++j) e16[j] = cga[j * D];
    }
    ok = __syncthreads_and(mbar_wait(bar_a, it & 1, kWaitIters) &&
                           (V != 0 || mbar_wait(bar_g, it & 1, kWaitIters)));
    if (!ok) break;
    load_r(c - 1);

    // ---- [2] the chunk's gains from the context the forward saved: phat (diag) and
    //          gamma -> TMEM (lane = channel), per-token s_t (diag) or beta_t, |k_t|^2,
    //          a_t, bhat_t, b_{t-1} (iso)
    float dgc = 0.f;  // this thread's part of dgamma_C for channel ci
    {
      if constexpr (V == 0) {
        const float *gs = reinterpret_cast<const float *>(sm + (qq < 2 ? O_GA0 : O_GA1)) + (t0 & 31) * D + ci;
        const float *ps = reinterpret_cast<const float *>(sm + O_PHB) + t0 * D + ci;
#pragma unroll
        for (int j = 0; j < 16; ++j) {
          e16[j] = gs[j * D];
          ph16[j] = ps[j * D];
        }
        tmem_st16(TPH + lane_base + t0, ph16);
      }
      if (SD) {  // one gamma per token
#pragma unroll
        for (int j = 0; j < 16; ++j) e16[j] = n_gm[t0 + j];
      }
      tmem_st16(TGM + lane_base + t0, e16);
      if (qq == 3) {
        s_gC[ci] = e16[15];
        check_gamma_range(e16[15], a.status);
      }
      if (SD && ci == 0) {
#pragma unroll
        for (int j = 0; j < 16; ++j) s_gm[t0 + j] = e16[j];
      }
      if (tid < CM) {
        if (V == 0) {
          s_s[tid] = n_tok[tid];
          s_si[tid] = 1.f / n_tok[tid];
        } else {
          s_x[tid] = n_tok[tid];
          s_n2[tid] = n_tok[CM + tid];
          s_a[tid] = n_tok[2 * CM + tid];
          s_bh[tid] = n_tok[3 * CM + tid];
          s_bp[tid] = n_tok[4 * CM + tid];
        }
      }
      tmem_st_wait();
      __syncthreads();
    }
    // ---- [3] operands of the chunk adjoint from the context and the gains:
    //          A bf16 (from the saved fp16 A); dS -> fp16 [i][j] (the B1 / B4 operand; dS <-
    //          gamma_C dS follows in [11], before B2 accumulates into it); K_tail^T [i][s];
    //          lambda dO and v to fp16 in place
    {
      const uint4 ah = sm16(sm + O_AH, tid * 16);  // 512 chunks of 8: the whole 8 KB tile
      float v[8];
      unpack_h8(ah, v);
      sm16(sm + O_AB, tid * 16) = pack_bf8(v);
    }
    {
      const int i = 32 * wq + lane;
      for (int c0 = 0; c0 < 32; c0 += 16) {
        float v[16], sv[16];
        const int j0 = 32 * wg + c0, sl = j0 >> 6, cc0 = (j0 & 63) >> 3;
        const uint32_t o0 = sl * 16384 + chunk_off(i, cc0), o1 = sl * 16384 + chunk_off(i, cc0 + 1);
        tmem_ld16(TS + lane_base + j0, v);
        sm16(sm + O_DSH, o0) = pack_h8(v);
        sm16(sm + O_DSH, o1) = pack_h8(v + 8);
        unpack_h8(sm16(sin, o0), sv);
        unpack_h8(sm16(sin, o1), sv + 8);
#pragma unroll
        for (int u = 0; u < 16; ++u) dgc += v[u] * sv[u];
      }
    }
    if (SD && tid < CM) s_kf[tid] = s_x[tid] * __frcp_rn(s_gm[tid]);
    {
      float gf[16], ga[16];
      load_gain(gf, ga);
      const float gC = s_gC[ci];
#pragma unroll
      for (int j = 0; j < 16; ++j) gf[j] = gC * __fdividef(gf[j] * raw_k(t0 + j), ga[j]);
      st_row16_h(sm + O_KT, ci, qq, gf);  // K_tail^T [i][s]
    }
    ok = __syncthreads_and(mbar_wait(bar_b, it & 1, kWaitIters));
    if (!ok) break;
    for (int e = tid; e < 64 * 16; e += BT) {
      const int row = e >> 4, c16 = e & 15;
      const uint32_t off = (c16 >> 3) * 8192 + chunk_off(row, c16 & 7);
      float v[8];
      unpack_bf8(sm16(rdo, off), v);
#pragma unroll
      for (int j = 0; j < 8; ++j) v[j] *= lam;
      sm16(rdo, off) = pack_h8(v);
      if (V != 0) {
        unpack_bf8(sm16(rv, off), v);
        sm16(rv, off) = pack_h8(v);
      }
    }
    tmem_st_wait();
    fence_proxy_async();
    tc_fence_before();
    __syncthreads();
    // ---- [10] B1: X2 = dR^T;  B3: X3 = dA_qk^T (before masking);  B4: X0 = dK_tail^T
    if (warp_u == 0) {
      tc_fence_after();
      const uint32_t lead = elect_one();
      const uint32_t id11 = idesc_f16(128, 64, 1, 1), id00 = idesc_f16(128, 64, 0, 0);
#pragma unroll
      for (int kk = 0; kk < 4; ++kk)
        umma_if(lead, X2, step(mdesc(rdo, 8192), kk * 2048), step(mdesc(sm + O_AQ, 8192), kk * 2048), id11, kk > 0);
#pragma unroll
      for (int kk = 0; kk < 8; ++kk)
        umma_if(lead, X2, step(mdesc(sm + O_DSH, 16384), kk * 2048), step(mdesc(sm + O_KT, 8192), kk * 2048), id11, 1);
#pragma unroll
      for (int kk = 0; kk < 8; ++kk) {
        const uint32_t o8 = (kk >> 2) * 8192 + (kk & 3) * 32;
        umma_if(lead, X3, step(kdesc(sm + O_RH), o8), step(kdesc(rdo), o8), id00, kk > 0);
        umma_if(lead, X0, step(kdesc(sm + O_DSH), (kk >> 2) * 16384 + (kk & 3) * 32), step(kdesc(sm + O_RH), o8),
                  id00, kk > 0);
      }
      commit_if(lead, bar_mma);
    }
    bool mm_ok = mma_poll();
    tc_fence_after();
    // ---- [11] dR^T -> fp16 [j][t] (and its fp16 remainder); dA_qk^T (masked to s <= t) -> hi/lo bf16 [s][t];
    //           X0 <- gamma_C dK_tail^T (start of dKk^T) and its dgamma_C part; Qbar fp16
    {
      const int j = 32 * wq + lane, tc0 = 16 * wg;
      float v[16];
      tmem_ld16(X2 + lane_base + tc0, v);
      uint4 l0, l1;
      sm16(sm + O_DRT, chunk_off(j, tc0 >> 3)) = split_h8(v, &l0);
      sm16(sm + O_DRT, chunk_off(j, (tc0 >> 3) + 1)) = split_h8(v + 8, &l1);
      sm16(sm + O_DRTL, chunk_off(j, tc0 >> 3)) = l0;
      sm16(sm + O_DRTL, chunk_off(j, (tc0 >> 3) + 1)) = l1;
      if (wq < 2) {
        tmem_ld16(X3 + lane_base + tc0, v);
#pragma unroll
        for (int u = 0; u < 16; ++u)
          if (tc0 + u < j) v[u] = 0.f;
        uint4 lo0, lo1;
        if (SD) {  // row s of dA_qk^T: diag(tau gamma) dA_qk -> O_AQ | O_DT (B9a)
          float w[16];
#pragma unroll
          for (int u = 0; u < 16; ++u) w[u] = v[u] * (tau * s_gm[tc0 + u]);
          sm16(sm + O_AQ, chunk_off(j, tc0 >> 3)) = split_bf8(w, &lo0);
          sm16(sm + O_AQ, chunk_off(j, (tc0 >> 3) + 1)) = split_bf8(w + 8, &lo1);
          sm16(sm + O_DT, chunk_off(j, tc0 >> 3)) = lo0;
          sm16(sm + O_DT, chunk_off(j, (tc0 >> 3) + 1)) = lo1;
          const float f = s_kf[j];  // dA_qk diag(beta / gamma) (B8b)
#pragma unroll
          for (int u = 0; u < 16; ++u) v[u] *= f;
        }
        sm16(sm + O_DAQ, chunk_off(j, tc0 >> 3)) = split_bf8(v, &lo0);
        sm16(sm + O_DAQ, chunk_off(j, (tc0 >> 3) + 1)) = split_bf8(v + 8, &lo1);
        sm16(sm + O_DAQ + 8192, chunk_off(j, tc0 >> 3)) = lo0;
        sm16(sm + O_DAQ + 8192, chunk_off(j, (tc0 >> 3) + 1)) = lo1;
      }
    }
    {
      float gf[16], ga[16], x[16];
      load_gain(gf, ga);
      tmem_ld16(X0 + lane_base + t0, x);
      const float gC = s_gC[ci];
#pragma unroll
      for (int j = 0; j < 16; ++j) {
        const int t = t0 + j;
        dgc += x[j] * __fdividef(gf[j] * raw_k(t), ga[j]);
        x[j] *= gC;
        gf[j] = tau * ga[j] * raw_q(t);
      }
      tmem_st16(X0 + lane_base + t0, x);
      st_row16_h(sm + O_QH, ci, qq, gf);  // Qbar^T [i][t]
    }
    {  // dS <- gamma_C dS in TMEM, before B2 accumulates into it
      const int i = 32 * wq + lane;
      const float gC = s_gC[i];
      for (int c0 = 0; c0 < 32; c0 += 16) {
        float v[16];
        const int j0 = 32 * wg + c0;
        tmem_ld16(TS + lane_base + j0, v);
#pragma unroll
        for (int u = 0; u < 16; ++u) v[u] *= gC;
        tmem_st16(TS + lane_base + j0, v);
      }
    }
    tmem_st_wait();
    fence_proxy_async();
    tc_fence_before();
    if (!__syncthreads_and(mm_ok)) {
      ok = false;
      break;
    }
    if constexpr (V == 0) {
      // Diagonal KDN: five tensor-core rounds.  With Y = V - Kbar S_in (the tile the
      // forward formed R = A Y from, in the context), dA = dR V^T + dW Kbar^T =
      // dR Y^T, since dW = -dR S_in^T: it comes out of the round that forms dR's
      // other products, and X = A^T dA one round later.
      // ---- [12] B2: TS += Qbar^T dO - W^T dR;  B5: X1 = -dW^T;  B6: X2 = dA^T = (dR Y^T)^T;
      //           B8a: X3 = (dO S_in^T)^T
      if (warp_u == 0) {
        tc_fence_after();
        const uint32_t lead = elect_one();
        const uint32_t idS01 = idesc_f16(128, 128, 0, 1), idS10 = idesc_f16(128, 128, 1, 0);
        const uint32_t id01 = idesc_f16(128, 64, 0, 1), id00 = idesc_f16(128, 64, 0, 0);
#pragma unroll
        for (int kk = 0; kk < 4; ++kk) {
          umma_if(lead, TS, step(kdesc(sm + O_QH), kk * 32), step(mdesc(rdo, 8192), kk * 2048), idS01, 1);
          umma_if(lead, TS, step(mdesc(sm + O_WN, 8192), kk * 2048), step(kdesc(sm + O_DRT), kk * 32), idS10, 1);
        }
#pragma unroll
        for (int kk = 0; kk < 8; ++kk) {
          const uint64_t as = step(kdesc(sin), (kk >> 2) * 16384 + (kk & 3) * 32);
          const uint64_t drt = step(mdesc(sm + O_DRT, 8192), kk * 2048);
          umma_if(lead, X1, as, drt, id01, kk > 0);
          umma_if(lead, X3, as, step(kdesc(rdo), (kk >> 2) * 8192 + (kk & 3) * 32), id00, kk > 0);
          umma_if(lead, X2, step(kdesc(rv), (kk >> 2) * 8192 + (kk & 3) * 32), drt, id01, kk > 0);
        }
        commit_if(lead, bar_mma);
      }
      mm_ok = mma_poll();
      tc_fence_after();
      // ---- [13] dW^T -> bf16 [i][t] (over Y);  dA^T -> fp16 [s][t] (over A_qk);
      //           second operand set: [Kbar; Qbar] hi (interleaved), Qbar lo, Kk hi / lo
      {
        const int j = 32 * wq + lane, tc0 = 16 * wg;
        float v[16];
        tmem_ld16(X1 + lane_base + tc0, v);
#pragma unroll
        for (int u = 0; u < 16; ++u) v[u] = -v[u];
        sm16(sm + O_DWY, chunk_off(j, tc0 >> 3)) = pack_bf8(v);
        sm16(sm + O_DWY, chunk_off(j, (tc0 >> 3) + 1)) = pack_bf8(v + 8);
        if (wq < 2) {
          tmem_ld16(X2 + lane_base + tc0, v);
          sm16(sm + O_DAY, chunk_off(j, tc0 >> 3)) = pack_h8(v);
          sm16(sm + O_DAY, chunk_off(j, (tc0 >> 3) + 1)) = pack_h8(v + 8);
        }
      }
      {
        float gf[16], ga[16], v[16];
        load_gain(gf, ga);
#pragma unroll
        for (int j = 0; j < 16; ++j) v[j] = ga[j] * raw_k(t0 + j);
        st_row16_bf(sm + O_KQH2, ci, qq, v);  // Kbar^T hi
      }
      {
        float gf[16], ga[16], v[16];
        load_gain(gf, ga);
#pragma unroll
        for (int j = 0; j < 16; ++j) v[j] = tau * ga[j] * raw_q(t0 + j);
        st_row16_split(sm + O_KQH2 + 16384, sm + O_QL2, ci, qq, v);  // Qbar^T hi / lo
#pragma unroll
        for (int j = 0; j < 16; ++j) v[j] = __fdividef(gf[j] * raw_k(t0 + j), ga[j]);
        st_row16_split(sm + O_KKH2, sm + O_KKL2, ci, qq, v);  // Kk^T hi / lo
      }
      fence_proxy_async();
      tc_fence_before();
      if (!__syncthreads_and(mm_ok)) {
        ok = false;
        break;
      }
      // ---- [14] B8b: X3 += (dA_qk Kk)^T;  B9a: X0 += (dA_qk^T Qbar)^T (hi/lo bf16 pairs);
      //           B7: X2 = dV^T = (A^T dR)^T (dR as hi + lo fp16);  X1 = A^T dA (fp16)
      if (warp_u == 0) {
        tc_fence_after();
        const uint32_t lead = elect_one();
        const uint32_t id01 = idesc_bf16(128, 64, 0, 1), id00 = idesc_bf16(128, 64, 0, 0);
        const uint32_t ih01 = idesc_f16(128, 64, 0, 1), ih10 = idesc_f16(128, 64, 1, 0);
#pragma unroll
        for (int kk = 0; kk < 4; ++kk) {
          const uint64_t kh = step(kdesc(sm + O_KKH2), kk * 32), kl = step(kdesc(sm + O_KKL2), kk * 32);
          const uint64_t dh = step(mdesc(sm + O_DAQ, 8192), kk * 2048), dl = step(mdesc(sm + O_DAQ + 8192, 8192), kk * 2048);
          umma_if(lead, X3, kh, dh, id01, 1);
          umma_if(lead, X3, kl, dh, id01, 1);
          umma_if(lead, X3, kh, dl, id01, 1);
          const uint64_t qh = step(kdesc(sm + O_KQH2 + 16384), kk * 32), ql = step(kdesc(sm + O_QL2), kk * 32);
          const uint64_t eh = step(kdesc(sm + O_DAQ), kk * 32), el = step(kdesc(sm + O_DAQ + 8192), kk * 32);
          umma_if(lead, X0, qh, eh, id00, 1);
          umma_if(lead, X0, ql, eh, id00, 1);
          umma_if(lead, X0, qh, el, id00, 1);
          const uint64_t ah = step(mdesc(sm + O_AH, 8192), kk * 2048);
          umma_if(lead, X2, step(kdesc(sm + O_DRT), kk * 32), ah, ih01, kk > 0);
          umma_if(lead, X2, step(kdesc(sm + O_DRTL), kk * 32), ah, ih01, 1);
          umma_if(lead, X1, ah, step(kdesc(sm + O_DAY), kk * 32), ih10, kk > 0);
        }
        commit_if(lead, bar_mma);
      }
      mm_ok = mma_poll();
      tc_fence_after();
      if (c > 0) issue_b_do(c - 1);  // the dO / Qbar lo buffer is free
      issue_w(c);  // into the dR^T buffer (free until [3] of the next chunk)
      // ---- [15] dV^T -> dv (bf16: into the dR^T lo tile, free since B7, in the layout of
      //           the TMA box, then two TMA stores; rows past T are clipped by the map);
      //           X = A^T dA -> fp16 [r][s]
      {
        const int j = 32 * wq + lane, tc0 = 16 * wg;
        float v[16];
        tmem_ld16(X2 + lane_base + tc0, v);
        if constexpr (DVT) {
          unsigned char *slab = sm + O_DVS + (j >> 6) * 8192;
#pragma unroll
          for (int u = 0; u < 16; ++u)
            *reinterpret_cast<__nv_bfloat16 *>(slab + chunk_off(tc0 + u, (j & 63) >> 3) + 2 * (j & 7)) =
                __float2bfloat16_rn(v[u] * invl);
        } else {
#pragma unroll
          for (int u = 0; u < 16; ++u) {
            const int t = c * CM + tc0 + u;
            if (t < a.T) st_grad<OBF>(a.dv_, tok_index(a, b, t, h) * D + j, v[u] * invl);
          }
        }
        if (wq < 2) {
          tmem_ld16(X1 + lane_base + tc0, v);
          sm16(sm + O_XT, chunk_off(j, tc0 >> 3)) = pack_h8(v);
          sm16(sm + O_XT, chunk_off(j, (tc0 >> 3) + 1)) = pack_h8(v + 8);
        }
      }
      fence_proxy_async();
      tc_fence_before();
      if (!__syncthreads_and(mm_ok)) {
        ok = false;
        break;
      }
      store_dv(c);
      // ---- [16] X1 = X A^T (fp16), so that dT = strict_lower(-A^T dA A^T);  B10a: X2 = (A^T dW)^T
      if (warp_u == 0) {
        tc_fence_after();
        const uint32_t lead = elect_one();
        const uint32_t ih00 = idesc_f16(128, 64, 0, 0), ib01 = idesc_bf16(128, 64, 0, 1);
#pragma unroll
        for (int kk = 0; kk < 4; ++kk) {
          umma_if(lead, X1, step(kdesc(sm + O_XT), kk * 32), step(kdesc(sm + O_AH), kk * 32), ih00, kk > 0);
          umma_if(lead, X2, step(kdesc(sm + O_DWY), kk * 32), step(mdesc(sm + O_AB, 8192), kk * 2048), ib01, kk > 0);
        }
        commit_if(lead, bar_mma);
      }
      mm_ok = mma_poll();
      tc_fence_after();
      if (wq < 2) {  // dT -> bf16
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
      // ---- [17] B9b: X0 += (dT^T Kbar)^T;  B10b: X2 += (dT Kk)^T
      if (warp_u == 0) {
        tc_fence_after();
        const uint32_t lead = elect_one();
        const uint32_t id01 = idesc_bf16(128, 64, 0, 1), id00 = idesc_bf16(128, 64, 0, 0);
#pragma unroll
        for (int kk = 0; kk < 4; ++kk) {
          umma_if(lead, X0, step(kdesc(sm + O_KQH2), kk * 32), step(mdesc(sm + O_DT, 8192), kk * 2048), id01, 1);
          umma_if(lead, X2, step(kdesc(sm + O_KKH2), kk * 32), step(kdesc(sm + O_DT), kk * 32), id00, 1);
        }
        commit_if(lead, bar_mma);
      }
    } else {
      // Isotropic KDN: seven rounds (its context keeps no Y; B6 forms dA from V and dW)
      // ---- [12] B2: TS += Qbar^T dO - W^T dR;  B5: X1 = -dW^T;  B7: X2 = dV^T (dR as hi + lo fp16);
      //           B8a: X3 = (dO S_in^T)^T
      if (warp_u == 0) {
        tc_fence_after();
        const uint32_t lead = elect_one();
        const uint32_t idS01 = idesc_f16(128, 128, 0, 1), idS10 = idesc_f16(128, 128, 1, 0);
        const uint32_t id01 = idesc_f16(128, 64, 0, 1), id00 = idesc_f16(128, 64, 0, 0);
#pragma unroll
        for (int kk = 0; kk < 4; ++kk) {
          umma_if(lead, TS, step(kdesc(sm + O_QH), kk * 32), step(mdesc(rdo, 8192), kk * 2048), idS01, 1);
          umma_if(lead, TS, step(mdesc(sm + O_WN, 8192), kk * 2048), step(kdesc(sm + O_DRT), kk * 32), idS10, 1);
          const uint64_t ah = step(mdesc(sm + O_AH, 8192), kk * 2048);
          umma_if(lead, X2, step(kdesc(sm + O_DRT), kk * 32), ah, id01, kk > 0);
          umma_if(lead, X2, step(kdesc(sm + O_DRTL), kk * 32), ah, id01, 1);
        }
#pragma unroll
        for (int kk = 0; kk < 8; ++kk) {
          const uint64_t as = step(kdesc(sin), (kk >> 2) * 16384 + (kk & 3) * 32);
          umma_if(lead, X1, as, step(mdesc(sm + O_DRT, 8192), kk * 2048), id01, kk > 0);
          umma_if(lead, X3, as, step(kdesc(rdo), (kk >> 2) * 8192 + (kk & 3) * 32), id00, kk > 0);
        }
        commit_if(lead, bar_mma);
      }
      mm_ok = mma_poll();
      tc_fence_after();
      // ---- [13] second operand set: [Kbar; Qbar] hi (interleaved), Qbar lo, Kk hi / lo;
      //           B8b: X3 += (dA_qk Kk)^T;  B9a: X0 += (dA_qk^T Qbar)^T
      {
        float gf[16], ga[16], v[16];
        load_gain(gf, ga);
  #pragma unroll
        for (int j = 0; j < 16; ++j) v[j] = ga[j] * raw_k(t0 + j);
        st_row16_bf(sm + O_KQH2, ci, qq, v);  // Kbar^T hi
      }
      if (!SD) {
        float gf[16], ga[16], v[16];
        load_gain(gf, ga);
  #pragma unroll
        for (int j = 0; j < 16; ++j) v[j] = tau * ga[j] * raw_q(t0 + j);
        st_row16_split(sm + O_KQH2 + 16384, sm + O_QL2, ci, qq, v);  // Qbar^T hi / lo
  #pragma unroll
        for (int j = 0; j < 16; ++j) v[j] = __fdividef(gf[j] * raw_k(t0 + j), ga[j]);
        st_row16_split(sm + O_KKH2, sm + O_KKL2, ci, qq, v);  // Kk^T hi / lo
      }
      fence_proxy_async();
      tc_fence_before();
      if (!__syncthreads_and(mm_ok)) {
        ok = false;
        break;
      }
      if (SD && warp_u == 0) {  // raw K^T, Q^T (channel-major) against the scaled 64 x 64 partners
        tc_fence_after();
        const uint32_t lead = elect_one();
        const uint32_t id11 = idesc_bf16(128, 64, 1, 1), id10 = idesc_bf16(128, 64, 1, 0);
#pragma unroll
        for (int kk = 0; kk < 4; ++kk) {
          const uint64_t kt = step(mdesc(rkq, 16384), kk * 2048), qt = step(mdesc(rkq + 8192, 16384), kk * 2048);
          umma_if(lead, X3, kt, step(mdesc(sm + O_DAQ, 8192), kk * 2048), id11, 1);
          umma_if(lead, X3, kt, step(mdesc(sm + O_DAQ + 8192, 8192), kk * 2048), id11, 1);
          umma_if(lead, X0, qt, step(kdesc(sm + O_AQ), kk * 32), id10, 1);
          umma_if(lead, X0, qt, step(kdesc(sm + O_DT), kk * 32), id10, 1);
        }
        commit_if(lead, bar_mma);
      }
      if (!SD && warp_u == 0) {
        tc_fence_after();
        const uint32_t lead = elect_one();
        const uint32_t id01 = idesc_bf16(128, 64, 0, 1), id00 = idesc_bf16(128, 64, 0, 0);
#pragma unroll
        for (int kk = 0; kk < 4; ++kk) {
          const uint64_t kh = step(kdesc(sm + O_KKH2), kk * 32), kl = step(kdesc(sm + O_KKL2), kk * 32);
          const uint64_t dh = step(mdesc(sm + O_DAQ, 8192), kk * 2048), dl = step(mdesc(sm + O_DAQ + 8192, 8192), kk * 2048);
          umma_if(lead, X3, kh, dh, id01, 1);
          umma_if(lead, X3, kl, dh, id01, 1);
          umma_if(lead, X3, kh, dl, id01, 1);
          const uint64_t qh = step(kdesc(sm + O_KQH2 + 16384), kk * 32), ql = step(kdesc(sm + O_QL2), kk * 32);
          const uint64_t eh = step(kdesc(sm + O_DAQ), kk * 32), el = step(kdesc(sm + O_DAQ + 8192), kk * 32);
          umma_if(lead, X0, qh, eh, id00, 1);
          umma_if(lead, X0, ql, eh, id00, 1);
          umma_if(lead, X0, qh, el, id00, 1);
        }
        commit_if(lead, bar_mma);
      }
      mm_ok = mma_poll();
      tc_fence_after();
      if (c > 0) issue_b_do(c - 1);  // dO / Qbar lo buffer is free
      // ---- [14] dW^T -> bf16 [i][t];  dV^T -> dv
      {
        const int j = 32 * wq + lane, tc0 = 16 * wg;
        float v[16];
        tmem_ld16(X1 + lane_base + tc0, v);
  #pragma unroll
        for (int u = 0; u < 16; ++u) v[u] = -v[u];
        sm16(sm + O_DWT, chunk_off(j, tc0 >> 3)) = pack_bf8(v);
        sm16(sm + O_DWT, chunk_off(j, (tc0 >> 3) + 1)) = pack_bf8(v + 8);
        tmem_ld16(X2 + lane_base + tc0, v);
        if constexpr (DVT) {  // into the dR^T lo tile (free since B7) for two TMA stores
          unsigned char *slab = sm + O_DVS + (j >> 6) * 8192;
  #pragma unroll
          for (int u = 0; u < 16; ++u)
            *reinterpret_cast<__nv_bfloat16 *>(slab + chunk_off(tc0 + u, (j & 63) >> 3) + 2 * (j & 7)) =
                __float2bfloat16_rn(v[u] * invl);
        } else {
  #pragma unroll
          for (int u = 0; u < 16; ++u) {
            const int t = c * CM + tc0 + u;
            if (t < a.T) st_grad<OBF>(a.dv_, tok_index(a, b, t, h) * D + j, v[u] * invl);
          }
        }
      }
      fence_proxy_async();
      tc_fence_before();
      if (!__syncthreads_and(mm_ok)) {
        ok = false;
        break;
      }
      store_dv(c);
      // ---- [15] B6: X1 = dA^T = (dR V^T + dW Kbar^T)^T;  B10a: X2 = (A^T dW)^T
      if (warp_u == 0) {
        tc_fence_after();
        const uint32_t lead = elect_one();
        const uint32_t ih01 = idesc_f16(128, 64, 0, 1), ib01 = idesc_bf16(128, 64, 0, 1);
        const uint32_t ib11 = idesc_bf16(128, 64, 1, 1);
#pragma unroll
        for (int kk = 0; kk < 8; ++kk) {
          umma_if(lead, X1, step(kdesc(rv), (kk >> 2) * 8192 + (kk & 3) * 32), step(mdesc(sm + O_DRT, 8192), kk * 2048),
                    ih01, kk > 0);
          umma_if(lead, X1, step(mdesc(sm + O_KQH2, 16384), kk * 2048), step(mdesc(sm + O_DWT, 8192), kk * 2048), ib11,
                    1);
        }
#pragma unroll
        for (int kk = 0; kk < 4; ++kk)
          umma_if(lead, X2, step(kdesc(sm + O_DWT), kk * 32), step(mdesc(sm + O_AB, 8192), kk * 2048), ib01, kk > 0);
        commit_if(lead, bar_mma);
      }
      mm_ok = mma_poll();
      tc_fence_after();
      if (c > 0) issue_b_v(c - 1);  // v buffer is free
      // ---- [16] dT = strict_lower(-A^T dA A^T): X = A^T dA, Y = X A^T (fp16)
      if (wq < 2) {
        const int s = 32 * wq + lane, tc0 = 16 * wg;
        float v[16];
        tmem_ld16(X1 + lane_base + tc0, v);
        sm16(sm + O_DAT, chunk_off(s, tc0 >> 3)) = pack_h8(v);
        sm16(sm + O_DAT, chunk_off(s, (tc0 >> 3) + 1)) = pack_h8(v + 8);
      }
      fence_proxy_async();
      tc_fence_before();
      if (!__syncthreads_and(mm_ok)) {
        ok = false;
        break;
      }
      if (warp_u == 0) {
        tc_fence_after();
        const uint32_t lead = elect_one();
        const uint32_t id = idesc_f16(128, 64, 1, 0);
#pragma unroll
        for (int kk = 0; kk < 4; ++kk)
          umma_if(lead, X1, step(mdesc(sm + O_AH, 8192), kk * 2048), step(kdesc(sm + O_DAT), kk * 32), id, kk > 0);
        commit_if(lead, bar_mma);
      }
      mm_ok = mma_poll();
      tc_fence_after();
      if (wq < 2) {
        const int r = 32 * wq + lane, tc0 = 16 * wg;
        float v[16];
        tmem_ld16(X1 + lane_base + tc0, v);
        sm16(sm + O_XT, chunk_off(r, tc0 >> 3)) = pack_h8(v);
        sm16(sm + O_XT, chunk_off(r, (tc0 >> 3) + 1)) = pack_h8(v + 8);
      }
      fence_proxy_async();
      tc_fence_before();
      if (!__syncthreads_and(mm_ok)) {
        ok = false;
        break;
      }
      if (warp_u == 0) {
        tc_fence_after();
        const uint32_t lead = elect_one();
        const uint32_t id = idesc_f16(128, 64, 0, 0);
#pragma unroll
        for (int kk = 0; kk < 4; ++kk)
          umma_if(lead, X1, step(kdesc(sm + O_XT), kk * 32), step(kdesc(sm + O_AH), kk * 32), id, kk > 0);
        commit_if(lead, bar_mma);
      }
      mm_ok = mma_poll();
      tc_fence_after();
      if (wq < 2) {
        const int r = 32 * wq + lane, tc0 = 16 * wg;
        float v[16];
        tmem_ld16(X1 + lane_base + tc0, v);
  #pragma unroll
        for (int u = 0; u < 16; ++u) v[u] = (tc0 + u < r) ? -v[u] : 0.f;
        if (SD) {  // dT diag(beta / gamma) -> O_AQ (B10b); diag(gamma) dT below (B9b)
          float w[16];
  #pragma unroll
          for (int u = 0; u < 16; ++u) w[u] = v[u] * s_kf[tc0 + u];
          sm16(sm + O_AQ, chunk_off(r, tc0 >> 3)) = pack_bf8(w);
          sm16(sm + O_AQ, chunk_off(r, (tc0 >> 3) + 1)) = pack_bf8(w + 8);
          const float f = s_gm[r];
  #pragma unroll
          for (int u = 0; u < 16; ++u) v[u] *= f;
        }
        sm16(sm + O_DT, chunk_off(r, tc0 >> 3)) = pack_bf8(v);
        sm16(sm + O_DT, chunk_off(r, (tc0 >> 3) + 1)) = pack_bf8(v + 8);
      }
      fence_proxy_async();
      tc_fence_before();
      if (!__syncthreads_and(mm_ok)) {
        ok = false;
        break;
      }
      // ---- [17] B9b: X0 += (dT^T Kbar)^T;  B10b: X2 += (dT Kk)^T
      if (warp_u == 0) {
        tc_fence_after();
        const uint32_t lead = elect_one();
        const uint32_t id01 = idesc_bf16(128, 64, 0, 1), id00 = idesc_bf16(128, 64, 0, 0);
        const uint32_t id11 = idesc_bf16(128, 64, 1, 1), id10 = idesc_bf16(128, 64, 1, 0);
#pragma unroll
        for (int kk = 0; kk < 4; ++kk) {
          if (SD) {
            const uint64_t kt = step(mdesc(rkq, 16384), kk * 2048);
            umma_if(lead, X0, kt, step(mdesc(sm + O_DT, 8192), kk * 2048), id11, 1);
            umma_if(lead, X2, kt, step(kdesc(sm + O_AQ), kk * 32), id10, 1);
          } else {
            umma_if(lead, X0, step(kdesc(sm + O_KQH2), kk * 32), step(mdesc(sm + O_DT, 8192), kk * 2048), id01, 1);
            umma_if(lead, X2, step(kdesc(sm + O_KKH2), kk * 32), step(kdesc(sm + O_DT), kk * 32), id00, 1);
          }
        }
        commit_if(lead, bar_mma);
      }
    }
    mm_ok = mma_poll();
    tc_fence_after();
    if (c > 0) {
      issue_a_ctx(c - 1);  // the context buffers are free
      // phat and gamma of chunk c - 1, which are read later, into L2 now
      if (tid == 480) bulk_prefetch_l2(rec - kCtxBytes + kCtxPh, SD ? 256 : 65536);
    }
    // ---- [18] per channel (lane ci, tokens t0..t0+15): back through Gamma and the
    //           gain emission, then the uncertainty recursion backwards in time.
    //           Free TMEM columns hold per-(channel, token) intermediates between passes:
    //           X2 <- dphat (gain part), X1 <- dk (memory + gain part), X0 <- alpha,
    //           X3 <- 1 / (1 + u phat).
    if (V == 0)
    {
      float *sdg = reinterpret_cast<float *>(sm + O_G);  // [16][512] dG_t
      float *s_tot = reinterpret_cast<float *>(sm + O_DT);  // [4][128] quarter sums of dG
      float *s_dgc = s_tot + 512;                           // [4][128] dgamma_C parts
      float *s_aff = s_dgc + 512;                           // [4][128][2] affine summaries
      float ph[16], ga[16], k16[16], q16[16];
      load_ph_ga(ph, ga);
#pragma unroll
      for (int j = 0; j < 16; ++j) {
        k16[j] = raw_k(t0 + j);
        q16[j] = raw_q(t0 + j);
      }
      const float kprev = qq > 0 ? raw_k(t0 - 1) : 0.f;
      fence_proxy_async();
      // raw k, q are in registers: the next chunk's tiles may land
      if (!__syncthreads_and(mm_ok)) {
        ok = false;
        break;
      }
      if (c > 0) issue_a_raw(c - 1);
      // outputs of token t0 + j live at obase + j * ostride; nval tokens of the quarter are real
      const size_t ostride = (size_t)a.H * D;
      const size_t obase = tok_index(a, b, c * CM + t0, h) * D + ci;
      const int nval = min(16, a.T - (c * CM + t0));
      auto out = [&](void *p, int j, float x) { st_grad<OBF>(p, obase + (size_t)j * ostride, x); };
      // pass A: dq, dG, the ds_t partial sums and the ds-free parts of dphat and dk
      {
        float part[16], tot = 0.f;
#pragma unroll
        for (int h8 = 0; h8 < 2; ++h8) {
          float xq[8], xk[8], xb[8], c1[8], c2[8];
          tmem_ld8(X3 + lane_base + t0 + 8 * h8, xq);
          tmem_ld8(X0 + lane_base + t0 + 8 * h8, xk);
          tmem_ld8(X2 + lane_base + t0 + 8 * h8, xb);
#pragma unroll
          for (int u = 0; u < 8; ++u) {
            const int j = 8 * h8 + u, t = t0 + j;
            const float kk = k16[j], qv = q16[j], si = s_si[t], g_ = ga[j], ig = __fdividef(1.f, g_);
            const float kap = ph[j] * kk * si;  // kappa_t (eq. kla-box-gain)
            const float dG = xb[u] * g_ * kk - xk[u] * kap * ig + xq[u] * tau * g_ * qv;
            sdg[j * BT + tid] = dG;
            tot += dG;
            const float dkap = xk[u] * ig;
            part[j] = dkap * kap;
            c1[u] = dkap * kk * si;
            c2[u] = xb[u] * g_ + dkap * ph[j] * si;
            if (j < nval) out(a.dq, j, tau * g_ * xq[u] * invl);
          }
          tmem_st8(X2 + lane_base + t0 + 8 * h8, c1);
          tmem_st8(X1 + lane_base + t0 + 8 * h8, c2);
        }
        s_dgc[qq * D + ci] = dgc;
        s_tot[qq * D + ci] = tot;
        const float rsum = rs16(part, lane);
        if ((lane & 1) == 0) s_red[wq * 64 + t0 + (lane >> 1)] = rsum;
      }
      tmem_st_wait();
      __syncthreads();
      if (tid < CM) s_ds[tid] = -((s_red[tid] + s_red[64 + tid]) + (s_red[128 + tid] + s_red[192 + tid])) * s_si[tid];
      __syncthreads();
      // entry values of this quarter: gamma_{t0-1}, p_{t0-1}
      float ga_prev = 1.f, p_prev;
      if (qq > 0) {
        float t8[8], g8[8];
        tmem_ld8(TPH + lane_base + t0 - 8, t8);
        tmem_ld8(TGM + lane_base + t0 - 8, g8);
        const float kk = kprev;
        ga_prev = g8[7];  // gamma_{t0-1}
        p_prev = __fdividef(t8[7], 1.f + mu * kk * kk * s_ri[t0 - 1] * t8[7]);
      } else {
        p_prev = a.fpin[((size_t)bh * NC + c) * D + ci];
      }
      // pass B: per-token coefficients of dp_{t-1} = a_t dp_t + b_t and the quarter's
      //         composition dp_before = A dp_after + B
      {
        float A = 1.f, Bv = 0.f;
#pragma unroll
        for (int h8 = 1; h8 >= 0; --h8) {
          float c1[8], a2v[8], rdv[8];
          tmem_ld8(X2 + lane_base + t0 + 8 * h8, c1);
#pragma unroll
          for (int u = 7; u >= 0; --u) {
            const int j = 8 * h8 + u, t = t0 + j;
            const float kk = k16[j];
            const float al = __fdividef(ga[j], j > 0 ? ga[j - 1] : ga_prev), al2 = al * al;
            const float rd = __fdividef(1.f, 1.f + mu * kk * kk * s_ri[t] * ph[j]);
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
        s_aff[(qq * D + ci) * 2] = A;
        s_aff[(qq * D + ci) * 2 + 1] = Bv;
      }
      tmem_st_wait();
      if (WT) {  // logit gates: the omega-logit tile has landed
        ok = __syncthreads_and(tid != 0 || mbar_wait(bar_w, it & 1, kWaitIters));
        if (!ok) break;
      } else {
        __syncthreads();
      }
      // pass C: the recursion backwards through this quarter's tokens
      {
        float dp = s_dp[ci];
        for (int q2 = 3; q2 > qq; --q2) dp = s_aff[(q2 * D + ci) * 2] * dp + s_aff[(q2 * D + ci) * 2 + 1];
        const float dgC = (s_dgc[ci] + s_dgc[D + ci]) + (s_dgc[2 * D + ci] + s_dgc[3 * D + ci]);
        float run = dgC * s_gC[ci];  // dG_63 gains dgamma_C gamma_C; it lies in every suffix
        for (int q2 = qq + 1; q2 < 4; ++q2) run += s_tot[q2 * D + ci];
        float rd16[16], drp[16];
        // logit gates: the quarter's omega logits (TMA tile in O_KT; zero past T) for the
        // chain factor sigmoid(y) of domega
        float ylog[16];
        if (G) {
#pragma unroll
          for (int j = 0; j < 16; ++j) ylog[j] = bf(sm + O_KT, 8192, t0 + j, ci);
        }
        tmem_ld16(X3 + lane_base + t0, rd16);
#pragma unroll
        for (int h8 = 1; h8 >= 0; --h8) {
          float a2v[8], dphl[8], c2[8];
          tmem_ld8(X0 + lane_base + t0 + 8 * h8, a2v);
          tmem_ld8(X2 + lane_base + t0 + 8 * h8, dphl);
          tmem_ld8(X1 + lane_base + t0 + 8 * h8, c2);
#pragma unroll
          for (int u = 7; u >= 0; --u) {
            const int j = 8 * h8 + u, t = t0 + j;
            const float kk = k16[j], ds = s_ds[t], ri = s_ri[t];
            const float pt = ph[j] * rd16[j];
            const float pprev = j > 0 ? ph[j - 1] * rd16[j - 1] : p_prev;
            const float dph = dp * rd16[j] * rd16[j] + dphl[u];
            const float du = -dp * pt * pt;
            const float dkt = c2[u] + 2.f * ds * ph[j] * kk + du * 2.f * mu * kk * ri;
            drp[j] = -du * mu * kk * kk * ri * ri;
            run += sdg[j * BT + tid];
            const float al2 = a2v[u] * a2v[u];
            const float dgt = run + 2.f * al2 * pprev * dph;
            if (j < nval) {
              // logit gates: d omega / dy = sigmoid(y), d log alpha / dx = 1 - alpha
              const float fw = G ? sigmoid_f(ylog[j]) : 1.f;
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
        fence_proxy_async();
        __syncthreads();
        // every read of the dG scratch, the pass summaries and the omega logits is done:
        // the next chunk's phat and gamma may land over them
        if (c > 0) issue_g(c - 1);
        if (qq == 0) s_dp[ci] = dp;
        if (tid < CM) {
          const int tt = c * CM + tid;
          if (tt < a.T) {
            // the part of dr_t through u = mu k^2 / r: -sum_i du mu k^2 / r^2
            const float dru = (s_red2[tid] + s_red2[64 + tid]) + (s_red2[128 + tid] + s_red2[192 + tid]);
            const float dr = s_ds[tid] + dru;
            st_grad<OBF>(a.dr, tok_index(a, b, tt, h), dr * (G ? s_fr[tid] : 1.f) * invl);
            // dL/dmu gains sum_i du k^2 / r = -dru r / mu
            if (a.dmu) s_dmu[tid] += -dru * s_r[tid] / mu;
          }
        }
      }
    }
    else {
      // Isotropic KDN: kappa_t = beta_t k_t with one uncertainty b per head.
      float *sdg = reinterpret_cast<float *>(sm + O_G);  // [16][512] dG_t
      float *s_tot = reinterpret_cast<float *>(sm + O_DT);  // [4][128] quarter sums of dG
      float *s_dgc = s_tot + 512;                           // [4][128] dgamma_C parts
      float ga[16], k16[16], q16[16];
      tmem_ld16(TGM + lane_base + t0, ga);
#pragma unroll
      for (int j = 0; j < 16; ++j) {
        k16[j] = raw_k(t0 + j);
        q16[j] = raw_q(t0 + j);
      }
      fence_proxy_async();
      // raw k, q are in registers: the next chunk's tiles may land
      if (!__syncthreads_and(mm_ok)) {
        ok = false;
        break;
      }
      if (c > 0) issue_a_raw(c - 1);
      const size_t ostride = (size_t)a.H * D;
      const size_t obase = tok_index(a, b, c * CM + t0, h) * D + ci;
      const int nval = min(16, a.T - (c * CM + t0));
      auto out = [&](void *p, int j, float x) { st_grad<OBF>(p, obase + (size_t)j * ostride, x); };
      // pass A: dq, dG, the dbeta_t partial sums and dk from the memory path and kappa
      {
        float part[16], tot = 0.f;
#pragma unroll
        for (int h8 = 0; h8 < 2; ++h8) {
          float xq[8], xk[8], xb[8], c2[8];
          tmem_ld8(X3 + lane_base + t0 + 8 * h8, xq);
          tmem_ld8(X0 + lane_base + t0 + 8 * h8, xk);
          tmem_ld8(X2 + lane_base + t0 + 8 * h8, xb);
#pragma unroll
          for (int u = 0; u < 8; ++u) {
            const int j = 8 * h8 + u, t = t0 + j;
            const float kk = k16[j], qv = q16[j], g_ = ga[j], ig = __fdividef(1.f, g_);
            const float beta = s_x[t], kap = beta * kk;
            const float dG = xb[u] * g_ * kk - xk[u] * kap * ig + xq[u] * tau * g_ * qv;
            sdg[j * BT + tid] = dG;
            tot += dG;
            const float dkap = xk[u] * ig;
            part[j] = dkap * kk;
            c2[u] = xb[u] * g_ + beta * dkap;
            if (j < nval) out(a.dq, j, tau * g_ * xq[u] * invl);
          }
          tmem_st8(X1 + lane_base + t0 + 8 * h8, c2);
        }
        s_dgc[qq * D + ci] = dgc;
        s_tot[qq * D + ci] = tot;
        const float rsum = rs16(part, lane);
        if ((lane & 1) == 0) s_red[wq * 64 + t0 + (lane >> 1)] = rsum;
      }
      tmem_st_wait();
      __syncthreads();
      if (tid < CM) s_ds[tid] = (s_red[tid] + s_red[64 + tid]) + (s_red[128 + tid] + s_red[192 + tid]);
      __syncthreads();
      // the scalar recursion backwards over the chunk, db_{t-1} = A_t db_t + B_t with
      // A_t = a_t / den_t^2 and B_t = a_t dbeta_t r_t / dd_t^2, as a suffix scan of
      // these affine maps in one warp (lane l holds tokens 2l, 2l + 1); A_t <= 1
      float db_in = 0.f;
      if (warp == 0) {
        const int ta = 2 * lane, tb = ta + 1;
        auto coef = [&](int t, float &A_, float &B_, float &rden, float &dd) {
          const float bhat = s_bh[t], u = mu * s_n2[t] * s_ri[t] * (1.f / D);
          rden = __fdividef(1.f, 1.f + u * bhat);
          dd = s_r[t] + bhat * s_n2[t];
          A_ = s_a[t] * rden * rden;
          B_ = s_a[t] * __fdividef(s_ds[t] * s_r[t], dd * dd);
        };
        float Aa, Ba, rda, dda, Ab, Bb, rdb, ddb;
        coef(ta, Aa, Ba, rda, dda);
        coef(tb, Ab, Bb, rdb, ddb);
        // this pair's map db_{tb} -> db_{ta - 1}, then composed with the later pairs'
        float SA = Aa * Ab, SB = fmaf(Aa, Bb, Ba);
#pragma unroll
        for (int off = 1; off < 32; off <<= 1) {
          const float pA = __shfl_down_sync(0xffffffffu, SA, off);
          const float pB = __shfl_down_sync(0xffffffffu, SB, off);
          if (lane + off < 32) {
            SB = fmaf(SA, pB, SB);
            SA = SA * pA;
          }
        }
        // the later pairs' map applied to the cotangent entering from the next chunk
        float EA = __shfl_down_sync(0xffffffffu, SA, 1), EB = __shfl_down_sync(0xffffffffu, SB, 1);
        if (lane == 31) { EA = 1.f; EB = 0.f; }
        const float dbb = fmaf(EA, s_dp[0], EB);  // db_{tb}
        const float dba = fmaf(Ab, dbb, Bb);      // db_{ta}
        float dmu = 0.f;
        auto tok = [&](int t, float dbt, float rden, float dd) {
          const float bhat = s_bh[t], beta = s_x[t], n2 = s_n2[t], r = s_r[t], ri = s_ri[t];
          const float u = mu * n2 * ri * (1.f / D), bt = bhat * rden, dbeta = s_ds[t];
          const float dbhat = dbt * rden * rden + __fdividef(dbeta * r, dd * dd);
          const float du = -dbt * bt * bt;
          dmu += du * n2 * ri * (1.f / D);  // u = mu |k|^2 / (dk r)
          s_dn2[t] = -dbeta * beta * beta + du * mu * ri * (1.f / D);
          s_da[t] = s_bp[t] * dbhat;
          const int tt = c * CM + t;
          if (tt < a.T) {
            const size_t th = tok_index(a, b, tt, h);
            st_grad<OBF>(a.domega, th, dbhat * (G ? s_fw[t] : 1.f) * invl);
            st_grad<OBF>(a.dr, th, (-__fdividef(dbeta * beta, dd) - du * u * ri) * (G ? s_fr[t] : 1.f) * invl);
          }
          return s_a[t] * dbhat;  // db_{t-1}
        };
        tok(tb, dbb, rdb, ddb);
        db_in = tok(ta, dba, rda, dda);  // lane 0: the cotangent leaving the chunk
        if (a.dmu) {
          dmu = warp_sum(dmu);
          if (lane == 0) s_dmu[0] += dmu;
        }
      }
      __syncthreads();
      if (tid == 0) s_dp[0] = db_in;
      // per element: dk and dg
      {
        const float dgC = (s_dgc[ci] + s_dgc[D + ci]) + (s_dgc[2 * D + ci] + s_dgc[3 * D + ci]);
        float run = dgC * s_gC[ci];  // dG_63 gains dgamma_C gamma_C; it lies in every suffix
        for (int q2 = qq + 1; q2 < 4; ++q2) run += s_tot[q2 * D + ci];
        float ga_prev = 1.f;
        if (qq > 0) {
          float g8[8];
          tmem_ld8(TGM + lane_base + t0 - 8, g8);
          ga_prev = g8[7];
        }
        float c2[16], dgp[16];
        tmem_ld16(X1 + lane_base + t0, c2);
#pragma unroll
        for (int j = 15; j >= 0; --j) {
          const int t = t0 + j;
          run += sdg[j * BT + tid];
          if (j < nval) out(a.dk_, j, (c2[j] + 2.f * k16[j] * s_dn2[t]) * invl);
          if (pcd) {
            const float al = __fdividef(ga[j], j > 0 ? ga[j - 1] : ga_prev);
            const float fg = G ? 1.f - al : 1.f;  // d log alpha / dx
            if (j < nval) out(a.dg, j, (run + s_da[t] * 2.f * al * al * (1.f / D)) * fg * invl);
          } else {
            dgp[j] = run;
          }
        }
        if (!pcd) {  // one decay per head: dg_t = sum_i dG-suffix + 2 alpha_t^2 da_t
          const float rs2 = rs16(dgp, lane);
          if ((lane & 1) == 0) s_red2[wq * 64 + t0 + (lane >> 1)] = rs2;
          __syncthreads();
          if (tid < CM) {
            const int tt = c * CM + tid;
            if (tt < a.T) {
              const float al = __expf(s_gs[tid]);
              const float dg = (s_red2[tid] + s_red2[64 + tid]) + (s_red2[128 + tid] + s_red2[192 + tid]) +
                               2.f * al * al * s_da[tid];
              const float fg = G ? -expm1f(s_gs[tid]) : 1.f;  // d log alpha / dx
              st_grad<OBF>(a.dg, tok_index(a, b, tt, h), dg * fg * invl);
            }
          }
        }
      }
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
  }

  if (ok) {
    if (a.dS0) {
      const int i = 32 * wq + lane;
      for (int c0 = 0; c0 < 32; c0 += 16) {
        float v[16];
        const int j0 = 32 * wg + c0;
        tmem_ld16(TS + lane_base + j0, v);
        float4 *dst = reinterpret_cast<float4 *>(a.dS0 + ((size_t)bh * D + i) * D + j0);
#pragma unroll
        for (int u = 0; u < 4; ++u)
          dst[u] = make_float4(v[4 * u] * invl, v[4 * u + 1] * invl, v[4 * u + 2] * invl, v[4 * u + 3] * invl);
      }
    }
    if (a.dp0 && tid < D) {
      if (V == 0) a.dp0[(size_t)bh * D + tid] = s_dp[tid] * invl;
      else if (tid == 0) a.dp0[bh] = s_dp[0] * invl;
    }
    if (a.dmu && tid == 0) {  // dL/dmu of this sequence: the warps' parts
      float tot = 0.f;
      for (int w = 0; w < CM; ++w) tot += s_dmu[w];
      a.dmu[bh] = tot * invl;
    }
    if (DVT && tid == 32) bulk_wait_all();  // the last chunk's dv stores
  } else {
    if (tid == 0) atomicExch(a.status, (unsigned)KDN_ERR_TIMEOUT);
    if (DVT && tid == 32) bulk_wait_all();
    // let copies already in flight land before the CTA's shared memory goes away
    if (tid == 0) {
      mbar_wait(bar_a, 0, kWaitIters);
      mbar_wait(bar_a, 1, kWaitIters);
      mbar_wait(bar_b, 0, kWaitIters);
      mbar_wait(bar_b, 1, kWaitIters);
      if (WT) {
        mbar_wait(bar_w, 0, kWaitIters);
        mbar_wait(bar_w, 1, kWaitIters);
      }
      if (V == 0) {
        mbar_wait(bar_g, 0, kWaitIters);
        mbar_wait(bar_g, 1, kWaitIters);
      }
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 0) tmem_dealloc(tb, 512);
}

}  // namespace

bool fused_bwd_supported(const Args &a) { return a.chunk != 32 && fused_fwd_supported(a); }

size_t fused_saved_bytes(const Args &a) {
  if (!fused_bwd_supported(a)) return 0;
  const size_t nc = (a.T + CM - 1) / CM;
  return (size_t)a.B * a.H * nc * (kCtxBytes + D * sizeof(float));
}

size_t fused_ctx_record_bytes() { return kCtxBytes; }

kdn_status_t launch_fused_bwd_sweep(const Args &a, cudaStream_t s) {
  if (split_bwd_supported(a)) return launch_split_bwd(a, a.T % CM == 0 ? nullptr : a.split_ws, s);
  BwdParams P;
  P.a = a;
  CUtensorMap mq, mk, mv, mdo;
  if (!make_map(&mq, a.q, a) || !make_map(&mk, a.k, a) || !make_map(&mv, a.v, a) ||
      !make_map(&mdo, a.dO, a))
    return KDN_ERR_CUDA;
  CUtensorMap mw = mq;  // the omega logits (diagonal KDN, logit gates)
  if (a.variant == 0 && a.gates && !make_map(&mw, a.omega, a))
    return KDN_ERR_CUDA;
  const bool obf = a.odt == KDN_BF16;
  CUtensorMap mdv = mq;  // dv (bf16 gradients: TMA stores)
  if (obf && !make_map(&mdv, a.dv_, a))
    return KDN_ERR_CUDA;
  decltype(&k_fused_bwd<0, 0, 0, 0>) kern;
  if (a.variant == 0)
    kern = a.gates ? (obf ? k_fused_bwd<0, 1, 1, 0> : k_fused_bwd<0, 0, 1, 0>)
                   : (obf ? k_fused_bwd<0, 1, 0, 0> : k_fused_bwd<0, 0, 0, 0>);
  else if (a.pcd)
    kern = a.gates ? (obf ? k_fused_bwd<1, 1, 1, 0> : k_fused_bwd<1, 0, 1, 0>)
                   : (obf ? k_fused_bwd<1, 1, 0, 0> : k_fused_bwd<1, 0, 0, 0>);
  else
    kern = a.gates ? (obf ? k_fused_bwd<1, 1, 1, 1> : k_fused_bwd<1, 0, 1, 1>)
                   : (obf ? k_fused_bwd<1, 1, 0, 1> : k_fused_bwd<1, 0, 0, 1>);
  if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, SMEM_BYTES) !=
      cudaSuccess)
    return KDN_ERR_CUDA;
  kern<<<a.B * a.H, BT, SMEM_BYTES, s>>>(mq, mk, mv, mdo, mw, mdv, P);
  return cudaGetLastError() == cudaSuccess ? KDN_OK : KDN_ERR_CUDA;
}

kdn_status_t launch_fused_bwd(const Args &a, cudaStream_t s) {
  // context-saving forward pass (o, S_T, p_T are not written)
  Args f = a;
  f.o = nullptr;
  f.ST = nullptr;
  f.pT = nullptr;
  // (the diagonal sweep reads Y = V - Kbar S_in from the context, which the WY forward writes)
  if (a.variant == 0 && !wy_fwd_supported(f)) return KDN_ERR_UNSUPPORTED;
  kdn_status_t st = wy_fwd_supported(f) ? launch_wy_fwd(f, s, a.fSin, a.fpin)
                                         : launch_fused_fwd(f, s, a.fSin, a.fpin, false);
  if (st != KDN_OK) return st;
  return launch_fused_bwd_sweep(a, s);
}

}  // namespace kdn
