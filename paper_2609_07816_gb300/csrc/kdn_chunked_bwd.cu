// kdn_chunked_bwd.cu -- general chunked backward of the Diagonal and Isotropic KDN
// on CUDA cores (float32 arithmetic, any dk, dv in {32,64,128}, float32 or
// bfloat16 activations).  The forward (kdn_chunked_fwd.cu) runs first and keeps
// its factors; then
//   k_state_bwd    carries the memory cotangent dS backwards over chunks;
//   k_chunk_bwd    forms every chunk-local adjoint, in parallel over chunks, and the
//                  chunk's summary of the uncertainty adjoint (dp_in = A dp_out + B);
//   k_dp_scan      chains the summaries backwards;
//   k_gain_bwd_*   runs the adjoint of the uncertainty recursion inside every chunk,
//                  in parallel over chunks, and writes the gradients that need it;
//   k_dmu_sum      adds up the chunks' parts of dmu, where that is asked for.
#include "kdn_chunked.cuh"

namespace kdn {
namespace {

constexpr int SB = 32;  // value columns per pass of k_chunk_bwd

// dR = A_qk^T dO + K_tail dS_out,  dS_in = Qbar^T dO + diag(gamma_C) dS_out - W^T dR
template <typename DT, int DK, int CW, int TM>
__global__ void __launch_bounds__(StateCfg<DK, CW, TM>::NTH) k_state_bwd(Args a) {
  using Cfg = StateCfg<DK, CW, TM>;
  constexpr int LD = Cfg::LD, LS = Cfg::LS, RS = Cfg::RS, TH = TM / 2;
  extern __shared__ __align__(16) float sm[];
  float *sS = sm + 2 * Cfg::FLOATS, *sdR = sS + DK * LS;
  const int ns = a.dv / CW, bh = (int)(blockIdx.x / (unsigned)ns), j0 = (int)(blockIdx.x % (unsigned)ns) * CW;
  const int tid = KDN_TID, dv = a.dv;
  const int col = 4 * (tid % (CW / 4)), ga = tid / (CW / 4), i0 = RS * ga, r0 = TH * ga;
  const size_t sbase = ((size_t)bh * DK + i0) * dv + j0 + col;
  float S[RS][4];
#pragma unroll
  for (int m = 0; m < RS; ++m) {
#pragma unroll
    for (int n = 0; n < 4; ++n) S[m][n] = 0.f;
    if (a.dST) ld4<float>(a.dST + sbase + (size_t)m * dv, 0, S[m]);
    st4(sS + (i0 + m) * LS + col, S[m]);
  }
  issue_chunk_factors<Cfg, DK, CW>(a, bh, a.NC - 1, sm + ((a.NC - 1) & 1) * Cfg::FLOATS, j0, true);
  cp_commit();
  for (int c = a.NC - 1; c >= 0; --c) {
    const float *buf = sm + (c & 1) * Cfg::FLOATS;
    cp_wait<0>();
    __syncthreads();
    if (c > 0) issue_chunk_factors<Cfg, DK, CW>(a, bh, c - 1, sm + ((c - 1) & 1) * Cfg::FLOATS, j0, true);
    cp_commit();
    const float *sW = buf, *sQ = sW + CC * LD, *sKt = sQ + CC * LD, *sAqk = sKt + CC * LD;
    const float *sgC = sAqk + CC * LC, *sdO = sgC + DK;
    const size_t base = (size_t)bh * a.NC + c;
    // four columns of dO row r (rows LS floats apart, activation dtype)
    auto dO = [&](int r, float *v) { ld4<DT>(reinterpret_cast<const DT *>(sdO + r * LS), col, v); };
#pragma unroll
    for (int m = 0; m < RS; ++m) st4(a.dSout + (base * DK + i0 + m) * dv + j0 + col, S[m]);
    float acc[TH][4];
    zero<TH>(acc);
    for (int s2 = r0; s2 < CC; ++s2) {  // A_qk is zero above its diagonal
      float d[4];
      dO(s2, d);
#pragma unroll
      for (int m = 0; m < TH; ++m)
#pragma unroll
        for (int n = 0; n < 4; ++n) acc[m][n] = fmaf(sAqk[s2 * LC + r0 + m], d[n], acc[m][n]);
    }
    tile_mm2<DK, TH>(acc, sKt + r0 * LD, LD, sS + col, LS);
#pragma unroll
    for (int m = 0; m < TH; ++m) {
      st4(sdR + (r0 + m) * LS + col, acc[m]);
      st4(a.dR + (base * CC + r0 + m) * dv + j0 + col, acc[m]);
    }
    __syncthreads();
    float inc[2][RS][4];  // the chunk's part first, in halves, so that S is rounded once
#pragma unroll
    for (int hf = 0; hf < 2; ++hf) {
      zero<RS>(inc[hf]);
#pragma unroll 4
      for (int r = hf * (CC / 2); r < (hf + 1) * (CC / 2); ++r) {
        float d[4], e[4];
        dO(r, d);
        ld4<float>(sdR + r * LS, col, e);
#pragma unroll
        for (int m = 0; m < RS; ++m) {
          const float qv = sQ[r * LD + i0 + m], wv = sW[r * LD + i0 + m];
#pragma unroll
          for (int n = 0; n < 4; ++n) inc[hf][m][n] = fmaf(qv, d[n], fmaf(-wv, e[n], inc[hf][m][n]));
        }
      }
    }
#pragma unroll
    for (int m = 0; m < RS; ++m) {
      const float g = sgC[i0 + m];
#pragma unroll
      for (int n = 0; n < 4; ++n) S[m][n] = fmaf(g, S[m][n], inc[0][m][n] + inc[1][m][n]);
      st4(sS + (i0 + m) * LS + col, S[m]);
    }
  }
  if (a.dS0) {
#pragma unroll
    for (int m = 0; m < RS; ++m) st4(a.dS0 + sbase + (size_t)m * dv, S[m]);
  }
}

// ---------------------------------------------------------------------------
// Chunk-local adjoints, in parallel over chunks.  Three groups of threads hold the
// 32 x dk accumulators dQbar, dK_tail (then dKk) and dW (then dKbar) in registers
// over the passes through the value columns; a thread's tile is rows ga + 8 m and
// four adjacent columns.  The 32 x 32 matrices that enter transposed are stored both
// ways, so that every left operand is read 16 bytes along k.

template <int DK>
struct BwdCfg {
  static constexpr int LD = DK + 4;
  static constexpr int GT = DK >= 64 ? 128 : 64;     // threads per group
  static constexpr int NTH = 3 * GT, NTL = 2 * DK / GT;  // threads, tiles per thread
  static constexpr int SLICE = 2 * DK * LC + 4 * CC * LC, SMALL = 6 * CC * LC;
  static constexpr int POOL = SLICE > SMALL ? SLICE : SMALL;
  static constexpr int FLOATS = 7 * CC * LD + 2 * CC * LC + POOL + 4 * CC + 2 * DK;
  static constexpr size_t SMEM = sizeof(float) * FLOATS;
};

template <int V, typename DT, int DK>
__global__ void __launch_bounds__(BwdCfg<DK>::NTH) k_chunk_bwd(Args a) {
  using Cfg = BwdCfg<DK>;
  constexpr int LD = Cfg::LD, GT = Cfg::GT, NTH = Cfg::NTH, NTL = Cfg::NTL;
  extern __shared__ __align__(16) float sm[];
  float *sK = sm, *sQ = sK + CC * LD, *sKk = sQ + CC * LD, *sGa = sKk + CC * LD;
  float *sdW = sGa + CC * LD, *sdQ = sdW + CC * LD, *sdKk = sdQ + CC * LD;
  float *sA = sdKk + CC * LD, *sAt = sA + CC * LC, *pool = sAt + CC * LC;
  // tenants of the pool: the value-column slices, then the small matrices
  float *sSin = pool, *sdSo = sSin + DK * LC, *sR = sdSo + DK * LC, *sdR = sR + CC * LC;
  float *sdO = sdR + CC * LC, *sV = sdO + CC * LC;
  float *sdAqk = pool, *sdAqkT = sdAqk + CC * LC, *sdA = sdAqkT + CC * LC, *sX = sdA + CC * LC;
  float *sdT = sX + CC * LC, *sdTt = sdT + CC * LC;
  float *s_s = pool + Cfg::POOL, *s_r = s_s + CC, *s_x = s_r + CC, *s_n2 = s_x + CC, *s_gC = s_n2 + CC;
  float *s_dgc = s_gC + DK;
  const int tid = KDN_TID, lane = tid & 31, warp = tid >> 5;
  const int bh = (int)(blockIdx.x / (unsigned)a.NC), c = (int)(blockIdx.x % (unsigned)a.NC);
  const int b = bh / a.H, h = bh % a.H, dv = a.dv, tn = min(CC, a.T - c * CC);
  const size_t base = (size_t)bh * a.NC + c, row0 = (size_t)bh * a.Tp + c * CC;

  if (tid < CC) {
    s_s[tid] = a.stok[row0 + tid];
    s_r[tid] = tid < tn ? gate_r(a.gates, a.rmin, ld<DT>(a.r, tok_index(a, b, c * CC + tid, h))) : 1.f;
    if (V == 1) s_n2[tid] = a.isotok[(row0 + tid) * 2 + 1];
  }
  for (int e = tid; e < CC * (CC / 4); e += NTH) {
    const int r = e >> 3, q = 4 * (e & 7);
    float x[4];
    ld4<float>(a.Ainv + base * CC * CC, 4 * e, x);
    st4(sA + r * LC + q, x);
#pragma unroll
    for (int u = 0; u < 4; ++u) sAt[(q + u) * LC + r] = x[u];
  }
  __syncthreads();
  for (int e = tid; e < CC * (DK / 4); e += NTH) {
    const int t = e / (DK / 4), i4 = 4 * (e % (DK / 4));
    float kx[4] = {0.f, 0.f, 0.f, 0.f}, gx[4], px[4], x[4];
    if (t < tn) ld4<DT>(a.k, tok_index(a, b, c * CC + t, h) * DK + i4, kx);
    ld4<float>(a.gam + (row0 + t) * DK, i4, gx);
    ld4<float>(a.Qb + (base * CC + t) * DK, i4, x);
    st4(sQ + t * LD + i4, x);
    st4(sGa + t * LD + i4, gx);
    if (V == 0) ld4<float>(a.phat + (row0 + t) * DK, i4, px);
    const float f = s_s[t];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      x[u] = kx[u] * gx[u];
      px[u] = V == 0 ? px[u] * kx[u] / f / gx[u] : f * kx[u] / gx[u];
    }
    st4(sK + t * LD + i4, x);
    st4(sKk + t * LD + i4, px);
    if (t == CC - 1) st4(s_gC + i4, gx);
  }

  const int grp = tid / GT, tl = tid % GT;
  const int ga = lane >> 2, gb = (lane & 3) + 4 * (tl >> 5);  // tile rows ga + 8 m, columns 4 gb (+ 4 (GT / 8) l)
  constexpr int CS = GT / 2;  // columns between a thread's tiles
  float acc[NTL][4][4], am[4][4], dgc = 0.f;
#pragma unroll
  for (int l = 0; l < NTL; ++l) zero<4>(acc[l]);
  zero<4>(am);
  const int mg = 4 * ((lane & 3) + 4 * (warp & 1));  // column of the 32 x 32 (and 32 x SB) tiles
  for (int j0 = 0; j0 < dv; j0 += SB) {
    __syncthreads();
    for (int e = tid; e < DK * (SB / 4); e += NTH) {
      const int i = e >> 3, q = 4 * (e & 7);
      float x[4];
      ld4<float>(a.Sin + (base * DK + i) * dv + j0, q, x);
      st4(sSin + i * LC + q, x);
      ld4<float>(a.dSout + (base * DK + i) * dv + j0, q, x);
      st4(sdSo + i * LC + q, x);
    }
    for (int e = tid; e < CC * (SB / 4); e += NTH) {
      const int r = e >> 3, q = 4 * (e & 7);
      float x[4], y[4] = {0.f, 0.f, 0.f, 0.f}, z[4] = {0.f, 0.f, 0.f, 0.f};
      ld4<float>(a.R + (base * CC + r) * dv + j0, q, x);
      st4(sR + r * LC + q, x);
      ld4<float>(a.dR + (base * CC + r) * dv + j0, q, x);
      st4(sdR + r * LC + q, x);
      if (r < tn) {
        const size_t th = tok_index(a, b, c * CC + r, h);
        ld4<DT>(a.dO, th * dv + j0 + q, y);
        ld4<DT>(a.v, th * dv + j0 + q, z);
      }
      st4(sdO + r * LC + q, y);
      st4(sV + r * LC + q, z);
    }
    __syncthreads();
    // dQbar += dO S_in^T; dK_tail += R dS_out^T; -dW += dR S_in^T
    const float *lft = grp == 0 ? sdO : grp == 1 ? sR : sdR, *rgt = grp == 1 ? sdSo : sSin;
#pragma unroll
    for (int l = 0; l < NTL; ++l)
      tile_mm<SB, 4, true>(acc[l], lft + ga * LC, 8 * LC, rgt + (4 * gb + l * CS) * LC, LC);
    if (warp < 2) {         // dA_qk += dO R^T
      tile_mm<SB, 4, true>(am, sdO + ga * LC, 8 * LC, sR + mg * LC, LC);
    } else if (warp < 4) {  // dA += dR V^T
      tile_mm<SB, 4, true>(am, sdR + ga * LC, 8 * LC, sV + mg * LC, LC);
    } else if (warp < 6) {  // dV = A^T dR
      float x[4][4];
      zero<4>(x);
      tile_mm<CC, 4, false>(x, sAt + ga * LC, 8 * LC, sdR + mg, LC);
#pragma unroll
      for (int m = 0; m < 4; ++m) {
        const int tt = c * CC + ga + 8 * m;
        if (tt < a.T) sto4(a.odt, a.dv_, tok_index(a, b, tt, h) * dv + j0 + mg, x[m]);
      }
    }
    if (tid >= NTH - DK) {  // dgamma_C += rowsum(dS_out (.) S_in)
      const int i = tid - (NTH - DK);
#pragma unroll
      for (int q = 0; q < SB; q += 4) {
        float x[4], y[4];
        ld4<float>(sdSo + i * LC, q, x);
        ld4<float>(sSin + i * LC, q, y);
#pragma unroll
        for (int u = 0; u < 4; ++u) dgc = fmaf(x[u], y[u], dgc);
      }
    }
  }
  __syncthreads();
  if (tid >= NTH - DK) s_dgc[tid - (NTH - DK)] = dgc;
  if (warp < 2) {
#pragma unroll
    for (int m = 0; m < 4; ++m) {
      const int r = ga + 8 * m;
#pragma unroll
      for (int n = 0; n < 4; ++n) {
        const float x = mg + n <= r ? am[m][n] : 0.f;
        sdAqk[r * LC + mg + n] = x;
        sdAqkT[(mg + n) * LC + r] = x;
      }
    }
  }
  if (grp == 2) {
#pragma unroll
    for (int l = 0; l < NTL; ++l)
#pragma unroll
      for (int m = 0; m < 4; ++m) {
#pragma unroll
        for (int n = 0; n < 4; ++n) acc[l][m][n] = -acc[l][m][n];
        st4(sdW + (ga + 8 * m) * LD + 4 * gb + l * CS, acc[l][m]);
      }
  }
  __syncthreads();
  if (warp >= 2 && warp < 4) {  // dA += dW Kbar^T
    tile_mm<DK, 4, true>(am, sdW + ga * LD, 8 * LD, sK + mg * LD, LD);
#pragma unroll
    for (int m = 0; m < 4; ++m) st4(sdA + (ga + 8 * m) * LC + mg, am[m]);
  }
#pragma unroll
  for (int l = 0; l < NTL; ++l) {
    const int col = 4 * gb + l * CS;
    if (grp == 0) {  // dQbar += dA_qk Kk
      tile_mm<CC, 4, false>(acc[l], sdAqk + ga * LC, 8 * LC, sKk + col, LD);
    } else if (grp == 1) {  // dgamma_C += colsum(dK_tail (.) Kk); dKk = gamma_C dK_tail + dA_qk^T Qbar
      float cs[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
      for (int m = 0; m < 4; ++m) {
        float y[4];
        ld4<float>(sKk + (ga + 8 * m) * LD, col, y);
#pragma unroll
        for (int n = 0; n < 4; ++n) {
          cs[n] = fmaf(acc[l][m][n], y[n], cs[n]);
          acc[l][m][n] *= s_gC[col + n];
        }
      }
#pragma unroll
      for (int n = 0; n < 4; ++n) {
#pragma unroll
        for (int o = 4; o < 32; o <<= 1) cs[n] += __shfl_xor_sync(0xffffffffu, cs[n], o);
        if (lane < 4) s_dgc[col + n] += cs[n];
      }
      tile_mm<CC, 4, false>(acc[l], sdAqkT + ga * LC, 8 * LC, sQ + col, LD);
    } else {  // dKbar = A^T dW
      zero<4>(acc[l]);
      tile_mm<CC, 4, false>(acc[l], sAt + ga * LC, 8 * LC, sdW + col, LD);
    }
  }
  __syncthreads();
  if (warp < 2) {  // X = A^T dA
    zero<4>(am);
    tile_mm<CC, 4, false>(am, sAt + ga * LC, 8 * LC, sdA + mg, LC);
#pragma unroll
    for (int m = 0; m < 4; ++m) st4(sX + (ga + 8 * m) * LC + mg, am[m]);
  }
  __syncthreads();
  if (warp < 2) {  // dT = strict lower part of -X A^T
    zero<4>(am);
    tile_mm<CC, 4, true>(am, sX + ga * LC, 8 * LC, sA + mg * LC, LC);
#pragma unroll
    for (int m = 0; m < 4; ++m) {
      const int r = ga + 8 * m;
#pragma unroll
      for (int n = 0; n < 4; ++n) {
        const float x = mg + n < r ? -am[m][n] : 0.f;
        sdT[r * LC + mg + n] = x;
        sdTt[(mg + n) * LC + r] = x;
      }
    }
  }
  __syncthreads();
  // dKbar += dT Kk; dKk += dT^T Kbar; the three adjoints to shared memory
#pragma unroll
  for (int l = 0; l < NTL; ++l) {
    const int col = 4 * gb + l * CS;
    if (grp == 2) tile_mm<CC, 4, false>(acc[l], sdT + ga * LC, 8 * LC, sKk + col, LD);
    if (grp == 1) tile_mm<CC, 4, false>(acc[l], sdTt + ga * LC, 8 * LC, sK + col, LD);
    float *dst = grp == 0 ? sdQ : grp == 1 ? sdKk : sdW;
#pragma unroll
    for (int m = 0; m < 4; ++m) st4(dst + (ga + 8 * m) * LD + col, acc[l][m]);
  }
  __syncthreads();
  // Back through the scaling by gamma = exp(G): dq, the key/gain cotangents, and dG (into sdQ).
  for (int e = tid; e < CC * (DK / 4); e += NTH) {
    const int t = e / (DK / 4), i4 = 4 * (e % (DK / 4)), o = t * LD + i4;
    float gam[4], dKb[4], dKx[4], dQb[4], kb[4], kk[4], qb[4], dq[4], kx[4] = {0.f, 0.f, 0.f, 0.f}, px[4];
    if (t < tn) ld4<DT>(a.k, tok_index(a, b, c * CC + t, h) * DK + i4, kx);
    if (V == 0) ld4<float>(a.phat + (row0 + t) * DK, i4, px);
    ld4<float>(sGa, o, gam);
    ld4<float>(sdW, o, dKb);
    ld4<float>(sdKk, o, dKx);
    ld4<float>(sdQ, o, dQb);
    ld4<float>(sK, o, kb);
    ld4<float>(sKk, o, kk);
    ld4<float>(sQ, o, qb);
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      float dG = dKb[u] * kb[u] - dKx[u] * kk[u] + dQb[u] * qb[u];
      if (t == CC - 1) dG += s_dgc[i4 + u] * s_gC[i4 + u];
      dq[u] = a.tau * dQb[u] * gam[u];
      dQb[u] = dG;
      dKb[u] *= gam[u];  // dK from the memory path
      dKx[u] /= gam[u];  // d kappa
      kk[u] *= gam[u];   // kappa
    }
    if (t < tn) sto4(a.odt, a.dq, tok_index(a, b, c * CC + t, h) * DK + i4, dq);
    st4(sdQ + o, dQb);
    st4(sdW + o, dKb);
    st4(sdKk + o, dKx);
    st4(sKk + o, kk);
    st4(sGa + o, kx);  // k and phat for the gain adjoint, over tiles that are dead now
    if (V == 0) st4(sQ + o, px);
  }
  float gvv[CC];  // the decay inputs of this thread's channel, loaded ahead of the chunk's summary
  if (V == 0 && tid < DK) {
#pragma unroll
    for (int t = 0; t < CC; ++t)
      gvv[t] = t < tn ? ld<DT>(a.g, tok_index(a, b, c * CC + t, h) * DK + tid) : 0.f;
  }
  __syncthreads();
  // reverse cumulative sum over the chunk: dg_j = sum_{r >= j} dG_r
  if (tid < DK) {
    float acc2 = 0.f;
#pragma unroll 8
    for (int t = CC - 1; t >= 0; --t) {
      acc2 += sdQ[t * LD + tid];
      a.dgpart[(row0 + t) * DK + tid] = acc2;
    }
  }
  // local part of the gain adjoint, one warp per token
  for (int t = warp; t < CC; t += NTH / 32) {
    const size_t row = row0 + t;
    const float rr = s_r[t];
    float kv[DK / 32];
#pragma unroll
    for (int m = 0; m < DK / 32; ++m)
      kv[m] = sGa[t * LD + lane + 32 * m];
    float part = 0.f;
#pragma unroll
    for (int m = 0; m < DK / 32; ++m) {
      const int i = lane + 32 * m;
      part = fmaf(sdKk[t * LD + i], V == 0 ? sKk[t * LD + i] : kv[m], part);
    }
    if (V == 0) {
      const float s = s_s[t], ds = -warp_sum(part) / s;
#pragma unroll
      for (int m = 0; m < DK / 32; ++m) {
        const int i = lane + 32 * m;
        const float dkap = sdKk[t * LD + i], ph = sQ[t * LD + i];
        const float dphl = dkap * kv[m] / s + ds * kv[m] * kv[m];
        a.dphloc[row * DK + i] = dphl;
        a.dkpart[row * DK + i] = sdW[t * LD + i] + dkap * ph / s + 2.f * ds * ph * kv[m];
        sdKk[t * LD + i] = dphl;  // for the summary below: dphat, 1 / (1 + u phat)
        sKk[t * LD + i] = 1.f / (1.f + a.mu * kv[m] * kv[m] / rr * ph);
      }
      if (lane == 0) a.drpart[row] = ds;
    } else {
      const float dbeta = warp_sum(part), beta = s_s[t], bhat = a.phat[row];
      const float den = rr + bhat * s_n2[t], dn2 = -dbeta * beta * beta;
#pragma unroll
      for (int m = 0; m < DK / 32; ++m) {
        const int i = lane + 32 * m;
        a.dkpart[row * DK + i] = sdW[t * LD + i] + beta * sdKk[t * LD + i] + 2.f * kv[m] * dn2;
      }
      if (lane == 0) {
        const float dphl = dbeta * rr / (den * den);
        a.dphloc[row] = dphl;
        a.drpart[row] = -dbeta * beta / den;
        s_x[t] = dphl;
      }
    }
  }
  __syncthreads();
  // the chunk's summary of the uncertainty adjoint, dp_{t-1} = a_t (dp_t / den_t^2 + dphat_t)
  if (V == 0) {
    if (tid < DK) {
      float A = 1.f, Bv = 0.f;
#pragma unroll
      for (int t = CC - 1; t >= 0; --t) {
        const float lg = t < tn ? gate_logalpha(a.gates, gvv[t]) : 0.f;
        const float al2 = expf(2.f * lg), rd = sKk[t * LD + tid], f = al2 * rd * rd;
        Bv = fmaf(f, Bv, al2 * sdKk[t * LD + tid]);
        A *= f;
      }
      reinterpret_cast<float2 *>(a.aff)[base * DK + tid] = make_float2(A, Bv);
    }
  } else if (warp == 0) {
    const float aa = a.isotok[(row0 + lane) * 2], bhat = a.phat[row0 + lane];
    const float rd = 1.f / (1.f + a.mu * s_n2[lane] / (DK * s_r[lane]) * bhat);
    float A = aa * rd * rd, Bv = aa * s_x[lane];
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
      const float pA = __shfl_down_sync(0xffffffffu, A, off), pB = __shfl_down_sync(0xffffffffu, Bv, off);
      if (lane + off < 32) {
        Bv = fmaf(A, pB, Bv);
        A *= pA;
      }
    }
    if (lane == 0) reinterpret_cast<float2 *>(a.aff)[base] = make_float2(A, Bv);
  }
}

// ---------------------------------------------------------------------------
// Adjoint of the uncertainty recursion, backwards in time.

// One thread per (sequence, channel): the cotangent of p leaving every chunk.
__global__ void __launch_bounds__(128) k_dp_scan(Args a) {
  const size_t e = blockIdx.x * (size_t)128 + KDN_TID, n = (size_t)a.B * a.H * a.P;
  if (e >= n) return;
  const size_t bh = e / a.P, i = e % a.P, o = bh * a.NC * a.P + i;
  float dp = a.dpT ? a.dpT[e] : 0.f;
  const float2 *af = reinterpret_cast<const float2 *>(a.aff) + o;
  for (int c0 = a.NC - 1; c0 >= 0; c0 -= 8) {
    float2 x[8];
#pragma unroll
    for (int u = 0; u < 8; ++u)
      if (c0 - u >= 0) x[u] = af[(size_t)(c0 - u) * a.P];
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      if (c0 - u >= 0) {
        a.dpout[o + (size_t)(c0 - u) * a.P] = dp;
        dp = fmaf(x[u].x, dp, x[u].y);
      }
    }
  }
  if (a.dp0) a.dp0[e] = dp;
}

// A chunk's part of dmu, in its summary's place (which k_dp_scan has read).
__device__ __forceinline__ float *dmu_part(const Args &a, size_t chunk) { return a.aff + chunk * a.P * 2; }

// One warp per sequence: dmu, its chunks' parts in an order of their own, so that it repeats exactly.
__global__ void __launch_bounds__(32) k_dmu_sum(Args a) {
  const size_t base = (size_t)blockIdx.x * a.NC;
  float s = 0.f;
  for (int c = KDN_TID; c < a.NC; c += 32) s += *dmu_part(a, base + c);
  s = warp_sum(s);
  if (KDN_TID == 0) a.dmu[blockIdx.x] = s;
}

// One CTA per chunk, one thread per channel, eight tokens loaded at a time.
template <typename DT, int DK>
__global__ void __launch_bounds__(DK) k_gain_bwd_diag(Args a) {
  __shared__ float s_r[CC], s_dr[CC][DK / 32], s_mu[DK / 32];
  const int i = KDN_TID, lane = i & 31, warp = i >> 5;
  const int bh = (int)(blockIdx.x / (unsigned)a.NC), c = (int)(blockIdx.x % (unsigned)a.NC);
  const int b = bh / a.H, h = bh % a.H, tn = min(CC, a.T - c * CC);
  const size_t base = (size_t)bh * a.NC + c, row0 = (size_t)bh * a.Tp + c * CC;
  if (i < CC)
    s_r[i] = i < tn ? gate_r(a.gates, a.rmin, ld<DT>(a.r, tok_index(a, b, c * CC + i, h))) : 1.f;
  float dp = a.dpout[base * DK + i], dmu = 0.f;
  const float p_in = a.pin[base * DK + i];
  __syncthreads();
  // phat, k of the token before the block (its p is the block's entry uncertainty)
  for (int t0 = ((tn - 1) / 8) * 8; t0 >= 0; t0 -= 8) {
    float ph[8], kv[8], lg[8], dl[8], dk[8], dg[8], wl[8];
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      const int t = min(t0 + j, tn - 1);
      const size_t th = tok_index(a, b, c * CC + t, h) * DK + i, row = (row0 + t) * DK + i;
      ph[j] = a.phat[row];
      kv[j] = ld<DT>(a.k, th);
      lg[j] = ld<DT>(a.g, th);
      dl[j] = a.dphloc[row];
      dk[j] = a.dkpart[row];
      dg[j] = a.dgpart[row];
      wl[j] = a.gates ? ld<DT>(a.omega, th) : 0.f;
    }
    float pprev = p_in;
    if (t0 > 0) {
      const float pb = a.phat[(row0 + t0 - 1) * DK + i];
      const float kb = ld<DT>(a.k, tok_index(a, b, c * CC + t0 - 1, h) * DK + i);
      pprev = pb / (1.f + a.mu * kb * kb / s_r[t0 - 1] * pb);
    }
    float pt[8];
#pragma unroll
    for (int j = 0; j < 8; ++j) pt[j] = ph[j] / (1.f + a.mu * kv[j] * kv[j] / s_r[min(t0 + j, CC - 1)] * ph[j]);
#pragma unroll
    for (int j = 7; j >= 0; --j) {
      const int t = t0 + j;
      if (t >= tn) continue;  // (uniform over the CTA)
      const size_t th = tok_index(a, b, c * CC + t, h) * DK + i;
      const float rr = s_r[t], u = a.mu * kv[j] * kv[j] / rr, den = 1.f + u * ph[j];
      const float dph = dp / (den * den) + dl[j];
      const float du = -dp * pt[j] * pt[j];
      dmu += du * kv[j] * kv[j] / rr;  // u = mu k^2 / r
      const float drp = warp_sum(-du * u / rr);
      if (lane == 0) s_dr[t][warp] = drp;
      const float pp = j > 0 ? pt[j - 1] : pprev;
      const float la = gate_logalpha(a.gates, lg[j]), al2 = expf(2.f * la);
      // logit gates: d omega / dy = sigmoid(y), d log alpha / dx = 1 - alpha
      const float fw = a.gates ? sigmoid_f(wl[j]) : 1.f;
      const float fg = a.gates ? -expm1f(la) : 1.f;
      sto(a.odt, a.domega, th, dph * fw);
      sto(a.odt, a.dg, th, (dg[j] + 2.f * al2 * pp * dph) * fg);
      sto(a.odt, a.dk_, th, dk[j] + du * 2.f * a.mu * kv[j] / rr);
      dp = al2 * dph;
    }
  }
  if (a.dmu) {
    dmu = warp_sum(dmu);
    if (lane == 0) s_mu[warp] = dmu;
  }
  __syncthreads();
  if (i < tn) {
    float acc = a.drpart[row0 + i];
#pragma unroll
    for (int w = 0; w < DK / 32; ++w) acc += s_dr[i][w];
    const size_t th = tok_index(a, b, c * CC + i, h);
    if (a.gates) acc *= sigmoid_f(ld<DT>(a.r, th));  // d r / dz
    sto(a.odt, a.dr, th, acc);
  }
  if (a.dmu && i == 0) {
    float tot = 0.f;
#pragma unroll
    for (int w = 0; w < DK / 32; ++w) tot += s_mu[w];
    *dmu_part(a, base) = tot;
  }
}

// One CTA per chunk: warp 0 runs the scalar recursion (one token a lane, the affine
// maps composed by shuffles), then every thread finishes dk and dg.
template <typename DT, int DK>
__global__ void __launch_bounds__(128) k_gain_bwd_iso(Args a) {
  __shared__ float s_dn2[CC], s_da[CC], s_dg[CC];
  const int tid = KDN_TID, lane = tid & 31, warp = tid >> 5;
  const int bh = (int)(blockIdx.x / (unsigned)a.NC), c = (int)(blockIdx.x % (unsigned)a.NC);
  const int b = bh / a.H, h = bh % a.H, tn = min(CC, a.T - c * CC);
  const size_t base = (size_t)bh * a.NC + c, row0 = (size_t)bh * a.Tp + c * CC;
  if (warp == 0) {
    const size_t th = tok_index(a, b, c * CC + min(lane, tn - 1), h);
    const float aa = a.isotok[(row0 + lane) * 2], n2 = a.isotok[(row0 + lane) * 2 + 1];
    const float rr = lane < tn ? gate_r(a.gates, a.rmin, ld<DT>(a.r, th)) : 1.f;
    const float bhat = lane < tn ? a.phat[row0 + lane] : 0.f;
    const float dl = lane < tn ? a.dphloc[row0 + lane] : 0.f;
    const float u = a.mu * n2 / (DK * rr), den = 1.f + u * bhat, bt = bhat / den;
    float A = aa / (den * den), Bv = aa * dl;
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
      const float pA = __shfl_down_sync(0xffffffffu, A, off), pB = __shfl_down_sync(0xffffffffu, Bv, off);
      if (lane + off < 32) {
        Bv = fmaf(A, pB, Bv);
        A *= pA;
      }
    }
    // db_t of this lane: the later lanes' map applied to the cotangent leaving the chunk
    float eA = __shfl_down_sync(0xffffffffu, A, 1), eB = __shfl_down_sync(0xffffffffu, Bv, 1);
    const float dpo = a.dpout[base];
    const float db = lane == 31 ? dpo : fmaf(eA, dpo, eB);
    const float dbh = db / (den * den) + dl, du = -db * bt * bt;
    float bprev = __shfl_up_sync(0xffffffffu, bt, 1);
    if (lane == 0) bprev = a.pin[base];
    s_dn2[lane] = du * a.mu / (DK * rr);  // d|k|^2 through u
    s_da[lane] = bprev * dbh;             // d a_t
    if (lane < tn) {
      const float fw = a.gates ? sigmoid_f(ld<DT>(a.omega, th)) : 1.f;  // d omega / dy
      const float fr = a.gates ? sigmoid_f(ld<DT>(a.r, th)) : 1.f;      // d r / dz
      sto(a.odt, a.domega, th, dbh * fw);
      sto(a.odt, a.dr, th, (a.drpart[row0 + lane] - du * u / rr) * fr);
    }
    if (a.dmu) {
      const float dmu = warp_sum(lane < tn ? du * n2 / (DK * rr) : 0.f);  // u = mu |k|^2 / (dk r)
      if (lane == 0) *dmu_part(a, base) = dmu;
    }
  }
  __syncthreads();
  // four channels a thread; a token's DK / 4 threads lie in one warp
  for (int e = tid; e < CC * (DK / 4); e += 128) {
    const int t = e / (DK / 4), i4 = 4 * (e % (DK / 4));
    const bool live = t < tn;
    const size_t th = tok_index(a, b, c * CC + (live ? t : 0), h), row = row0 + t;
    float kv[4], dk[4], dg[4];
    ld4<DT>(a.k, th * DK + i4, kv);
    ld4<float>(a.dkpart + row * DK, i4, dk);
    ld4<float>(a.dgpart + row * DK, i4, dg);
#pragma unroll
    for (int q = 0; q < 4; ++q) dk[q] += 2.f * kv[q] * s_dn2[t];
    if (live) sto4(a.odt, a.dk_, th * DK + i4, dk);
    if (a.pcd) {
      float gv[4];
      ld4<DT>(a.g, th * DK + i4, gv);
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const float lal = gate_logalpha(a.gates, gv[q]), al2 = expf(2.f * lal);
        const float fg = a.gates ? -expm1f(lal) : 1.f;  // d log alpha / dx
        dg[q] = (dg[q] + 2.f * al2 * s_da[t] / DK) * fg;
      }
      if (live) sto4(a.odt, a.dg, th * DK + i4, dg);
    } else {
      float part = (dg[0] + dg[1]) + (dg[2] + dg[3]);
#pragma unroll
      for (int o = DK / 8; o > 0; o >>= 1) part += __shfl_xor_sync(0xffffffffu, part, o);
      if (i4 == 0) s_dg[t] = part;
    }
  }
  if (!a.pcd) {
    __syncthreads();
    if (tid < tn) {
      const size_t th = tok_index(a, b, c * CC + tid, h);
      const float lal = gate_logalpha(a.gates, ld<DT>(a.g, th)), al2 = expf(2.f * lal);
      const float fg = a.gates ? -expm1f(lal) : 1.f;  // d log alpha / dx
      sto(a.odt, a.dg, th, (s_dg[tid] + 2.f * al2 * s_da[tid]) * fg);
    }
  }
}

// ---------------------------------------------------------------------------
// Launchers

template <typename DT, int DK, int CW, int TM>
bool state_bwd(const Args &a, cudaStream_t s) {
  using Cfg = StateCfg<DK, CW, TM>;
  return launch(k_state_bwd<DT, DK, CW, TM>, (size_t)a.B * a.H * (a.dv / CW), Cfg::NTH, Cfg::SMEM, s, a);
}

template <int V, typename DT, int DK>
kdn_status_t bwd_impl(const Args &a0, cudaStream_t s) {
  Args a = a0;
  a.o = nullptr;
  a.ST = nullptr;
  a.pT = nullptr;
  kdn_status_t st0 = launch_chunked_fwd(a, s, true);
  if (st0 != KDN_OK) return st0;
  const size_t BH = (size_t)a.B * a.H, n = BH * a.NC;
  bool ok;
  switch (state_cols(a)) {
    case 64: ok = state_bwd<DT, DK, 64, 4>(a, s); break;
    case 32: ok = state_bwd<DT, DK, 32, 4>(a, s); break;
    default: ok = state_bwd<DT, DK, 16, 2>(a, s);
  }
  ok = ok && launch(k_chunk_bwd<V, DT, DK>, n, BwdCfg<DK>::NTH, BwdCfg<DK>::SMEM, s, a);
  ok = ok && launch(k_dp_scan, (BH * a.P + 127) / 128, 128, 0, s, a);
  if (V == 0) ok = ok && launch(k_gain_bwd_diag<DT, DK>, n, DK, 0, s, a);
  else ok = ok && launch(k_gain_bwd_iso<DT, DK>, n, 128, 0, s, a);
  if (a.dmu) ok = ok && launch(k_dmu_sum, BH, 32, 0, s, a);
  return ok ? KDN_OK : KDN_ERR_CUDA;
}

template <int V, typename DT>
kdn_status_t bwd_dk(const Args &a, cudaStream_t s) {
  switch (a.dk) {
    case 32: return bwd_impl<V, DT, 32>(a, s);
    case 64: return bwd_impl<V, DT, 64>(a, s);
    case 128: return bwd_impl<V, DT, 128>(a, s);
  }
  return KDN_ERR_UNSUPPORTED;
}

}  // namespace

int chunked_bwd_launches(const Args &a) { return chunked_fwd_launches(a) + 5; }

kdn_status_t launch_chunked_bwd(const Args &a, cudaStream_t s) {
  if (a.variant == 0)
    return a.dtype == KDN_BF16 ? bwd_dk<0, __nv_bfloat16>(a, s) : bwd_dk<0, float>(a, s);
  return a.dtype == KDN_BF16 ? bwd_dk<1, __nv_bfloat16>(a, s) : bwd_dk<1, float>(a, s);
}

}  // namespace kdn
