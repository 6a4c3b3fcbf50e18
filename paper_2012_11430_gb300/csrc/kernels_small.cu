// Small per-problem kernels (one thread block per problem of a batch).
//
//  k_chol     FP32 Cholesky of the Gram X^* X with diagonal pivoting: the R factor of a
//             column-pivoted QR (Algorithm 3, lines with QR / QR with column pivoting),
//             the rank criterion ||R(i:r0,i:r0)||_F <= tol ||R||_F (Section 2.2) read off the
//             trailing Schur-complement trace, and the map X -> X P R^{-1}.
//  k_solve_c  FP64 L D L^H solve of the normal equations of Eq. ls_probl (the Gram matrix from k_powers);
//             results sorted by t.
// All loops are bounded; a cap that is hit sets PRONY_ENOCONV in the problem's state.
#include "common.cuh"
#include <algorithm>


namespace {

__device__ inline int swidth(const ProbState& s, const ProbDesc& p, int sel) { return sel_width(s, p, sel); }
__device__ inline void set_width(ProbState& s, int sel, int w) {
  if (sel == W_U) s.wu = w;
  else if (sel == W_V) s.wv = w;
}
__device__ inline void set_status(ProbState& s, int st) {
  if (s.status == ST_OK) s.status = st;
}

// ----------------------------------------------------------------------------- pivoted Cholesky (FP32)
// P^T A P = L L^H and R^{-1} = L^{-H} by elimination in place: a step with pivot column pv takes, from
// every row j that remains, T[j] -= (T[j][pv] / d) T[pv], where the columns that remain hold the Schur
// complement of A and the eliminated ones the same row operations applied to the identity (column pv
// becomes -T[j][pv] / d).  Row pv then holds row b of L^{-1} up to 1 / sqrt(d): no substitution follows, and
// nothing is swapped or scaled on the way.
// Warp 0 keeps the remaining diagonal in registers, updates it from row pv, and chooses the next pivot
// (largest entry, lowest index on ties; without pivoting the next column) and whether to stop while the
// other warps update the rows, four at a time so that their loads overlap: one barrier per step.
// One CTA per problem, bound by the latency of its w dependent steps.  The version that searched, swapped
// and scaled between barriers and then substituted back took 37 us at w = 40.
template <int NQ>                              // 32-column groups: LDR <= 32 NQ
__global__ void __launch_bounds__(NQ > 2 ? 512 : 256) k_chol(Dev D, int wsel, int target, int mode_in, double tol,
                                                             int rank_mode) {
  extern __shared__ float2 T[];                 // [w][LDR]
  __shared__ int perm[PRONY_RMAX];
  __shared__ int order[PRONY_RMAX];             // step at which a column was eliminated (w: not)
  __shared__ float dinv[PRONY_RMAX];            // 1 / sqrt of the pivots
  __shared__ float s_dp[2];                     // pivot and its column, of this step and the next
  __shared__ int s_piv[2];                      // (-1: stop)
  __shared__ int s_bad, s_rho, s_rank;
  const ProbDesc& p = D.P[blockIdx.x];
  ProbState& st = D.st[blockIdx.x];
  if (st.done) return;
  // QR_AUTO: the rank step (column pivoting and rank test, Algorithm 3) on a problem's first
  // power iteration, plain CholeskyQR afterwards
  const int mode = mode_in == QR_AUTO ? (st.iter == 0 ? QR_RANK : QR_PLAIN) : mode_in;
  const int w = swidth(st, p, wsel);
  const int LR = D.L.LDR;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarp = blockDim.x >> 5;
  const double2* G = (const double2*)(D.small + p.soff + D.L.gram);
#pragma unroll 4
  for (int idx = threadIdx.x; idx < w * LR; idx += blockDim.x) {
    const double2 g = G[idx];
    T[idx] = make_float2((float)g.x, (float)g.y);
  }
  for (int j = threadIdx.x; j < w; j += blockDim.x) order[j] = w;
  __syncthreads();
  const float tol2 = (float)(tol * tol);
  int limit = w;  // columns that may be accepted (never more than m after the rank step)
  if (mode == QR_RANK) limit = min(w, p.m);
  // warp 0: the remaining diagonal (0 where eliminated or past w), start values of the tests
  float d[NQ], trace0 = 0.f, maxd0 = 0.f;
  int rank = -1;
  // warp 0, before step i: choose its pivot or stop
  auto choose = [&](int i) {
    int pv = i;
    float dp = 0.f;
    bool stop = i >= w;
    if (mode == QR_PLAIN) {
#pragma unroll
      for (int q = 0; q < NQ; ++q)
        if (q == i >> 5) dp = d[q];
      dp = __shfl_sync(0xffffffffu, dp, i & 31);
    } else {
      unsigned key = 0;                         // bits of a non-negative float are ordered as integers
      int bi = PRONY_RMAX;
      float tr = 0.f;
#pragma unroll
      for (int q = NQ - 1; q >= 0; --q) {
        const int j = lane + 32 * q;
        if (j < w && order[j] == w) {
          const float dd = fmaxf(d[q], 0.f);
          tr += dd;
          if (bi == PRONY_RMAX || __float_as_uint(dd) >= key) {
            key = __float_as_uint(dd);
            bi = j;
          }
        }
      }
      const unsigned best = __reduce_max_sync(0xffffffffu, key);
      pv = __reduce_min_sync(0xffffffffu, key == best ? bi : PRONY_RMAX);
      if (mode == QR_RANK && rank < 0) {
        for (int o = 16; o > 0; o >>= 1) tr += __shfl_xor_sync(0xffffffffu, tr, o);
        if (!stop && tr <= tol2 * trace0) rank = i;
      }
      float mine = 0.f;
#pragma unroll
      for (int q = 0; q < NQ; ++q)
        if (q == pv >> 5) mine = d[q];
      dp = __shfl_sync(0xffffffffu, mine, pv & 31);
      if (mode == QR_DROP && dp <= tol2 * maxd0) stop = true;
      if (i >= limit && (mode != QR_RANK || rank >= 0)) stop = true;
      if (mode == QR_RANK && rank_mode == 1 && rank >= 0) stop = true;
    }
    if (!(dp > 1e-30f * maxd0) || !(dp > 0.f)) stop = true;                          // exhausted / not PD
    if (lane == 0) {
      s_piv[i & 1] = stop ? -1 : pv;
      s_dp[i & 1] = dp;
      if (stop) s_rho = min(i, limit);
      s_rank = rank;
    }
  };
  if (warp == 0) {
    bool finite = true;
#pragma unroll
    for (int q = 0; q < NQ; ++q) {
      const int j = lane + 32 * q;
      d[q] = j < w ? T[j * LR + j].x : 0.f;
      finite = finite && isfinite(d[q]);
      trace0 += fmaxf(d[q], 0.f);
      maxd0 = fmaxf(maxd0, d[q]);
    }
    for (int o = 16; o > 0; o >>= 1) {
      trace0 += __shfl_xor_sync(0xffffffffu, trace0, o);
      maxd0 = fmaxf(maxd0, __shfl_xor_sync(0xffffffffu, maxd0, o));
    }
    const bool bad = !__all_sync(0xffffffffu, finite) || !isfinite(trace0);
    if (lane == 0) {
      s_bad = bad;
      if (bad) {                        // non-finite block: the problem stops with ENAN
        st.status = ST_ENAN;
        st.done = 1;
        st.w_in = w;
        st.w_out = 0;
        set_width(st, target, 0);
      }
    }
    choose(0);
  }
  __syncthreads();
  if (s_bad) return;
  for (int i = 0;; ++i) {
    const int pv = s_piv[i & 1];
    if (pv < 0) break;
    const float inv = rsqrtf(s_dp[i & 1]), inv2 = inv * inv;
    float2 lk[NQ];                              // row pv, 1 in the place of the pivot
#pragma unroll
    for (int q = 0; q < NQ; ++q) {
      const int k = lane + 32 * q;
      lk[q] = k < w ? T[pv * LR + k] : make_float2(0.f, 0.f);
    }
    if (warp == 0) {
#pragma unroll
      for (int q = 0; q < NQ; ++q) {            // (scaled before they are squared: the Gram's unit is the samples' squared)
        const float x = lk[q].x * inv, y = lk[q].y * inv;
        d[q] -= x * x + y * y;
      }
      if (lane == 0) {
        perm[i] = pv;
        dinv[i] = inv;
        order[pv] = i;
      }
      __syncwarp();
      choose(i + 1);
    } else {
#pragma unroll
      for (int q = 0; q < NQ; ++q)
        if (lane + 32 * q == pv) lk[q] = make_float2(1.f, 0.f);
      for (int j0 = warp - 1; j0 < w; j0 += 4 * (nwarp - 1)) {
        float2 f[4], t[4][NQ];
        bool go[4];
#pragma unroll
        for (int r = 0; r < 4; ++r) {
          const int j = j0 + r * (nwarp - 1);
          // (order[pv] is written by warp 0 meanwhile: pv is excluded by its index)
          go[r] = j < w && j != pv && order[j] == w;
          const int jj = go[r] ? j : pv;
          const float2 v = T[jj * LR + pv];
          f[r] = make_float2(v.x * inv2, v.y * inv2);
#pragma unroll
          for (int q = 0; q < NQ; ++q) {
            const int k = lane + 32 * q;
            t[r][q] = (k < w && k != pv) ? T[jj * LR + k] : make_float2(0.f, 0.f);
          }
        }
        __syncwarp();                           // every lane has read T[j][pv] before one of them overwrites it
#pragma unroll
        for (int r = 0; r < 4; ++r) {
          if (!go[r]) continue;
          float2* row = T + (j0 + r * (nwarp - 1)) * LR;
#pragma unroll
          for (int q = 0; q < NQ; ++q) {
            const int k = lane + 32 * q;
            float2 v = t[r][q];
            v.x -= f[r].x * lk[q].x - f[r].y * lk[q].y;
            v.y -= f[r].x * lk[q].y + f[r].y * lk[q].x;
            if (k < w) row[k] = v;
          }
        }
      }
    }
    __syncthreads();
  }
  const int rho = min(s_rho, limit);
  // M[j][b] = R^{-1} in the original column order: conj(L^{-1}[b][j]) for the columns j eliminated up to step b
  float2* M = (float2*)(D.small + p.soff + D.L.mapm);
  for (int b = warp; b < rho; b += nwarp) {
    const float s = dinv[b];
    const float2* row = T + perm[b] * LR;
#pragma unroll
    for (int q = 0; q < NQ; ++q) {
      const int j = lane + 32 * q;
      if (j >= w) break;
      float2 v = make_float2(0.f, 0.f);
      if (order[j] < b) v = make_float2(row[j].x * s, -row[j].y * s);
      else if (order[j] == b) v = make_float2(s, 0.f);
      M[j * LR + b] = v;
    }
  }
  if (threadIdx.x == 0) {
    st.w_in = w;
    st.w_out = rho;
    set_width(st, target, rho);
    if (mode == QR_RANK) {
      st.rank_det = s_rank >= 0 ? s_rank : w;
      st.rank_used = rho;
      if (rho < p.m || st.rank_det < p.m) set_status(st, ST_ERANK);   // Section 2.2: rank below m
    }
    if (rho == 0) {
      set_status(st, ST_ERANK);
      st.done = 1;
    }
  }
}

// ----------------------------------------------------------------------------- c by normal equations (FP64)
__global__ void __launch_bounds__(256) k_solve_c(Dev D) {
  extern __shared__ double2 G[];                     // [m][MMAX]
  __shared__ double2 bb[PRONY_MMAX];
  __shared__ double ts[PRONY_MMAX * PRONY_DMAX];
  __shared__ int s_bad;
  const ProbDesc& p = D.P[blockIdx.x];
  ProbState& st = D.st[blockIdx.x];
  const int m = st.rank_used, d = p.d, LD = PRONY_MMAX;
  if (st.done || m <= 0 || m > p.m) return;
  double* t = (double*)(D.small + p.soff + D.L.t);
  double2* b = (double2*)(D.small + p.soff + D.L.rhs);
  double2* cout = (double2*)(D.small + p.soff + D.L.c);
  for (int q = threadIdx.x; q < m * d; q += blockDim.x) ts[(q / d) * PRONY_DMAX + q % d] = t[(q / d) * PRONY_DMAX + q % d];
  for (int i = threadIdx.x; i < m; i += blockDim.x) bb[i] = b[i];
  if (threadIdx.x == 0) s_bad = 0;
  __syncthreads();
  const double2* Gp = (const double2*)(D.small + p.soff + D.L.gram);   // lower triangle, packed (k_powers)
  for (int q = threadIdx.x; q < m * (m + 1) / 2; q += blockDim.x) {
    int i = (int)((sqrtf(8.f * q + 1.f) - 1.f) * 0.5f);
    if (i * (i + 1) / 2 > q) --i;
    if ((i + 1) * (i + 2) / 2 <= q) ++i;
    G[i * LD + q - i * (i + 1) / 2] = Gp[q];
  }
  __syncthreads();
  // G = L D L^H (unit lower L in place, reciprocals of D beside it): a step takes the reciprocal of its pivot
  // (one thread), the scaled column, then the trailing update, with three barriers and no square root
  // (4096 problems of m 1..5: 0.31 -> 0.16 ms; 64 of m = 40: 0.26 -> 0.10 ms)
  __shared__ double rd[PRONY_MMAX];
  __shared__ double2 col[PRONY_MMAX];
  for (int k = 0; k < m; ++k) {
    if (threadIdx.x == 0) {
      double dkk = G[k * LD + k].x;
      if (!(dkk > 0.0)) { s_bad = 1; dkk = 1e-300; }
      rd[k] = 1.0 / dkk;
    }
    __syncthreads();
    for (int i = k + 1 + threadIdx.x; i < m; i += blockDim.x) {
      const double2 g = G[i * LD + k];
      col[i] = cconj(g);
      G[i * LD + k] = cscale(g, rd[k]);
    }
    __syncthreads();
    const int rem = m - k - 1;
    for (int q = threadIdx.x; q < rem * (rem + 1) / 2; q += blockDim.x) {
      int i = (int)((sqrtf(8.f * q + 1.f) - 1.f) * 0.5f);
      if (i * (i + 1) / 2 > q) --i;
      if ((i + 1) * (i + 2) / 2 <= q) ++i;
      const int j = k + 1 + q - i * (i + 1) / 2;
      i += k + 1;
      G[i * LD + j] = csub(G[i * LD + j], cmul(G[i * LD + k], col[j]));
    }
    __syncthreads();
  }
  __shared__ double2 cs_[PRONY_MMAX];
  if (threadIdx.x < 32) {
    // L y = b, then L^H c = D^{-1} y, column by column on one warp: lane l keeps the running residuals
    // r_j (j = l, l + 32); each step updates the residuals of the rows that remain, so a step costs a
    // few dependent FP64 operations instead of a dot product of growing length
    const int lane = threadIdx.x;
    double2 r[2];
#pragma unroll
    for (int q = 0; q < 2; ++q) r[q] = lane + 32 * q < m ? bb[lane + 32 * q] : make_double2(0.0, 0.0);
    for (int i = 0; i < m; ++i) {
      const int q = i >> 5;
      double2 ri = q ? r[1] : r[0];
      ri.x = __shfl_sync(0xffffffffu, ri.x, i & 31);
      ri.y = __shfl_sync(0xffffffffu, ri.y, i & 31);
      const double2 yi = ri;
      if (lane == (i & 31)) cs_[i] = yi;
#pragma unroll
      for (int qq = 0; qq < 2; ++qq) {
        const int j = lane + 32 * qq;
        if (j > i && j < m) r[qq] = csub(r[qq], cmul(G[j * LD + i], yi));
      }
    }
    __syncwarp();
#pragma unroll
    for (int q = 0; q < 2; ++q)
      r[q] = lane + 32 * q < m ? cscale(cs_[lane + 32 * q], rd[lane + 32 * q]) : make_double2(0.0, 0.0);
    for (int i = m - 1; i >= 0; --i) {
      const int q = i >> 5;
      double2 ri = q ? r[1] : r[0];
      ri.x = __shfl_sync(0xffffffffu, ri.x, i & 31);
      ri.y = __shfl_sync(0xffffffffu, ri.y, i & 31);
      const double2 ci = ri;
      if (lane == (i & 31)) cs_[i] = ci;
#pragma unroll
      for (int qq = 0; qq < 2; ++qq) {
        const int j = lane + 32 * qq;
        if (j < i) r[qq] = csub(r[qq], cmul(cconj(G[i * LD + j]), ci));
      }
    }
    if (lane == 0 && s_bad) set_status(st, ST_ERANK);
  }
  __syncthreads();
  // sort (t, c) lexicographically by t (and the raw eigenvalues with them)
  __shared__ double2 zs[PRONY_MMAX * PRONY_DMAX];
  double2* zw = (double2*)(D.small + p.soff + D.L.zraw);
  for (int q = threadIdx.x; q < m * d; q += blockDim.x) zs[(q / d) * PRONY_DMAX + q % d] = zw[(q / d) * PRONY_DMAX + q % d];
  __syncthreads();
  for (int j = threadIdx.x; j < m; j += blockDim.x) {
    int r = 0;
    for (int i = 0; i < m; ++i) {
      bool less = false, eq = true;
      for (int l = 0; l < d && eq; ++l) {
        double a = ts[i * PRONY_DMAX + l], bq = ts[j * PRONY_DMAX + l];
        if (a < bq) { less = true; eq = false; }
        else if (a > bq) { eq = false; }
      }
      if (less || (eq && i < j)) ++r;
    }
    for (int l = 0; l < d; ++l) {
      t[r * PRONY_DMAX + l] = ts[j * PRONY_DMAX + l];
      zw[r * PRONY_DMAX + l] = zs[j * PRONY_DMAX + l];
    }
    cout[r] = cs_[j];
    b[j] = cs_[j];                                   // for the residual, in the order of the powers
  }
  if (threadIdx.x == 0) st.ls_num2 = 0.0;
}

// ----------------------------------------------------------------------------- convergence check
__global__ void k_check(Dev D, double tol_power, int max_iter, int* all_done) {
  int pi = blockIdx.x * blockDim.x + threadIdx.x;
  if (pi >= D.nprob) return;
  ProbState& s = D.st[pi];
  if (s.nonfinite) {
    s.status = ST_ENAN;
    s.done = 1;
  }
  if (s.done) return;
  s.iter += 1;
  double r2 = s.resid2, t2 = tol_power * tol_power * s.normT2;
  bool conv = r2 <= t2;
  bool stagn = s.resid2_prev >= 0.0 && r2 >= 0.64 * s.resid2_prev;
  bool nan = !(r2 == r2);
  if (nan) {
    s.status = ST_ENAN;
    s.done = 1;
  } else if (conv || stagn) {
    s.done = 1;
  } else if (s.iter >= max_iter) {
    set_status(s, ST_ENOCONV);
    s.done = 1;
  } else {
    s.resid2_prev = r2;
    s.resid2 = 0.0;
  }
  if (!s.done) atomicExch(all_done, 0);
}

// After the power loop: problems that stopped iterating take part in the finishing steps
// again (non-finite input stays excluded).
// A problem that failed (non-finite data, an empty U or V block, or a V block that never went
// through the rank step and is still wider than m) takes no part: rank_used = 0, so every
// finishing kernel skips it and its outputs are zero.
__global__ void k_reset_done(Dev D) {
  int pi = blockIdx.x * blockDim.x + threadIdx.x;
  if (pi >= D.nprob) return;
  ProbState& s = D.st[pi];
  const ProbDesc& p = D.P[pi];
  const bool failed = s.status == ST_ENAN || s.wv <= 0 || s.wu <= 0 || s.wv > p.m || s.wu > p.r0;
  if (failed) {
    if (s.status == ST_OK) set_status(s, ST_ERANK);
    s.rank_used = 0;
  }
  s.done = failed ? 1 : 0;
}

}  // namespace

void launch_reset_done(const Dev& D, cudaStream_t s) { note_launch(); k_reset_done<<<(D.nprob + 127) / 128, 128, 0, s>>>(D); }

template <int NQ>
static void run_chol(const Dev& D, int wsel, int target, int mode, double tol, int rank_mode, cudaStream_t s) {
  allow_smem(k_chol<NQ>, sizeof(float2) * 1024 * NQ * NQ);   // (a failure shows in the launch)
  note_launch();
  k_chol<NQ><<<D.nprob, NQ > 2 ? 512 : 256, sizeof(float2) * D.L.LDR * D.L.LDR, s>>>(D, wsel, target, mode, tol, rank_mode);
}

void launch_chol(const Dev& D, int wsel, int target, int mode, double tol, int rank_mode, cudaStream_t s) {
  switch ((D.L.LDR + 31) / 32) {
    case 1: return run_chol<1>(D, wsel, target, mode, tol, rank_mode, s);
    case 2: return run_chol<2>(D, wsel, target, mode, tol, rank_mode, s);
    case 3: return run_chol<3>(D, wsel, target, mode, tol, rank_mode, s);
    default: return run_chol<4>(D, wsel, target, mode, tol, rank_mode, s);
  }
}

void launch_solve_c(const Dev& D, cudaStream_t s) {
  const size_t sm = sizeof(double2) * PRONY_MMAX * PRONY_MMAX;
  allow_smem(k_solve_c, sm);
  note_launch();
  k_solve_c<<<D.nprob, 256, sm, s>>>(D);
}

void launch_check(const Dev& D, double tol_power, int max_iter, int* all_done, cudaStream_t s) {
  note_launch();
  k_check<<<(D.nprob + 127) / 128, 128, 0, s>>>(D, tol_power, max_iter, all_done);
}

namespace {
// Condition of the device-side power loop: run the body again while some problem iterates and
// fewer than `cap` bodies ran (the cap bounds the loop whatever the flags say).
__global__ void k_loop_cond(cudaGraphConditionalHandle h, const int* all_done, int* count, int cap) {
  const int c = ++(*count);
  cudaGraphSetConditional(h, (*all_done == 0 && c < cap) ? 1u : 0u);
}
}  // namespace

void launch_loop_cond(cudaGraphConditionalHandle h, const int* all_done, int* count, int cap, cudaStream_t s) {
  note_launch();
  k_loop_cond<<<1, 1, 0, s>>>(h, all_done, count, cap);
}
