// FP64-accurate small steps of Algorithm 1, designed for GB300's FP64 unit (about two FMAs per clock and
// SM): iterations run in FP32, and the quantities that fix the results are then computed or refined in
// FP64 with matrix products only.  Two launches, each a cluster of CTAs per problem: the FP32 iterations
// on the first CTA, the FP64 products spread over all of them, a cluster barrier between dependent products
// (operands go through L2 and are staged in shared memory).
//
//  k_svd_S  SVD of Q = U^* T V (Algorithm 3, final step): FP32 one-sided Jacobi gives a starting V; FP64
//           refinement of V as eigenvectors of H = Q^*Q (Ogita & Aishima 2018, iterative refinement for
//           the symmetric eigenvalue problem based on matrix multiplication, Hermitian form): per step
//           T1 = V^*V, T2 = H V, S = V^* T2, the correction F = I + E, V <- V F, until ||E||_F <= 1e-9; the
//           eigenpairs sorted, sigma = sqrt(eigenvalues); U_Q = Q V_Q Sigma^{-1} and
//           S_l = (U_Q^* (U^* T_l V)) V_Q Sigma^{-1} (Eq. generateSl).
//  k_eig_t  C_mu = sum_l mu_l S_l, its eigenvectors W (FP32 Hessenberg reduction, shifted complex QR,
//           triangular eigenvectors Y: W = Z Y) and the FP32 inverse X = Y^{-1} Z^*; one first-order
//           correction of W from its FP64 residual; two FP64 Newton-Schulz steps X <- 2X - X (W X); z_j(l) = (X S_l W)_jj,
//           t_j(l) = -arg z_j(l) / 2pi mod 1 (Eq. diagonalizeSl).  The diagonal of W^{-1} S_l W is
//           stationary in W: an error E in W (W = W_0 (I + E)) changes it only at second order, and the
//           correction squares E once more, so z carries FP64 accuracy even though W comes from FP32
//           iterations.
//  k_canon  phase-canonical singular basis for the S_l output.
//
// One launch per product (25 of them, 16 x 16 tiles) and one-CTA iterations before took, at m = 5 / 20 /
// 40 (one problem), 300 / 910 / 2900 us; now 120 / 340 / 1000 us; 64 problems of m = 40 in one call 4.4 -> 2.2 ms.
#include "common.cuh"

#include <algorithm>
#include <cmath>


namespace {

__device__ inline void set_status_e(ProbState& s, int st) {
  if (s.status == ST_OK) s.status = st;
}

// a problem takes part in the SVD of Q: its power loop ended with a U of width a <= r0 and a V of
// width b <= m
__device__ inline bool svd_live(const ProbDesc& p, const ProbState& st) {
  return !st.done && st.status != ST_ENAN && st.wv > 0 && st.wu > 0 && st.wv <= p.m && st.wu <= p.r0;
}
// ... and in the eigen step (width m = wv of its S_l)
__device__ inline bool eig_live(const ProbDesc& p, const ProbState& st) {
  return !st.done && st.status != ST_ENAN && st.wv > 0 && st.wv <= p.m;
}

// ----------------------------------------------------------------------------- FP32 complex
__device__ inline float2 fc(float x, float y) { return make_float2(x, y); }
__device__ inline float2 fmul(float2 a, float2 b) { return fc(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x); }
__device__ inline float2 fmulc(float2 a, float2 b) { return fc(a.x * b.x + a.y * b.y, a.x * b.y - a.y * b.x); }
__device__ inline float2 fadd(float2 a, float2 b) { return fc(a.x + b.x, a.y + b.y); }
__device__ inline float2 fsub(float2 a, float2 b) { return fc(a.x - b.x, a.y - b.y); }
__device__ inline float2 fconj(float2 a) { return fc(a.x, -a.y); }
__device__ inline float2 fscale(float2 a, float s) { return fc(a.x * s, a.y * s); }
__device__ inline float fabs2(float2 a) { return a.x * a.x + a.y * a.y; }
__device__ inline float fabs1(float2 a) { return fabsf(a.x) + fabsf(a.y); }
__device__ inline float2 fdiv(float2 a, float2 b) {
  if (fabsf(b.x) >= fabsf(b.y)) {
    float r = b.y / b.x, den = b.x + b.y * r;
    return fc((a.x + a.y * r) / den, (a.y - a.x * r) / den);
  }
  float r = b.x / b.y, den = b.x * r + b.y;
  return fc((a.x * r + a.y) / den, (a.y * r - a.x) / den);
}
__device__ inline float rsqrt_a(float x) {       // approximation (0 for denormals' infinity is not asked for)
  float r;
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
}
// a square root for the shifts of the QR iteration (approximate: a shift need not be exact)
__device__ inline float2 fsqrtc(float2 a) {
  const float q = fabs2(a);
  if (!(q > 1e-36f)) return fc(0.f, 0.f);
  const float t = 0.5f * (q * rsqrt_a(q) + fabsf(a.x)), rt = rsqrt_a(t), sx = t * rt, o = 0.5f * a.y * rt;
  if (a.x >= 0.f) return fc(sx, o);
  return fc(fabsf(o), a.y >= 0.f ? sx : -sx);
}
// 1 / sqrt(x) correctly rounded but for the last step (a Newton step on the approximation): rotations and
// reflectors built from it stay unitary to FP32 rounding
__device__ inline float rsqrt_n(float x) {
  const float r = rsqrt_a(x);
  return fmaf(0.5f * r, fmaf(-x * r, r, 1.f), r);
}
__device__ inline float2 shfl2(float2 v, int src) {
  return fc(__shfl_sync(0xffffffffu, v.x, src), __shfl_sync(0xffffffffu, v.y, src));
}
// element i of a row spread over a warp: lane i & 31, register i >> 5
template <int NQ>
__device__ __forceinline__ float2 pick(const float2 (&v)[NQ], int i) {
  return shfl2(NQ == 1 || i < 32 ? v[0] : v[NQ - 1], i & 31);
}

// block-wide sum of a double, in thread 0 (every FP64 instruction of a warp holds the pipe for about sixteen
// cycles: one warp adds the partial sums of the others)
__device__ double block_sum_d(double v, double* sh) {
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  __syncthreads();
  if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = v;
  __syncthreads();
  if (threadIdx.x < 32) {
    v = threadIdx.x < blockDim.x >> 5 ? sh[threadIdx.x] : 0.0;
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  }
  return v;
}

// pair k of a round-robin step (circle ordering: position 0 fixed, positions 1..nb-1 rotate), step < nb - 1
__device__ inline void rr_pair(int step, int k, int nb, int& pa, int& pb) {
  auto who = [&](int pos) {
    const int q = pos - 1 + step;
    return pos == 0 ? 0 : (q >= nb - 1 ? q - (nb - 1) : q) + 1;
  };
  const int x = who(k), y = who(nb - 1 - k);
  pa = min(x, y);
  pb = max(x, y);
}

// ----------------------------------------------------------------------------- clusters and FP64 products
// Barrier over the CTAs of a problem; global writes before it are visible after it (read with ld.cg, so
// never from a stale L1 line).
template <int CL>
__device__ __forceinline__ void cl_sync() {
  if (CL > 1) {
    asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
  } else {
    __syncthreads();
  }
}

// rows x cols of a row-major matrix in global memory -> packed in shared memory
__device__ inline void stage(double2* dst, const double2* src, int ld, int rows, int cols) {
  for (int q = threadIdx.x; q < rows * cols; q += blockDim.x) dst[q] = __ldcg(src + (q / cols) * ld + q % cols);
}

// sum_k op(A[k as]) B[k bs], op = conjugation when CJ.  Four partial sums (k mod 4) keep eight
// independent FP64 chains per thread in flight.
template <bool CJ>
__device__ inline double2 zdot(const double2* A, int as, const double2* B, int bs, int K) {
  double2 acc[4];
#pragma unroll
  for (int u = 0; u < 4; ++u) acc[u] = make_double2(0.0, 0.0);
  int k = 0;
  for (; k + 4 <= K; k += 4) {
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const double2 a = A[(k + u) * as], b = B[(k + u) * bs];
      const double ay = CJ ? -a.y : a.y;
      acc[u].x = fma(a.x, b.x, acc[u].x);
      acc[u].y = fma(a.x, b.y, acc[u].y);
      acc[u].x = fma(-ay, b.y, acc[u].x);
      acc[u].y = fma(ay, b.x, acc[u].y);
    }
  }
#pragma unroll
  for (int u = 0; u < 3; ++u)
    if (k + u < K) {
      const double2 a = A[(k + u) * as], b = B[(k + u) * bs];
      const double ay = CJ ? -a.y : a.y;
      acc[u].x = fma(a.x, b.x, acc[u].x);
      acc[u].y = fma(a.x, b.y, acc[u].y);
      acc[u].x = fma(-ay, b.y, acc[u].x);
      acc[u].y = fma(ay, b.x, acc[u].y);
    }
  return cadd(cadd(acc[0], acc[1]), cadd(acc[2], acc[3]));
}

// entry e of the upper triangle (j (j + 1) / 2 + i, i <= j)
__device__ inline void tri(int e, int& i, int& j) {
  j = (int)((sqrtf(8.f * e + 1.f) - 1.f) * 0.5f);
  if (j * (j + 1) / 2 > e) --j;
  if ((j + 1) * (j + 2) / 2 <= e) ++j;
  i = e - j * (j + 1) / 2;
}

// Refinement steps at most.  Two where singular values are well apart, three to five at relative gaps of 1e-3 to
// 1e-4; below that a pair is now and then held for a cluster by another pair's correction, and 7 to 20 steps were
// seen.  Stopped at six, m = 64 with gaps of 1e-4 kept an error of 1e-4 in z (2e-12 converged).
constexpr int OA_MAX = 32;

// FP32 one-sided Jacobi on the columns of Q (a x b, a <= 32 NA): right singular vectors -> V (FP64, ld LM).
// A warp takes a pair of columns and holds both, and those of V, in registers from the inner product to
// the rotation; the squared norms are kept and updated with the rotations (and computed afresh every
// sweep), so a pair costs one inner product.  Rotations are unitary to FP32 rounding; angles need not be.
template <int NA>
__device__ void svd_jacobi(const Dev& D, ProbState& st, const double2* Q, int a, int b, int LM, double2* V, float2* fsm) {
  __shared__ int s_rot;
  __shared__ float nrm[PRONY_MMAX];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nwarp = blockDim.x >> 5;
  float2* Qc = fsm;                                             // [b][a] columns
  float2* Vc = fsm + (size_t)a * b;                             // [b][b] columns
  // Q times the power of two that takes its largest entry to [2^24, 2^25): the squares and fourth powers below then
  // stay in range whatever the unit of the samples (V does not depend on the factor), columns down to 1e-15 of
  // the largest included.  On the exponent bits: FP64 operations and conversions are slow here.
  if (threadIdx.x == 0) s_rot = 0;
  __syncthreads();
  {
    int e = 0;
    for (int idx = threadIdx.x; idx < a * b; idx += blockDim.x) {
      const double2 q = Q[idx / b * LM + idx % b];
      e = max(e, max((__double2hiint(q.x) >> 20) & 0x7FF, (__double2hiint(q.y) >> 20) & 0x7FF));
    }
    e = __reduce_max_sync(0xffffffffu, e);
    if (lane == 0) atomicMax(&s_rot, e);
  }
  __syncthreads();
  const int shift = 1023 + 24 - s_rot;
  auto scaled = [&](double v) {                  // v 2^shift; v itself where not finite
    const int hi = __double2hiint(v), e = (hi >> 20) & 0x7FF;
    if (e == 0x7FF) return (float)v;
    return e == 0 || e + shift <= 0 ? 0.f : (float)__hiloint2double(hi + shift * (1 << 20), __double2loint(v));
  };
  for (int idx = threadIdx.x; idx < a * b; idx += blockDim.x) {
    const int i = idx / b, j = idx % b;
    const double2 q = Q[i * LM + j];
    Qc[j * a + i] = fc(scaled(q.x), scaled(q.y));
  }
  for (int idx = threadIdx.x; idx < b * b; idx += blockDim.x) {
    const int i = idx % b, j = idx / b;
    Vc[j * b + i] = fc(i == j ? 1.f : 0.f, 0.f);
  }
  const int nb = b + (b & 1);
  const float jtol = 4.f * a * 5.9604645e-8f, jtol2 = jtol * jtol;
  const int max_sweeps = D.cap_jacobi > 0 ? D.cap_jacobi : 30;
  int sweep = 0;
  bool rotated = b > 1;                          // the last sweep still rotated (not converged)
  for (; sweep < max_sweeps && b > 1; ++sweep) {
    __syncthreads();
    if (threadIdx.x == 0) s_rot = 0;
    for (int j = warp; j < b; j += nwarp) {
      float s = 0.f;
      for (int i = lane; i < a; i += 32) s += fabs2(Qc[j * a + i]);
      for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
      if (lane == 0) nrm[j] = s;
    }
    __syncthreads();
    for (int step = 0; step < nb - 1; ++step) {
      for (int k = warp; k < nb / 2; k += nwarp) {
        int pa, pb;
        rr_pair(step, k, nb, pa, pb);
        if (pb >= b) continue;
        float2* xa = Qc + pa * a;
        float2* xb = Qc + pb * a;
        float2* va = Vc + pa * b;
        float2* vb = Vc + pb * b;
        float2 x[NA], y[NA], u[2], v[2], ga = fc(0.f, 0.f);
#pragma unroll
        for (int q = 0; q < NA; ++q) {
          const int i = lane + 32 * q;
          x[q] = i < a ? xa[i] : fc(0.f, 0.f);
          y[q] = i < a ? xb[i] : fc(0.f, 0.f);
        }
#pragma unroll
        for (int q = 0; q < 2; ++q) {
          const int i = lane + 32 * q;
          u[q] = i < b ? va[i] : fc(0.f, 0.f);
          v[q] = i < b ? vb[i] : fc(0.f, 0.f);
        }
        const float al = nrm[pa], be = nrm[pb];
#pragma unroll
        for (int q = 0; q < NA; ++q) ga = fadd(ga, fmulc(x[q], y[q]));
        for (int o = 16; o > 0; o >>= 1) {
          ga.x += __shfl_xor_sync(0xffffffffu, ga.x, o);
          ga.y += __shfl_xor_sync(0xffffffffu, ga.y, o);
        }
        const float ag2 = fabs2(ga);
        // (|gamma| below 3e-19, where the square of the largest column is above 2e14: nothing to rotate)
        if (!(ag2 > jtol2 * fmaxf(al * be, 0.f)) || ag2 < 1e-37f) continue;
        const float ri = rsqrtf(ag2), ag = ag2 * ri;             // 1 / |gamma|, |gamma|
        const float zeta = fminf(fmaxf((be - al) * 0.5f * ri, -1e18f), 1e18f), z1 = fmaf(zeta, zeta, 1.f);
        const float tt = copysignf(__fdividef(1.f, fabsf(zeta) + z1 * rsqrtf(z1)), zeta);
        const float c = rsqrt_n(fmaf(tt, tt, 1.f)), s = c * tt;
        const float rn = rsqrt_n(ag2);
        const float2 ph = fc(ga.x * rn, -ga.y * rn);             // e^{-i arg gamma}
#pragma unroll
        for (int q = 0; q < NA; ++q) {
          const int i = lane + 32 * q;
          const float2 yp = fmul(y[q], ph);
          if (i < a) {
            xa[i] = fsub(fscale(x[q], c), fscale(yp, s));
            xb[i] = fadd(fscale(x[q], s), fscale(yp, c));
          }
        }
#pragma unroll
        for (int q = 0; q < 2; ++q) {
          const int i = lane + 32 * q;
          const float2 vp = fmul(v[q], ph);
          if (i < b) {
            va[i] = fsub(fscale(u[q], c), fscale(vp, s));
            vb[i] = fadd(fscale(u[q], s), fscale(vp, c));
          }
        }
        if (lane == 0) {
          nrm[pa] = al - tt * ag;
          nrm[pb] = be + tt * ag;
          s_rot = 1;
        }
      }
      __syncthreads();
    }
    rotated = s_rot != 0;
    if (!rotated) break;
  }
  for (int idx = threadIdx.x; idx < b * b; idx += blockDim.x) {
    const int i = idx / b, j = idx % b;
    const float2 v = Vc[j * b + i];
    V[i * LM + j] = make_double2(v.x, v.y);
  }
  if (threadIdx.x == 0 && sweep >= max_sweeps && rotated) set_status_e(st, ST_ENOCONV);
}

// ----------------------------------------------------------------------------- SVD of Q and S_l
template <int CL, int NT>
__global__ void __launch_bounds__(NT) k_svd_S(Dev D, int cols) {
  extern __shared__ double2 zsm[];
  __shared__ double s_red[32];
  __shared__ double s_lam[PRONY_MMAX], s_inv[PRONY_MMAX];
  __shared__ int s_rank[PRONY_MMAX];
  __shared__ double s_delta, s_en;
  // upper-triangle entries per thread: b (b + 1) / 2 <= EMAX CL NT for the widest b of this NT
  constexpr int BM = NT > 512 ? 64 : NT > 128 ? 32 : 16, EMAX = (BM * (BM + 1) / 2 + CL * NT - 1) / (CL * NT);
  const ProbDesc& p = D.P[blockIdx.y];
  ProbState& st = D.st[blockIdx.y];
  if (!svd_live(p, st)) return;                  // the whole cluster
  const int rank = CL > 1 ? blockIdx.x : 0;
  const int a = st.wu, b = st.wv, LM = D.L.LDM;
  char* sb = D.small + p.soff;
  const double2* Q = (const double2*)(sb + D.L.q);
  double2* Hm = (double2*)(sb + D.L.work1);
  double2* V = (double2*)(sb + D.L.work2);
  double2* Vn = (double2*)(sb + D.L.S);          // the first S_l slot is free until the end
  double2* F = (double2*)(sb + D.L.work3);
  double2* T2 = (double2*)(sb + D.L.work4);
  double* lam = (double*)(sb + D.L.sigma);
  double* part = (double*)(sb + D.L.gram);       // partial norms: [quantity][CTA]
  double2* s1 = zsm;                             // two operands in shared memory
  double2* s2 = zsm + (size_t)b * b;
  const int ntri = b * (b + 1) / 2;
  // ---- starting V on the first CTA; H = Q^* Q on the others meanwhile
  if (rank == 0) {
    if (a <= 32) svd_jacobi<1>(D, st, Q, a, b, LM, V, (float2*)zsm);
    else if (a <= 64) svd_jacobi<2>(D, st, Q, a, b, LM, V, (float2*)zsm);
    else svd_jacobi<4>(D, st, Q, a, b, LM, V, (float2*)zsm);
  }
  if (CL == 1 || rank > 0) {
    __syncthreads();
    stage(zsm, Q, LM, a, b);
    __syncthreads();
    constexpr int R = CL > 1 ? CL - 1 : 1;
    for (int e = threadIdx.x * R + (CL > 1 ? rank - 1 : 0); e < ntri; e += NT * R) {
      int i, j;
      tri(e, i, j);
      const double2 h = zdot<true>(zsm + i, b, zsm + j, b, a);
      Hm[i * LM + j] = h;
      if (i != j) Hm[j * LM + i] = cconj(h);
    }
  }
  cl_sync<CL>();
  double e2 = 0.0;                               // ||H||_F^2 (thread 0, once)
  for (int it = 0; it < OA_MAX; ++it) {
    stage(s1, V, LM, b, b);
    stage(s2, Hm, LM, b, b);
    __syncthreads();
    if (it == 0) {
      for (int q = threadIdx.x; q < b * b; q += NT) e2 += cabs2(s2[q]);
      e2 = block_sum_d(e2, s_red);
    }
    double2 t1[EMAX], sv[EMAX];
    double e3 = 0.0;
#pragma unroll
    for (int x = 0; x < EMAX; ++x) {             // T1 = V^* V (kept by the thread)
      const int e = (threadIdx.x + x * NT) * CL + rank;
      t1[x] = make_double2(0.0, 0.0);
      if (e >= ntri) continue;
      int i, j;
      tri(e, i, j);
      t1[x] = zdot<true>(s1 + i, b, s1 + j, b, b);
      const double rx = (i == j ? 1.0 : 0.0) - t1[x].x;
      e3 += (i == j ? 1.0 : 2.0) * (rx * rx + t1[x].y * t1[x].y);
    }
    for (int e = threadIdx.x * CL + rank; e < b * b; e += NT * CL)   // T2 = H V
      T2[e / b * LM + e % b] = zdot<false>(s2 + (e / b) * b, 1, s1 + e % b, b, b);
    cl_sync<CL>();
    stage(s2, T2, LM, b, b);
    __syncthreads();
#pragma unroll
    for (int x = 0; x < EMAX; ++x) {             // S = V^* T2; lambda_i = s_ii / (V^* V)_ii
      const int e = (threadIdx.x + x * NT) * CL + rank;
      sv[x] = make_double2(0.0, 0.0);
      if (e >= ntri) continue;
      int i, j;
      tri(e, i, j);
      sv[x] = zdot<true>(s1 + i, b, s2 + j, b, b);
      if (i == j) lam[i] = sv[x].x / t1[x].x;
    }
    cl_sync<CL>();
    for (int i = threadIdx.x; i < b; i += NT) s_lam[i] = __ldcg(lam + i);
    __syncthreads();
    double e1 = 0.0;
#pragma unroll
    for (int x = 0; x < EMAX; ++x) {
      const int e = (threadIdx.x + x * NT) * CL + rank;
      if (e >= ntri) continue;
      int i, j;
      tri(e, i, j);
      const double sx = sv[x].x - (i == j ? s_lam[i] : 0.0);
      e1 += (i == j ? 1.0 : 2.0) * (sx * sx + sv[x].y * sv[x].y);
    }
    e1 = block_sum_d(e1, s_red);
    e3 = block_sum_d(e3, s_red);
    if (threadIdx.x == 0) {
      part[rank] = e1;
      part[CL + rank] = e3;
    }
    cl_sync<CL>();
    // E: e_ij = (s_ij + lambda_j r_ij) / (lambda_j - lambda_i) with R = I - V^*V, r_ij / 2 within a
    // cluster of eigenvalues closer than delta = 2 (||S - diag(lambda)||_F + ||H||_F ||R||_F)
    if (threadIdx.x == 0) {
      e1 = e3 = 0.0;
      for (int r = 0; r < CL; ++r) {
        e1 += __ldcg(part + r);
        e3 += __ldcg(part + CL + r);
      }
      s_delta = 2.0 * (sqrt(e1) + sqrt(e2 * e3));
    }
    __syncthreads();
    const double delta = s_delta;
    double en = 0.0;
#pragma unroll
    for (int x = 0; x < EMAX; ++x) {
      const int e = (threadIdx.x + x * NT) * CL + rank;
      if (e >= ntri) continue;
      int i, j;
      tri(e, i, j);
      const double2 r = make_double2((i == j ? 1.0 : 0.0) - t1[x].x, -t1[x].y);
      double2 eij = cscale(r, 0.5), eji = cconj(eij);
      const double gap = s_lam[j] - s_lam[i];
      if (i != j && fabs(gap) > delta) {
        const double ig = 1.0 / gap;
        eij = cscale(cadd(sv[x], cscale(r, s_lam[j])), ig);
        eji = cscale(cconj(cadd(sv[x], cscale(r, s_lam[i]))), -ig);
      }
      F[i * LM + j] = make_double2((i == j ? 1.0 : 0.0) + eij.x, eij.y);
      en += cabs2(eij);
      if (i != j) {
        F[j * LM + i] = eji;
        en += cabs2(eji);
      }
    }
    en = block_sum_d(en, s_red);
    if (threadIdx.x == 0) part[2 * CL + rank] = en;
    cl_sync<CL>();
    stage(s2, F, LM, b, b);
    if (threadIdx.x == 0) {
      en = 0.0;
      for (int r = 0; r < CL; ++r) en += __ldcg(part + 2 * CL + r);
      s_en = en;
    }
    __syncthreads();
    for (int e = threadIdx.x * CL + rank; e < b * b; e += NT * CL)   // V <- V F
      Vn[e / b * LM + e % b] = zdot<false>(s1 + (e / b) * b, 1, s2 + e % b, b, b);
    double2* t = V;
    V = Vn;
    Vn = t;
    cl_sync<CL>();
    // a step (after the first) with ||E||_F <= 1e-9 is the last: another would change V by less than
    // the FP64 rounding of the products
    if (it >= 1 && s_en <= 1e-18) break;
  }
  // ---- eigenpairs of H in descending order: V_Q, sigma = sqrt(lambda)
  double2* sVQ = zsm;
  double2* sA = zsm + (size_t)b * b;             // a x b operand
  __syncthreads();
  for (int j = threadIdx.x; j < b; j += NT) {
    int r = 0;
    for (int i = 0; i < b; ++i)
      if (s_lam[i] > s_lam[j] || (s_lam[i] == s_lam[j] && i < j)) ++r;
    s_rank[j] = r;
  }
  __syncthreads();
  double2* VQ = (double2*)(sb + D.L.vq);
  for (int q = threadIdx.x; q < b * b; q += NT) {
    const int i = q / b, j = q % b;
    const double2 v = __ldcg(V + i * LM + j);
    sVQ[i * b + s_rank[j]] = v;
    if (rank == 0) VQ[i * LM + s_rank[j]] = v;
  }
  double mine = 0.0;
  if (threadIdx.x < b) mine = sqrt(fmax(s_lam[threadIdx.x], 0.0));
  stage(sA, Q, LM, a, b);
  // every CTA has read lambda from its shared copy; the sorted sigma replaces it
  if (threadIdx.x < b) {
    s_inv[s_rank[threadIdx.x]] = mine > 0.0 ? 1.0 / mine : 0.0;
    if (rank == 0) lam[s_rank[threadIdx.x]] = mine;
    if (rank == 0 && s_rank[threadIdx.x] == b - 1) s_red[0] = mine;
    if (rank == 0 && s_rank[threadIdx.x] == 0) s_red[1] = mine;
  }
  // (over the cluster: after an odd number of steps V lies in the first S_l slot, which the CTAs write below)
  cl_sync<CL>();
  if (rank == 0 && threadIdx.x == 0) st.sigma_ratio = s_red[1] > 0.0 ? s_red[0] / s_red[1] : 0.0;
  // ---- U_Q = Q V_Q Sigma^{-1}, S_l = (U_Q^* M_l) V_Q Sigma^{-1}: this CTA takes the columns (of U_Q) and
  // rows (of S_l) i = rank mod CL, so no other CTA's results are needed
  const int ni = (b - rank + CL - 1) / CL;       // how many
  // `cols` of them at a time where shared memory does not hold all (a = 128, b = 64 and narrow clusters)
  const int cw = min(cols, (b + CL - 1) / CL);
  double2* sU = sA + (size_t)max(a, b) * b;      // a x cw
  double2* sP = sU + (size_t)a * cw;             // cw x b
  double2* UQ = (double2*)(sb + D.L.uq);
  for (int e = threadIdx.x; e < a * ni; e += NT) {
    const int r = e / ni, c = e % ni, i = rank + c * CL;
    const double2 u = cscale(zdot<false>(sA + r * b, 1, sVQ + i, b, b), s_inv[i]);
    if (ni <= cw) sU[e] = u;
    UQ[r * LM + i] = u;
  }
  for (int l = 0; l < p.d; ++l) {
    __syncthreads();
    stage(sA, (const double2*)(sb + D.L.mproj) + (size_t)l * D.L.LDR * LM, LM, a, b);
    double2* S = (double2*)(sb + D.L.S) + (size_t)l * LM * LM;
    for (int c0 = 0; c0 < ni; c0 += cw) {
      const int nc = min(cw, ni - c0);
      if (ni > cw)                               // (this CTA's own columns, written above)
        for (int e = threadIdx.x; e < a * nc; e += NT) sU[e] = UQ[(e / nc) * LM + rank + (c0 + e % nc) * CL];
      __syncthreads();
      for (int e = threadIdx.x; e < nc * b; e += NT) sP[e] = zdot<true>(sU + e / b, nc, sA + e % b, b, a);
      __syncthreads();
      for (int e = threadIdx.x; e < nc * b; e += NT)
        S[(rank + (c0 + e / b) * CL) * LM + e % b] = cscale(zdot<false>(sP + (e / b) * b, 1, sVQ + e % b, b, b), s_inv[e % b]);
    }
  }
}

// Canonical phases: ph_j = v_j[argmax] / |.| of V_final = V V_Q (in B1); S_l <- D^* S_l D with
// D = diag(conj ph); U_Q, V_Q columns times conj(ph).
__global__ void k_canon(Dev D) {
  const ProbDesc& p = D.P[blockIdx.x];
  ProbState& st = D.st[blockIdx.x];
  const int b = st.wv, a = st.wu;
  if (st.done || b <= 0 || a <= 0 || b > p.m || a > p.r0) return;
  const int LM = D.L.LDM;
  __shared__ double2 ph[PRONY_MMAX];
  const unsigned long long* am = (const unsigned long long*)(D.small + p.soff + D.L.argmx);
  for (int j = threadIdx.x; j < b; j += blockDim.x) {
    unsigned row = am[j] == 0ull ? 0u : 0xFFFFFFFFu - (unsigned)(am[j] & 0xFFFFFFFFull);
    if (row >= (unsigned)p.N) row = 0u;
    float2 v = D.B1[p.xoff + (long long)j * p.N + row];
    double r = hypot((double)v.x, (double)v.y);
    ph[j] = r > 0.0 ? make_double2(v.x / r, v.y / r) : make_double2(1.0, 0.0);
    ((double2*)(D.small + p.soff + D.L.phase))[j] = ph[j];
  }
  __syncthreads();
  for (int l = 0; l < p.d; ++l) {
    double2* S = (double2*)(D.small + p.soff + D.L.S) + (size_t)l * LM * LM;
    for (int idx = threadIdx.x; idx < b * b; idx += blockDim.x) {
      int i = idx / b, j = idx % b;
      S[i * LM + j] = cmul(cmul(ph[i], S[i * LM + j]), cconj(ph[j]));
    }
  }
  double2* UQ = (double2*)(D.small + p.soff + D.L.uq);
  double2* VQ = (double2*)(D.small + p.soff + D.L.vq);
  for (int idx = threadIdx.x; idx < a * b; idx += blockDim.x) {
    int i = idx / b, j = idx % b;
    UQ[i * LM + j] = cmul(UQ[i * LM + j], cconj(ph[j]));
  }
  for (int idx = threadIdx.x; idx < b * b; idx += blockDim.x) {
    int i = idx / b, j = idx % b;
    VQ[i * LM + j] = cmul(VQ[i * LM + j], cconj(ph[j]));
  }
}

// ----------------------------------------------------------------------------- eigen step
// mu of C_mu for every dimension: Philox draws, unit vectors (the same for every problem of a call)
struct MuTable { double2 v[PRONY_DMAX][PRONY_DMAX]; };   // [d - 1][l]

__device__ __forceinline__ void bar4() { asm volatile("bar.sync 1, 128;" ::: "memory"); }

// Eigenvectors W of the m x m matrix H (m <= 32 NQ; shared memory, pitch 32 NQ + 1, zero beyond m) and X ~ W^{-1}, both FP32 values, to
// global memory in FP64.  The whole block (at least 128 threads).
// (FP32 copies Wf, Xf, packed, and the eigenvalues lamf, times `unit`, beside them).
template <int NQ>
__device__ void eig_w(const Dev& D, ProbState& st, int m, float2* H, float2* Z, float2* Y, double2* Wd, double2* Xd,
                      int LM, float2* Wf, float2* Xf, float2* lamf, float unit) {
  constexpr int LD = 32 * NQ + 1;
  __shared__ float2 hv[PRONY_MMAX];
  __shared__ float4 rot[PRONY_MMAX];             // rotations of a sweep: c, Re s, Im s
  __shared__ float sv[PRONY_MMAX];
  __shared__ float s_red[32];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nwarp = blockDim.x >> 5;
  // ---- Householder reduction to Hessenberg form: warp 0 forms the reflector, then eight threads share
  // a column of H (sums over its rows), then a row of H or Z
  for (int k = 0; k + 2 < m; ++k) {
    if (warp == 0) {
      float2 x[NQ];
      float nx = 0.f;
#pragma unroll
      for (int q = 0; q < NQ; ++q) {
        const int i = lane + 32 * q;
        x[q] = (i > k && i < m) ? H[i * LD + k] : fc(0.f, 0.f);
        nx += fabs2(x[q]);
      }
      for (int o = 16; o > 0; o >>= 1) nx += __shfl_xor_sync(0xffffffffu, nx, o);
      nx = sqrtf(nx);
      const float2 x0 = pick<NQ>(x, k + 1);
      const float ax0 = sqrtf(fabs2(x0));
      const float2 ph = ax0 > 0.f ? fscale(x0, 1.f / ax0) : fc(1.f, 0.f);
      const float2 v0 = fadd(x0, fscale(ph, nx));
      // ||v||^2 = 2 nx (nx + |x0|)
      const float nv = 2.f * nx * (nx + ax0), inv = nv > 1e-36f ? rsqrt_n(nv) : 0.f;
#pragma unroll
      for (int q = 0; q < NQ; ++q) {
        const int i = lane + 32 * q;
        if (i < m) hv[i] = fscale(i == k + 1 ? v0 : x[q], inv);
      }
      if (lane == 0) s_red[0] = inv;
    }
    __syncthreads();
    if (s_red[0] > 0.f) {                        // (uniform)
      const int part = threadIdx.x & 7, grp = threadIdx.x >> 3, ngrp = blockDim.x >> 3;
      for (int j0 = k; j0 < m; j0 += ngrp) {
        const int j = j0 + grp;
        float2 h[4 * NQ], s = fc(0.f, 0.f);
#pragma unroll
        for (int e = 0; e < 4 * NQ; ++e) {
          const int i = k + 1 + part + 8 * e;
          h[e] = (i < m && j < m) ? H[i * LD + j] : fc(0.f, 0.f);
          if (i < m) s = fadd(s, fmulc(hv[i], h[e]));
        }
#pragma unroll
        for (int o = 4; o > 0; o >>= 1) {
          s.x += __shfl_xor_sync(0xffffffffu, s.x, o);
          s.y += __shfl_xor_sync(0xffffffffu, s.y, o);
        }
        s = fscale(s, 2.f);
#pragma unroll
        for (int e = 0; e < 4 * NQ; ++e) {
          const int i = k + 1 + part + 8 * e;
          if (i < m && j < m) H[i * LD + j] = (j == k && i > k + 1) ? fc(0.f, 0.f) : fsub(h[e], fmul(hv[i], s));
        }
      }
      __syncthreads();
      for (int i0 = 0; i0 < 2 * m; i0 += ngrp) {
        const int i = i0 + grp;
        float2* R = i < m ? H + i * LD : Z + (i - m) * LD;
        float2 h[4 * NQ], s = fc(0.f, 0.f);
#pragma unroll
        for (int e = 0; e < 4 * NQ; ++e) {
          const int j = k + 1 + part + 8 * e;
          h[e] = (j < m && i < 2 * m) ? R[j] : fc(0.f, 0.f);
          if (j < m) s = fadd(s, fmul(h[e], hv[j]));
        }
#pragma unroll
        for (int o = 4; o > 0; o >>= 1) {
          s.x += __shfl_xor_sync(0xffffffffu, s.x, o);
          s.y += __shfl_xor_sync(0xffffffffu, s.y, o);
        }
        s = fscale(s, 2.f);
#pragma unroll
        for (int e = 0; e < 4 * NQ; ++e) {
          const int j = k + 1 + part + 8 * e;
          if (j < m && i < 2 * m) R[j] = fsub(h[e], fmul(s, fconj(hv[j])));
        }
      }
    }
    __syncthreads();
  }
  // ---- shifted complex QR iteration, full Schur form, by four warps.  A sweep on the active block
  // l..hi: H - sigma I = Q R row by row on warp 0 (a lane owns a column; the rotation of step k is
  // formed from column k, which all earlier rotations have reached), then R Q + sigma I and Z Q with a
  // thread per row.  The dependent chain is one rotation per row instead of one with its row, column
  // and Z updates (180 cycles instead of about 420).  Entries of R left of the subdiagonal are stored
  // as they come and never read.
  if (warp < 4) {
    const float eps = 5.9604645e-8f;
    int hi = m - 1, its = 0, total = 0;
    const int cap = D.cap_eigqr > 0 ? D.cap_eigqr : 30 * m + 30;
    while (hi > 0) {
      if (total > cap) break;
      int l = 0;
#pragma unroll
      for (int q = NQ - 1; q >= 0; --q) {        // largest index with a negligible subdiagonal entry
        const int i = lane + 32 * q;
        bool small = false;
        if (i >= 1 && i <= hi) {
          float s = fabs1(H[(i - 1) * LD + i - 1]) + fabs1(H[i * LD + i]);
          if (s == 0.f) s = 1.f;
          small = fabs1(H[i * LD + i - 1]) <= eps * s;
        }
        const unsigned bal = __ballot_sync(0xffffffffu, small);
        if (l == 0 && bal) l = 32 * q + 31 - __clz(bal);
      }
      if (l == hi) {
        --hi;
        its = 0;
        continue;
      }
      float2 sh;
      if (its == 10 || its == 20) {
        sh = fadd(H[hi * LD + hi], fc(0.75f * fabs1(H[hi * LD + hi - 1]), 0.f));
      } else {
        const float2 a = H[(hi - 1) * LD + hi - 1], bb = H[(hi - 1) * LD + hi], c = H[hi * LD + hi - 1], dd = H[hi * LD + hi];
        const float2 hd = fscale(fsub(a, dd), 0.5f);
        const float2 disc = fsqrtc(fadd(fmul(hd, hd), fmul(bb, c)));
        const float2 mid = fscale(fadd(a, dd), 0.5f);
        const float2 l1 = fadd(mid, disc), l2 = fsub(mid, disc);
        sh = fabs2(fsub(l1, dd)) <= fabs2(fsub(l2, dd)) ? l1 : l2;
      }
      bar4();                                    // every warp has read H
      if ((int)threadIdx.x >= l && (int)threadIdx.x <= hi) {
        H[threadIdx.x * LD + threadIdx.x] = fsub(H[threadIdx.x * LD + threadIdx.x], sh);
        if ((int)threadIdx.x == l && l > 0) H[l * LD + l - 1] = fc(0.f, 0.f);
      }
      bar4();
      if (warp == 0) {
        float2 cur[NQ], nx[NQ];
        float2* row = H + l * LD + lane;
#pragma unroll
        for (int q = 0; q < NQ; ++q) {
          cur[q] = row[32 * q];
          nx[q] = row[LD + 32 * q];
        }
#pragma unroll 2
        for (int k = l; k < hi; ++k, row += LD) {
          float2 nn[NQ];                         // the row after next (the last: any)
          const int ahead = k + 2 <= hi ? 2 * LD : LD;
#pragma unroll
          for (int q = 0; q < NQ; ++q) nn[q] = row[ahead + 32 * q];
          const float2 x = pick<NQ>(cur, k), y = pick<NQ>(nx, k);
          // c = |x| / r, s = x conj(y) / (|x| r), r^2 = |x|^2 + |y|^2, by one reciprocal root
          const float ax2 = fabs2(x), n2 = ax2 + fabs2(y), pr = ax2 * n2;
          const float2 xy = fmul(x, fconj(y));
          const float rr = rsqrt_n(pr);
          float c = ax2 * rr;
          float2 s = fscale(xy, rr);
          if (!(pr > 1e-36f)) {                  // x (or both) negligible
            c = n2 > 1e-36f ? 0.f : 1.f;
            s = n2 > 1e-36f ? fscale(fconj(y), rsqrt_n(n2)) : fc(0.f, 0.f);
          }
#pragma unroll
          for (int q = 0; q < NQ; ++q) {
            row[32 * q] = fadd(fscale(cur[q], c), fmul(s, nx[q]));
            cur[q] = fsub(fscale(nx[q], c), fmul(fconj(s), cur[q]));
            nx[q] = nn[q];
          }
          if (lane == 0) rot[k] = make_float4(c, s.x, s.y, 0.f);
        }
#pragma unroll
        for (int q = 0; q < NQ; ++q) row[32 * q] = cur[q];
      }
      bar4();
      {
        const bool zrow = threadIdx.x >= 64;
        const int i = threadIdx.x & 63;
        if (i < m && (zrow || i <= hi)) {
          float2* R = (zrow ? Z : H) + i * LD;
          // row i of R starts at its diagonal; the entry left of it is zero
          const bool low = !zrow && i > l;
          const int k0 = low ? i - 1 : l;
          float2 cur = low ? fc(0.f, 0.f) : R[l];
          float2 nx = R[k0 + 1];
          float4 rn = rot[k0];
#pragma unroll 2
          for (int k = k0; k < hi; ++k) {
            const float2 nn = R[min(k + 2, hi)];
            const float4 r = rn;
            rn = rot[min(k + 1, hi - 1)];
            const float2 s = fc(r.y, r.z);
            R[k] = fadd(fscale(cur, r.x), fmul(fconj(s), nx));
            cur = fsub(fscale(nx, r.x), fmul(s, cur));
            nx = nn;
          }
          if (!zrow && i >= l && i < hi) R[i] = fadd(R[i], sh);
          if (!zrow && i == hi) cur = fadd(cur, sh);
          R[hi] = cur;
        }
      }
      bar4();
      ++its;
      ++total;
    }
    if (threadIdx.x == 0 && hi > 0) set_status_e(st, ST_ENOCONV);
  }
  __syncthreads();
  // ---- triangular eigenvectors, a warp per column: (H_ii - lambda_k) y_i = -(H_ik + sum_{i < j < k} H_ij y_j)
  {
    float hn = 0.f;
    for (int q = threadIdx.x; q < m * m; q += blockDim.x) {
      const int i = q / m, j = q % m;
      if (j >= i) hn = fmaxf(hn, fabs1(H[i * LD + j]));
    }
    for (int o = 16; o > 0; o >>= 1) hn = fmaxf(hn, __shfl_xor_sync(0xffffffffu, hn, o));
    if (lane == 0) s_red[warp] = hn;
    __syncthreads();
    hn = 0.f;
    for (int w = 0; w < nwarp; ++w) hn = fmaxf(hn, s_red[w]);
    const float small = fmaxf(hn, 1e-30f) * 5.9604645e-8f;
    for (int k = threadIdx.x; k < m; k += blockDim.x) lamf[k] = fscale(H[k * LD + k], unit);
    for (int k = warp; k < m; k += nwarp) {
      const float2 lamk = H[k * LD + k];
      float2 acc[NQ], rd[NQ];
#pragma unroll
      for (int q = 0; q < NQ; ++q) {
        const int i = lane + 32 * q;
        acc[q] = rd[q] = fc(0.f, 0.f);
        if (i < k) {
          float2 den = fsub(H[i * LD + i], lamk);
          if (fabs1(den) < small) den = fc(small, 0.f);
          rd[q] = fdiv(fc(1.f, 0.f), den);
          acc[q] = fc(-H[i * LD + k].x, -H[i * LD + k].y);
        }
      }
      for (int i = k - 1; i >= 0; --i) {
        float2 hc[NQ];
#pragma unroll
        for (int q = 0; q < NQ; ++q) hc[q] = lane + 32 * q < i ? H[(lane + 32 * q) * LD + i] : fc(0.f, 0.f);
        float2 own[NQ];
#pragma unroll
        for (int q = 0; q < NQ; ++q) own[q] = fmul(acc[q], rd[q]);
        const float2 y = pick<NQ>(own, i);
#pragma unroll
        for (int q = 0; q < NQ; ++q) {
          acc[q] = fsub(acc[q], fmul(hc[q], y));
          if (lane + 32 * q == i) Y[i * LD + k] = y;
        }
      }
#pragma unroll
      for (int q = 0; q < NQ; ++q) {
        const int i = lane + 32 * q;
        if (i >= k && i < m) Y[i * LD + k] = fc(i == k ? 1.f : 0.f, 0.f);
      }
    }
  }
  __syncthreads();
  // ---- W = Z Y with unit columns (into H, then FP64)
  for (int q = threadIdx.x; q < m * m; q += blockDim.x) {
    const int i = q / m, k = q % m;
    float2 acc = fc(0.f, 0.f);
    for (int j = 0; j <= k; ++j) acc = fadd(acc, fmul(Z[i * LD + j], Y[j * LD + k]));
    H[i * LD + k] = acc;
  }
  __syncthreads();
  for (int k = warp; k < m; k += nwarp) {
    float s = 0.f;
    for (int i = lane; i < m; i += 32) s += fabs2(H[i * LD + k]);
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if (lane == 0) sv[k] = s > 0.f ? rsqrtf(s) : 1.f;
  }
  __syncthreads();
  for (int q = threadIdx.x; q < m * m; q += blockDim.x) {
    const int i = q / m, k = q % m;
    const float2 w = fscale(H[i * LD + k], sv[k]);
    Wd[i * LM + k] = make_double2(w.x, w.y);
    Wf[q] = w;
  }
  __syncthreads();
  // ---- Y^{-1} (into H), a warp per column: u_k = 1, u_i = -(Y_ik + sum_{i < j < k} Y_ij u_j)
  for (int k = warp; k < m; k += nwarp) {
    float2 acc[NQ];
#pragma unroll
    for (int q = 0; q < NQ; ++q) {
      const int i = lane + 32 * q;
      acc[q] = i < k ? fc(-Y[i * LD + k].x, -Y[i * LD + k].y) : fc(0.f, 0.f);
      if (i >= k && i < m) H[i * LD + k] = fc(i == k ? 1.f : 0.f, 0.f);
    }
    for (int i = k - 1; i >= 0; --i) {
      float2 yc[NQ];
#pragma unroll
      for (int q = 0; q < NQ; ++q) yc[q] = lane + 32 * q < i ? Y[(lane + 32 * q) * LD + i] : fc(0.f, 0.f);
      const float2 u = pick<NQ>(acc, i);
#pragma unroll
      for (int q = 0; q < NQ; ++q) {
        acc[q] = fsub(acc[q], fmul(yc[q], u));
        if (lane + 32 * q == i) H[i * LD + k] = u;
      }
    }
  }
  __syncthreads();
  // ---- X = diag(1 / sv) Y^{-1} Z^*
  for (int q = threadIdx.x; q < m * m; q += blockDim.x) {
    const int j = q / m, i = q % m;
    float2 acc = fc(0.f, 0.f);
    for (int b = j; b < m; ++b) acc = fadd(acc, fmul(H[j * LD + b], fconj(Z[i * LD + b])));
    const float f = 1.f / sv[j];
    Xd[j * LM + i] = make_double2(acc.x * f, acc.y * f);
    Xf[q] = fscale(acc, f);
  }
}

template <int CL, int NT>
__global__ void __launch_bounds__(NT) k_eig_t(Dev D, MuTable mu) {
  extern __shared__ double2 zsm[];
  const ProbDesc& p = D.P[blockIdx.y];
  ProbState& st = D.st[blockIdx.y];
  if (!eig_live(p, st)) return;                  // the whole cluster
  const int rank = CL > 1 ? blockIdx.x : 0;
  const int m = st.wv, LM = D.L.LDM;
  constexpr int NQ = NT > 512 ? 2 : 1, LD = 32 * NQ + 1;   // (NT by the widest problem of the batch)
  char* sb = D.small + p.soff;
  const double2* S = (const double2*)(sb + D.L.S);
  double2* Wd = (double2*)(sb + D.L.work2);      // W (FP64)
  double2* Xd = (double2*)(sb + D.L.work3);      // X, alternating with work1
  double2* Xn = (double2*)(sb + D.L.work1);
  double2* Rd = (double2*)(sb + D.L.work4);
  float2* Cm = (float2*)(sb + D.L.mapm);         // C_mu
  float2* Wf = (float2*)(sb + D.L.gram);         // FP32 W, X, eigenvalues (packed)
  float2* Xf = Wf + (size_t)m * m;
  float2* lamf = (float2*)(sb + D.L.q);
  for (int e = threadIdx.x * CL + rank; e < m * m; e += NT * CL) {
    const double2* s = S + (e / m) * LM + e % m;
    double2 acc = make_double2(0.0, 0.0);
    for (int l = 0; l < p.d; ++l) acc = cadd(acc, cmul(mu.v[p.d - 1][l], s[(size_t)l * LM * LM]));
    Cm[e] = fc((float)acc.x, (float)acc.y);
  }
  cl_sync<CL>();
  if (rank == 0) {
    float2* H = (float2*)zsm;                    // m x m each, pitch LD
    float2* Z = H + m * LD;
    float2* Y = Z + m * LD;
    __shared__ int s_big;
    if (threadIdx.x == 0) s_big = 0;
    __syncthreads();
    int big = 0;                                 // bits of the largest entry
    for (int q = threadIdx.x; q < m * LD; q += NT) {
      const int i = q / LD, j = q % LD;
      const float2 c = j < m ? __ldcg(Cm + i * m + j) : fc(0.f, 0.f);
      big = max(big, max(__float_as_int(fabsf(c.x)), __float_as_int(fabsf(c.y))));
      H[q] = c;
      Z[q] = fc(i == j ? 1.f : 0.f, 0.f);
    }
    big = __reduce_max_sync(0xffffffffu, big);
    if ((threadIdx.x & 31) == 0) atomicMax(&s_big, big);
    __syncthreads();
    // the QR iteration forms fourth powers of the entries: a matrix whose largest lies outside 2^-8..2^8 is
    // scaled by a power of two (its eigenvectors stay the same)
    const int e = s_big >> 23;
    const bool scale = e > 0 && e < 254 && (e < 127 - 8 || e > 127 + 8);
    if (scale) {
      const float f = __int_as_float((254 - e) << 23);
      for (int q = threadIdx.x; q < m * LD; q += NT) H[q] = fscale(H[q], f);
      __syncthreads();
    }
    eig_w<NQ>(D, st, m, H, Z, Y, Wd, Xd, LM, Wf, Xf, lamf, scale ? __int_as_float(e << 23) : 1.f);
    if (threadIdx.x == 0) st.rank_used = m;
  }
  cl_sync<CL>();
  // ---- this CTA owns the columns (of W and S_l W) and rows (of X) j = rank mod CL
  const int nj = (m - rank + CL - 1) / CL;
  double2* sW = zsm;
  double2* sX = sW + (size_t)m * m;
  double2* sR = sX + (size_t)m * m;
  double2* Cl = (double2*)(sb + D.L.mproj);      // S_l W, own columns
  double2* Wc = (double2*)(sb + D.L.vq);         // the corrected W (V_Q has served; others may still read W)
  const long long lC = (long long)D.L.LDR * LM;
  stage(sW, Wd, LM, m, m);
  __syncthreads();
  for (int e = threadIdx.x; e < p.d * m * nj; e += NT) {
    const int c = e % nj, q = e / nj, i = q % m, l = q / m, j = rank + c * CL;
    Cl[l * lC + i * LM + j] = zdot<false>(S + (size_t)l * LM * LM + i * LM, 1, sW + j, m, m);
  }
  // One correction of W: W <- W + dW, dW = W E, E_kj = (X (C_mu W - W Lambda))_kj / (lambda_j - lambda_k) off the
  // diagonal.  The residual is formed in FP64; being of FP32 size itself, the rest of the step is FP32,
  // and leaves W accurate to about the square of its FP32 error.
  {
    float2* fres = (float2*)sX;                  // m x nj: the residual, then E
    float2* fE = fres + (size_t)m * nj;
    float2* fS = fE + (size_t)m * nj;            // m x m
    float2* fdW = fS + (size_t)m * m;            // m x nj
    __syncthreads();
    for (int e = threadIdx.x; e < m * nj; e += NT) {
      const int c = e % nj, i = e / nj, j = rank + c * CL;
      double2 acc = make_double2(0.0, 0.0);
      for (int l = 0; l < p.d; ++l) acc = cadd(acc, cmul(mu.v[p.d - 1][l], Cl[l * lC + i * LM + j]));
      const float2 lj = __ldcg(lamf + j);
      acc = csub(acc, cmul(sW[i * m + j], make_double2(lj.x, lj.y)));
      fres[e] = fc((float)acc.x, (float)acc.y);
    }
    __syncthreads();
    for (int e = threadIdx.x; e < m * nj; e += NT) {
      const int c = e % nj, k = e / nj, j = rank + c * CL;
      float2 o = fc(0.f, 0.f);
#pragma unroll 4
      for (int i = 0; i < m; ++i) o = fadd(o, fmul(__ldcg(Xf + k * m + i), fres[i * nj + c]));
      const float2 gap = fsub(__ldcg(lamf + j), __ldcg(lamf + k));
      float2 ev = (k == j || fabs1(gap) == 0.f) ? fc(0.f, 0.f) : fdiv(o, gap);
      if (!(fabs1(ev) < 0.25f)) ev = fc(0.f, 0.f);               // no correction: eigenvalues too close
      fE[e] = ev;
    }
    __syncthreads();
    for (int e = threadIdx.x; e < m * nj; e += NT) {
      const int c = e % nj, i = e / nj, j = rank + c * CL;
      float2 o = fc(0.f, 0.f);
#pragma unroll 4
      for (int k = 0; k < m; ++k) o = fadd(o, fmul(__ldcg(Wf + i * m + k), fE[k * nj + c]));
      fdW[e] = o;
      Wc[i * LM + j] = make_double2(sW[i * m + j].x + (double)o.x, sW[i * m + j].y + (double)o.y);
    }
    for (int l = 0; l < p.d; ++l) {
      __syncthreads();
      for (int q = threadIdx.x; q < m * m; q += NT) {
        const double2 v = S[(size_t)l * LM * LM + (q / m) * LM + q % m];
        fS[q] = fc((float)v.x, (float)v.y);
      }
      __syncthreads();
      for (int e = threadIdx.x; e < m * nj; e += NT) {
        const int c = e % nj, i = e / nj, j = rank + c * CL;
        float2 o = fc(0.f, 0.f);
#pragma unroll 4
        for (int k = 0; k < m; ++k) o = fadd(o, fmul(fS[i * m + k], fdW[k * nj + c]));
        double2* at = &Cl[l * lC + i * LM + j];
        *at = make_double2(at->x + (double)o.x, at->y + (double)o.y);
      }
    }
  }
  cl_sync<CL>();
  // ---- Newton-Schulz steps X <- 2X - X (W X) until ||I - W X||_max before the last is below 1e-8 (two,
  // unless the correction of W was large).  A step squares the deviation: a W singular to FP32 leaves one that does
  // not fall, and the steps end after two; what then stays above 1e-8 is PRONY_ENOCONV.
  __shared__ float s_dev[32];
  __shared__ int s_more;
  float* devs = (float*)(lamf + m);              // one slot per CTA and parity of the step
  stage(sW, Wc, LM, m, m);
  float last = 0.f;                              // (thread 0) the deviation before
  for (int it = 0; it < 6; ++it) {
    stage(sX, Xd, LM, m, m);
    __syncthreads();
    float dev = 0.f;
    for (int e = threadIdx.x; e < nj * m; e += NT) {
      const int j = rank + e / m * CL, c = e % m;
      const double2 r = zdot<false>(sW + j * m, 1, sX + c, m, m);
      Rd[j * LM + c] = r;
      const float q = fabsf((float)(r.x - (c == j ? 1.0 : 0.0))) + fabsf((float)r.y);
      dev = fmaxf(dev, q < 1e30f ? q : 1e30f);   // (NaN among the large)
    }
    for (int o = 16; o > 0; o >>= 1) dev = fmaxf(dev, __shfl_xor_sync(0xffffffffu, dev, o));
    if ((threadIdx.x & 31) == 0) s_dev[threadIdx.x >> 5] = dev;
    __syncthreads();
    if (threadIdx.x == 0) {
      for (int w = 1; w < NT / 32; ++w) dev = fmaxf(dev, s_dev[w]);
      devs[(it & 1) * CL + rank] = dev;
    }
    cl_sync<CL>();
    stage(sR, Rd, LM, m, m);
    if (threadIdx.x == 0) {
      dev = 0.f;
      for (int r = 0; r < CL; ++r) dev = fmaxf(dev, __ldcg(devs + (it & 1) * CL + r));
      s_more = dev > 1e-8f && it < 5 && (it == 0 || dev < last);
      last = dev;
      if (!s_more && rank == 0 && dev > 1e-4f) set_status_e(st, ST_ENOCONV);
    }
    __syncthreads();
    for (int e = threadIdx.x; e < nj * m; e += NT) {
      const int j = rank + e / m * CL, c = e % m;
      const double2 v = zdot<false>(sX + j * m, 1, sR + c, m, m), x = sX[j * m + c];
      Xn[j * LM + c] = make_double2(2.0 * x.x - v.x, 2.0 * x.y - v.y);
    }
    double2* t = Xd;
    Xd = Xn;
    Xn = t;
    if (!s_more) break;                          // (the same in every CTA)
    cl_sync<CL>();
  }
  __syncthreads();                               // of the last X only this CTA's own rows are read
  // ---- z_j(l) = sum_a X[j][a] (S_l W)[a][j] for the own j
  double* tout = (double*)(sb + D.L.t);
  double2* zr = (double2*)(sb + D.L.zraw);
  for (int e = threadIdx.x; e < nj * p.d; e += NT) {
    const int c = e % nj, l = e / nj, j = rank + c * CL;
    const double2 z = zdot<false>(Xd + j * LM, 1, Cl + l * lC + j, LM, m);
    zr[j * PRONY_DMAX + l] = z;
    double tj = -atan2(z.y, z.x) / 6.283185307179586;
    tj -= floor(tj);
    if (tj >= 1.0) tj = 0.0;
    tout[j * PRONY_DMAX + l] = tj;
  }
}

template <typename... Args>
cudaError_t launch_cluster(void (*kernel)(Args...), int cl, int threads, size_t smem, int nprob, cudaStream_t s, Args... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(cl, nprob);
  cfg.blockDim = dim3(threads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = cl;
  at[0].val.clusterDim.y = 1;
  at[0].val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = cl > 1 ? 1 : 0;
  note_launch();
  return cudaLaunchKernelEx(&cfg, kernel, args...);
}

// Shared memory of k_svd_S: V_Q, an a x b operand, columns of U_Q and rows of P (the Jacobi columns, FP32, fit as well).
constexpr size_t SVD_SMEM = 227 * 1024 - 2560;   // what a block may have, less the kernel's static part
template <int CL, int NT>
cudaError_t run_svd(const Dev& D, cudaStream_t s) {
  const size_t a = std::max(D.L.LDR, D.L.LDM), b = D.L.LDM;
  // as many of the CTA's columns of U_Q as fit: all of them but for a >= 98 (CL = 1) to 124 (CL = 4), r0 = 2 m; at
  // least ten (a = 128, b = 64)
  const size_t fixed = b * b + a * b, cols = std::min((b + CL - 1) / CL, (SVD_SMEM / sizeof(double2) - fixed) / (a + b));
  const size_t sm = sizeof(double2) * (fixed + (a + b) * cols);
  const cudaError_t e = allow_smem(k_svd_S<CL, NT>, sm);
  if (e != cudaSuccess) return e;
  return launch_cluster(k_svd_S<CL, NT>, CL, NT, sm, D.nprob, s, D, (int)cols);
}

template <int CL, int NT>
cudaError_t run_eig(const Dev& D, const MuTable& mu, cudaStream_t s) {
  const size_t m = D.L.LDM, own = (m + CL - 1) / CL;
  // W and two more m x m operands (the correction's FP32 blocks fit in those); the FP32 iterations' three
  const size_t sm = std::max(sizeof(double2) * (m * m + std::max(2 * m * m, (m * m + 3 * m * own + 1) / 2)),
                             sizeof(float2) * 3 * m * (NT > 512 ? 65 : 33));
  const cudaError_t e = allow_smem(k_eig_t<CL, NT>, sm);
  if (e != cudaSuccess) return e;
  return launch_cluster(k_eig_t<CL, NT>, CL, NT, sm, D.nprob, s, D, mu);
}
}  // namespace

// The widest cluster whose CTAs are all resident at once (two per SM): a problem's FP32 iterations run on one
// CTA, so a second wave of problems would wait for whole iterations of the first.
static int cluster_of(const Dev& D) {
  const int m = D.L.LDM, fit = 2 * 152 / std::max(1, D.nprob);
  const int want = m > 32 ? 8 : m > 8 ? 4 : 1;
  return want >= 8 && fit >= 8 ? 8 : want >= 4 && fit >= 4 ? 4 : want >= 4 && fit >= 2 ? 2 : 1;
}

cudaError_t launch_svd_S(const Dev& D, cudaStream_t s) {
  const int cl = cluster_of(D);
  if (D.L.LDM > 32) {
    if (cl == 8) return run_svd<8, 640>(D, s);
    if (cl == 4) return run_svd<4, 640>(D, s);
    if (cl == 2) return run_svd<2, 640>(D, s);
    return run_svd<1, 640>(D, s);
  } else if (D.L.LDM > 16) {
    if (cl == 4) return run_svd<4, 512>(D, s);
    if (cl == 2) return run_svd<2, 512>(D, s);
    return run_svd<1, 512>(D, s);
  } else {
    if (cl == 4) return run_svd<4, 128>(D, s);
    if (cl == 2) return run_svd<2, 128>(D, s);
    return run_svd<1, 128>(D, s);
  }
}

void launch_canon(const Dev& D, cudaStream_t s) {
  note_launch();
  k_canon<<<D.nprob, 256, 0, s>>>(D);
}

cudaError_t launch_eig_t(const Dev& D, unsigned long long seed, cudaStream_t s) {
  double2 g[PRONY_DMAX];                         // complex normals (the draw convention of Philox above)
  for (int l = 0; l < PRONY_DMAX; ++l) {
    uint64_t c[4] = {(uint64_t)l, 0, 0, 0};
    philox4x64(c, seed, PRONY_STREAM_MU);
    const double r = std::sqrt(-std::log(philox_u01(c[0]))), u = 6.283185307179586 * philox_u01(c[1]);
    g[l] = make_double2(r * std::cos(u), r * std::sin(u));
  }
  MuTable mu = {};
  double nrm = 0.0;
  for (int d = 1; d <= PRONY_DMAX; ++d) {
    nrm += cabs2(g[d - 1]);
    for (int l = 0; l < d; ++l) mu.v[d - 1][l] = cscale(g[l], 1.0 / std::sqrt(nrm));
  }
  const int cl = cluster_of(D);
  if (D.L.LDM > 32) {
    if (cl == 8) return run_eig<8, 640>(D, mu, s);
    if (cl == 4) return run_eig<4, 640>(D, mu, s);
    if (cl == 2) return run_eig<2, 640>(D, mu, s);
    return run_eig<1, 640>(D, mu, s);
  } else if (D.L.LDM > 16) {
    if (cl == 4) return run_eig<4, 512>(D, mu, s);
    if (cl == 2) return run_eig<2, 512>(D, mu, s);
    return run_eig<1, 512>(D, mu, s);
  } else {
    if (cl == 4) return run_eig<4, 128>(D, mu, s);
    if (cl == 2) return run_eig<2, 128>(D, mu, s);
    return run_eig<1, 128>(D, mu, s);
  }
}
