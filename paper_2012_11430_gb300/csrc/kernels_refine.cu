// Least-squares refinement of the exponential-sum parameters (t_j, c_j) by damped Gauss-Newton
// (Levenberg-Marquardt) steps on L(t, c) = sum_k |f(k; t, c) - y_k|^2, f from Eq. (1), over an
// integer box of sample points.  Every step runs on the device, in two launches:
//   k_lm_points  at the candidate parameters: one pass over the points for L and
//                V^{l}_a      = sum_k w_l(k) conj(e_ak) r_k  (residual r_k, w_0 = 1, w_l = k_l),
//                from which J^* r of the real parameters follows, and Re(J^* J) from the Grams
//                M^{ll'}_{ab} = sum_k w_l(k) w_l'(k) conj(e_ak) e_bk
//   k_lm_step    one CTA: accept the candidate (its loss is lower) or keep the old point, adapt the
//                damping, then the next candidate from the normal equations Re(J^*J) delta = -Re(J^*r)
//                with Marquardt damping, Jacobi-scaled and solved by an FP32 Cholesky factorisation
// Two sets of (J^* J, V, L) alternate: the accepted point's and the candidate's, so a rejected
// candidate costs no new pass and an accepted one needs none either.
//
// On a box the sum over k of M factorises over the axes: with q = conj(e_a) e_b of one axis,
// M^{ll'}_{ab} is a product of the d one-dimensional sums of x^p q^x (p = 0, 1, 2 times the axis occurs
// among l, l').  A CTA computes the sums of one pair (a >= b) directly, sum_l len_l terms in place of
// prod_l len_l, and its (d + 2)^2 entries of J^* J; the rest of the pass is the residual and V, m (d + 1) sums over the points.
// The exponentials are recomputed in every pass, never stored; phases <t_j, k> mod 1 are exact
// 64-bit fixed-point sums, the sums FP32 over at most 128 terms, then FP64 over the tiles of a CTA and twice FP32
// (error-free sums) over the CTAs' FP32 results, in a fixed order: a refinement is reproducible.
// Near the minimum the decision compares losses that differ by less than FP32 rounding of the model
// would leave, so the model is evaluated beyond FP32: exp(-2 pi i u) = T[round(32 u)] (1 + eps)
// with |eps| < 0.1, the sum of c_j T in twice FP32 (error-free sums) from a table of the CTA, the sum of
// c_j T eps in FP32, whose rounding is ten times smaller than that of the whole.
// Measured at d = 2, n = 63 (16384 points), m = 20: a step took 195 us (143 in a one-CTA solve with three
// barriers per column, 40 in the M sums over all points, 9 in a separate trial pass), now 40 us (k_lm_step
// 26, k_lm_points 16, their launches overlapped): 50 steps 10.05 -> 1.98 ms.  Both kernels are latency chains
// on an almost idle GPU.
#include "common.cuh"

#include <algorithm>

namespace {

constexpr int LM_TILE = 128;            // points per CTA (= threads) in the point pass
constexpr int LM_SEG_BITS = 5, LM_SEG = 1 << LM_SEG_BITS;   // table points of the unit circle
constexpr int LM_CTA = 304;             // point CTAs (two per SM) of fewer than 32 tiles each,
constexpr int LM_MAXCTA = 608;          // and of more (lm_point_ctas)
constexpr int LM_EP = LM_TILE + 1;      // pitch of the exponentials (threads of different terms: different banks)
constexpr int LM_NB = 16;               // column block of the Cholesky factorisation
constexpr int LM_SOLVE_THREADS = 512;
constexpr double TWO_PI = 6.283185307179586;

// The steps are launched as a chain (programmatic dependent launch): a kernel's blocks become resident as soon as
// every block of the one before has begun, and wait here until it has completed and its writes are visible; what
// that saves is the launch latency between kernels of 16 to 26 us (50 steps: 2.25 -> 1.98 ms; the kernels of a solve,
// launched from a graph, gained nothing by it).  Every kernel launched so begins with chain_begin().
__device__ __forceinline__ void chain_begin() {
  asm volatile("griddepcontrol.wait;" ::: "memory");
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}
template <class... P, class... A>
void chain_launch(void (*k)(P...), int blocks, int threads, size_t smem, cudaStream_t s, A... args) {
  cudaLaunchConfig_t c = {};
  c.gridDim = dim3(blocks);
  c.blockDim = dim3(threads);
  c.dynamicSmemBytes = smem;
  c.stream = s;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  c.attrs = at;
  c.numAttrs = 1;
  cudaLaunchKernelEx(&c, k, static_cast<P>(args)...);
}

struct LmState {
  double lambda;
  int accepted;
  int cur;                              // set of the accepted point (the candidate's is 1 - cur)
};

// One set of accumulators (double): Re(J^* J) [P][P] (lower triangle), V[d+1][m] (complex), the loss.
__host__ __device__ inline long long lm_set_elems(int m, int d) {
  const long long P = (long long)m * (d + 2);
  return P * P + 2LL * (d + 1) * m + 1;
}

// sigma_alpha(a): the factor of column (a, alpha) of J besides w_{lambda(alpha)}(k) e_ak.
// alpha < d: t_a(alpha) -> -2 pi i c_a, weight index alpha + 1;  alpha = d: Re c_a -> 1;  d + 1: Im c_a -> i.
__device__ inline double2 sigma_of(int alpha, int d, double2 ca, int& widx) {
  if (alpha < d) {
    widx = alpha + 1;
    return make_double2(TWO_PI * ca.y, -TWO_PI * ca.x);
  }
  widx = 0;
  return alpha == d ? make_double2(1.0, 0.0) : make_double2(0.0, 1.0);
}

// acc += b in FP32; returns the rounding error of the sum (Knuth).
__device__ inline float two_sum(float& acc, float b) {
  const float a = acc, s = __fadd_rn(a, b), bb = __fsub_rn(s, a);
  acc = s;
  return __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb));
}
// (a + al)(b + bl) + (c + cl)(e + el) as an FP32 value and its remainder (products exact by FMA, Dekker).
__device__ inline void dot2(float a, float al, float b, float bl, float c, float cl, float e, float el, float& hi, float& lo) {
  float s = __fmul_rn(a, b);
  const float r1 = __fmaf_rn(a, b, -s), p = __fmul_rn(c, e), r2 = __fmaf_rn(c, e, -p);
  const float r3 = two_sum(s, p);
  hi = s;
  lo = (r1 + r2) + (r3 + ((a * bl + al * b) + (c * el + cl * e)));
}

// Leading dimension of the P + 1 rows of the solve: whole 16-byte groups, an odd number of them (the
// rows of eight lanes then start in different banks).
__host__ __device__ inline int lm_ld(int P) {
  const int g = (P + 4) / 4;
  return 4 * (g | 1);
}

// Axes of more than 4096 points (32 FP32 terms per thread) are summed as S pieces' starts times a piece of S points:
// 2 sqrt(len) terms.  The one CTA of a pair of terms would otherwise be bound by its own loop (one axis of 2^22 points,
// m = 1: 2324 us a step, now 300; of 65536: 55, now 26); up to 4096 points the loop hides under the points' pass.
__device__ inline int lm_axis_split(int len) {
  if (len <= 32 * LM_TILE) return 0;
  int s = 6;
  while ((1LL << 2 * s) < len) ++s;
  return 1 << s;
}

__device__ inline double block_sum(double v, double* red) {
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  __syncthreads();
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
  __syncthreads();
  double s = 0.0;
  if (threadIdx.x == 0)
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) s += red[w];
  return s;
}

// Blocks [0, npt_blocks): tiles of 128 points.  The others: a pair (a >= b) each.  vs: V[d+1][m]
// of every point block, ls: its loss.
__global__ void __launch_bounds__(LM_TILE) k_lm_points(const double* t, const double2* c, int m, int d, Box B,
                                                       long long K, int npt_blocks, const float2* y,
                                                       const LmState* st, const float4* circle, double* sets,
                                                       float2* vs, double* ls) {
  chain_begin();
  extern __shared__ float4 lm_smem[];
  __shared__ uint64_t T[PRONY_MMAX * PRONY_DMAX];
  __shared__ float2 Tf[LM_SEG];
  __shared__ double red[LM_TILE / 32];
  const int P = m * (d + 2);
  double* H = sets + (1 - st->cur) * lm_set_elems(m, d);
  if ((int)blockIdx.x >= npt_blocks) {
    __shared__ double axis_sum[LM_TILE / 32][3][PRONY_DMAX][6];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int pair = (int)blockIdx.x - npt_blocks;                // a (a + 1) / 2 + b
    int a = (int)((sqrtf(8.f * pair + 1.f) - 1.f) * 0.5f);
    while (a * (a + 1) / 2 > pair) --a;
    while ((a + 1) * (a + 2) / 2 <= pair) ++a;
    const int b = pair - a * (a + 1) / 2;
    for (int l = threadIdx.x; l < d; l += LM_TILE)                // conj(e_a) e_b = exp(-2 pi i (t_b - t_a) x)
      T[l] = frac64(t[b * d + l]) - frac64(t[a * d + l]);
    __syncthreads();
    // the warps' sums of x^p q^x (p = 0, 1, 2; re, im) over an axis, or over its pieces' starts, a piece and the rest
    bool split = false;
    for (int l = 0; l < d; ++l) {
      const uint64_t dt = T[l];
      const int len = B.len[l], S = lm_axis_split(len), U = S ? len / S : 0;
      if (S) split = true;
      for (int w = 0; w < (S ? 3 : 1); ++w) {
        const int n = S == 0 ? len : w == 0 ? S : w == 1 ? U : len - U * S;             // at most 2^16
        const int x0 = S == 0 || w == 1 ? B.lo[l] : w == 0 ? 0 : B.lo[l] + U * S, step = w == 1 ? S : 1;
        double tot = 0.0;                                         // lane z < 6: the z-th sum of the warp
        for (int i0 = 0; i0 < n; i0 += 32 * LM_TILE) {            // at most 32 FP32 terms per thread, then FP64
          float s[6] = {};
          const int i1 = min(n, i0 + 32 * LM_TILE);
          for (int i = i0 + threadIdx.x; i < i1; i += LM_TILE) {
            const int x = x0 + i * step;
            const float u = (float)(int)((dt * (uint64_t)(long long)x) >> 32) * 2.3283064365386963e-10f;
            float sn, cn;
            sincospif(2.0f * u, &sn, &cn);
            const float xf = (float)x, x2 = xf * xf;
            s[0] += cn;
            s[1] -= sn;
            s[2] += xf * cn;
            s[3] -= xf * sn;
            s[4] += x2 * cn;
            s[5] -= x2 * sn;
          }
          float mine = 0.f;
#pragma unroll
          for (int z = 0; z < 6; ++z) {                           // FP32 over a warp, FP64 beyond
            for (int o = 16; o > 0; o >>= 1) s[z] += __shfl_xor_sync(0xffffffffu, s[z], o);
            if (lane == z) mine = s[z];
          }
          tot += (double)mine;
        }
        if (lane < 6) axis_sum[warp][w][l][lane] = tot;
      }
    }
    __syncthreads();
    const int al = threadIdx.x / (d + 2), be = threadIdx.x % (d + 2);
    const int p = a * (d + 2) + al, q = b * (d + 2) + be;
    for (int z = threadIdx.x; z < 6 * d; z += LM_TILE)            // the warps' sums, in order
      for (int w = 0; w < (lm_axis_split(B.len[z / 6]) ? 3 : 1); ++w)
        axis_sum[0][w][z / 6][z % 6] += axis_sum[1][w][z / 6][z % 6] + axis_sum[2][w][z / 6][z % 6] + axis_sum[3][w][z / 6][z % 6];
    __syncthreads();
    if (split) {
      if (threadIdx.x < d && lm_axis_split(B.len[threadIdx.x])) {
        // sum_u sum_v (X_u + v)^p q^(X_u + v), X_u = lo + S u, from V_k = sum v^k q^v and X_k = sum X_u^k q^X_u; and
        // the last len - U S terms
        auto sum = [&](int w, int k) { return make_double2(axis_sum[0][w][threadIdx.x][2 * k], axis_sum[0][w][threadIdx.x][2 * k + 1]); };
        const double2 v0 = sum(0, 0), v1 = sum(0, 1), v2 = sum(0, 2), x0 = sum(1, 0), x1 = sum(1, 1), x2 = sum(1, 2);
        const double2 r[3] = {cmul(x0, v0), cadd(cmul(x1, v0), cmul(x0, v1)),
                              cadd(cadd(cmul(x2, v0), cscale(cmul(x1, v1), 2.0)), cmul(x0, v2))};
#pragma unroll
        for (int k = 0; k < 3; ++k) {
          const double2 t = cadd(r[k], sum(2, k));
          axis_sum[0][0][threadIdx.x][2 * k] = t.x;
          axis_sum[0][0][threadIdx.x][2 * k + 1] = t.y;
        }
      }
      __syncthreads();
    }
    if (al < d + 2 && q <= p) {
      int wa, wb;
      const double2 sa = sigma_of(al, d, c[a], wa), sb = sigma_of(be, d, c[b], wb);
      double2 v = make_double2(sa.x * sb.x + sa.y * sb.y, sa.x * sb.y - sa.y * sb.x);   // conj(sa) sb M_ab
      for (int l = 0; l < d; ++l) {
        const int pw = 2 * ((wa == l + 1) + (wb == l + 1));
        v = cmul(v, make_double2(axis_sum[0][0][l][pw], axis_sum[0][0][l][pw + 1]));
      }
      H[(long long)p * P + q] = v.x;
    }
    return;
  }
  float4* CT = lm_smem;                                  // m x LM_SEG: c_j T as (Re, Im) + (Re, Im) 2^-24 below
  float2* E = (float2*)(CT + m * LM_SEG);                // m x LM_EP: exponentials of this thread's point
  float2* R = E + m * LM_EP;                             // LM_TILE: residuals
  float2* part = R + LM_TILE;                            // LM_TILE partial sums of V
  float* Wt = (float*)(part + LM_TILE);                  // d x LM_TILE
  for (int q = threadIdx.x; q < m * d; q += blockDim.x) T[q] = frac64(t[q]);
  for (int q = threadIdx.x; q < LM_SEG; q += blockDim.x) Tf[q] = make_float2(circle[q].x, circle[q].y);
  for (int q = threadIdx.x; q < m * LM_SEG; q += blockDim.x) {
    const double2 c2 = c[q / LM_SEG];
    const float4 T2 = circle[q % LM_SEG];
    const float cx = (float)c2.x, cy = (float)c2.y, cxl = (float)(c2.x - cx), cyl = (float)(c2.y - cy);
    float4 v;
    dot2(cx, cxl, T2.x, T2.z, -cy, -cyl, T2.y, T2.w, v.x, v.z);
    dot2(cx, cxl, T2.y, T2.w, cy, cyl, T2.x, T2.z, v.y, v.w);
    CT[q] = v;
  }
  __syncthreads();
  const int i = threadIdx.x;
  const int nv = m * (d + 1), slices = max(1, LM_TILE / nv), per = LM_TILE / slices;
  double2 vsum[2] = {make_double2(0.0, 0.0), make_double2(0.0, 0.0)};   // V entries i, i + 128 (nv <= 256)
  double lsum = 0.0;
  for (long long tile = blockIdx.x; tile * LM_TILE < K; tile += npt_blocks) {
    const long long q = tile * LM_TILE + i;
    double2 rd = make_double2(0.0, 0.0);
    int k[PRONY_DMAX] = {0, 0, 0, 0};
    if (q < K) {
      if (K <= 0xFFFFFFFFLL) {
        unsigned rem = (unsigned)q;
        for (int l = d - 1; l >= 0; --l) {
          const unsigned len = (unsigned)B.len[l], nx = rem / len;
          k[l] = B.lo[l] + (int)(rem - nx * len);
          rem = nx;
        }
      } else {
        box_point(B, d, q, k);
      }
      float2 fh = make_float2(0.f, 0.f), fe = fh;           // sum of c T, and of its remainders and c T eps
      for (int j = 0; j < m; ++j) {
        uint64_t ph = 0;
        for (int l = 0; l < d; ++l) ph += T[j * d + l] * (uint64_t)(long long)k[l];
        const int seg = (int)((ph + (1ull << (63 - LM_SEG_BITS))) >> (64 - LM_SEG_BITS));        // nearest table point
        const int rem = (int)((long long)(ph - ((uint64_t)seg << (64 - LM_SEG_BITS))) >> 27);   // the rest in 2^-37 turns
        const float x = (float)rem * 4.5716190e-11f, x2 = x * x;                                // 2 pi 2^-37; |x| <= pi / 32
        // Taylor polynomials: the first terms left out are below 2e-11
        const float sn = x * (1.f + x2 * (-1.f / 6.f + x2 * (1.f / 120.f)));
        const float cm = x2 * (-0.5f + x2 * (1.f / 24.f - x2 * (1.f / 720.f)));                 // cos x - 1
        const float4 ct = CT[j * LM_SEG + seg];
        const float2 tf = Tf[seg];
        fe.x += two_sum(fh.x, ct.x) + (ct.z + (ct.x * cm + ct.y * sn));     // c T (cm - i sn)
        fe.y += two_sum(fh.y, ct.y) + (ct.w + (ct.y * cm - ct.x * sn));
        E[j * LM_EP + i] = make_float2(tf.x + (tf.x * cm + tf.y * sn), tf.y + (tf.y * cm - tf.x * sn));
      }
      const float2 yk = y[q];
      rd = make_double2((double)fh.x - (double)yk.x + (double)fe.x, (double)fh.y - (double)yk.y + (double)fe.y);
    } else {
      for (int j = 0; j < m; ++j) E[j * LM_EP + i] = make_float2(0.f, 0.f);
    }
    R[i] = make_float2((float)rd.x, (float)rd.y);
    for (int l = 0; l < d; ++l) Wt[l * LM_TILE + i] = (float)k[l];
    lsum += block_sum(rd.x * rd.x + rd.y * rd.y, red);      // (thread 0)
    __syncthreads();
    // V: one thread per (a, l) and slice of the points, the slices added in order
#pragma unroll
    for (int base = 0; base < 2 * LM_TILE; base += LM_TILE) {
      if (base >= nv) break;
      const int idx = slices > 1 ? i % nv : base + i, sl = slices > 1 ? i / nv : 0;
      float2 acc = make_float2(0.f, 0.f);
      if (idx < nv && sl < slices) {
        const int a = idx % m, l = idx / m;
        const int p1 = sl + 1 == slices ? LM_TILE : (sl + 1) * per;
        for (int p = sl * per; p < p1; ++p) {
          const float2 ea = E[a * LM_EP + p], rp = R[p];
          const float w = l == 0 ? 1.f : Wt[(l - 1) * LM_TILE + p];
          acc.x += w * (ea.x * rp.x + ea.y * rp.y);          // conj(ea) r
          acc.y += w * (ea.x * rp.y - ea.y * rp.x);
        }
      }
      if (slices > 1) {
        part[i] = acc;
        __syncthreads();
        if (sl == 0)
          for (int s2 = 1; s2 < slices; ++s2) {
            acc.x += part[i + s2 * nv].x;
            acc.y += part[i + s2 * nv].y;
          }
      }
      if (idx < nv && sl == 0) {
        vsum[base / LM_TILE].x += (double)acc.x;
        vsum[base / LM_TILE].y += (double)acc.y;
      }
    }
    __syncthreads();                                       // E, R and part are reused by the next tile
  }
#pragma unroll
  for (int u = 0; u < 2; ++u)
    if (i + u * LM_TILE < nv) vs[(long long)blockIdx.x * nv + i + u * LM_TILE] = make_float2((float)vsum[u].x, (float)vsum[u].y);
  if (i == 0) ls[blockIdx.x] = lsum;
}

// GB300 does about two FP64 operations per clock and SM (an FP64 square root takes thousands of cycles,
// and conversions share the pipe), so the scaling of the normal matrix works on the bits.
__device__ inline int exponent_of(double v) { return (int)((__double_as_longlong(v) >> 52) & 0x7FF) - 1023; }
// v 2^(-shift) in FP32 (rounded to nearest, ties away; below the FP32 range: zero; NaN for NaN and infinity)
__device__ inline float scaled_float(double v, int shift) {
  const uint64_t b = (uint64_t)__double_as_longlong(v);
  const int e11 = (int)((b >> 52) & 0x7FF), e = e11 - 896 - shift;
  const uint32_t sign = (uint32_t)(b >> 63) << 31;
  uint32_t f = ((uint32_t)e << 23 | (uint32_t)((b >> 29) & 0x7FFFFF)) + (uint32_t)((b >> 28) & 1);
  if (e <= 0) f = 0;
  if (e11 == 0x7FF || e >= 255) f = 0x7FC00000u;
  return __uint_as_float(f | sign);
}

// One CTA.  Decision on the candidate (step > 0; step 0 takes the starting point), then (solve) the
// damped normal equations at the accepted point -> next candidate.  P = m (d + 2) real parameters.
//
// Cholesky in blocks of 16 columns, with the right-hand side as an extra row, so that the forward
// substitution comes with the factorisation: the diagonal block by one warp (a row per lane, in
// registers, columns by shuffles), the rows below it by one thread each (16 columns in registers),
// the trailing block in 4 x 4 register tiles on and below the diagonal, 16 bytes per shared-memory
// access.  Three barriers per block instead of three per column; bound by the chain of dependent
// square roots and shuffles of the diagonal blocks.
__global__ void __launch_bounds__(LM_SOLVE_THREADS) k_lm_step(double* t, double2* c, double* tc, double2* cc, int m,
                                                              int d, LmState* st, double* sets, const float2* vs, const double* ls, int nblk,
                                                              double* hist, int step,
                                                              int solve) {
  chain_begin();
  extern __shared__ __align__(16) float lm_f[];
  __shared__ int s_ok, s_cur;
  __shared__ float dinv[PRONY_LM_PMAX];
  __shared__ __align__(16) float Ld[LM_NB][LM_NB];
  __shared__ double2 cs[PRONY_MMAX];
  const int P = m * (d + 2), ld = lm_ld(P);
  const long long ns = lm_set_elems(m, d);
  float* A = lm_f;                                   // ld x ld, lower triangle; row P: right-hand side
  float* Pt = A + ld * ld;                           // LM_NB x ld: the rows below a diagonal block, transposed
  float* sc = Pt + LM_NB * ld;                       // P: 1 / sqrt(damped diagonal) = sc 2^(-sh)
  int* sh = (int*)(sc + ld);
  {                                                  // V and the loss of the candidate: eight threads per entry
    const int nv = m * (d + 1), sub = threadIdx.x & 7;
    double* Vc = sets + (1 - st->cur) * ns + (long long)P * P;
    for (int v0 = 0; v0 < nv; v0 += LM_SOLVE_THREADS / 8) {
      const int v = v0 + (threadIdx.x >> 3);
      float2 hi = make_float2(0.f, 0.f), lo = hi;
      for (int k0 = sub; k0 < nblk; k0 += 64) {      // eight loads in flight
        float2 x[8];
#pragma unroll
        for (int u = 0; u < 8; ++u)
          x[u] = (v < nv && k0 + 8 * u < nblk) ? vs[(long long)(k0 + 8 * u) * nv + v] : make_float2(0.f, 0.f);
#pragma unroll
        for (int u = 0; u < 8; ++u) {
          lo.x += two_sum(hi.x, x[u].x);
          lo.y += two_sum(hi.y, x[u].y);
        }
      }
#pragma unroll
      for (int o = 4; o > 0; o >>= 1) {
        const float hx = __shfl_down_sync(0xffffffffu, hi.x, o), hy = __shfl_down_sync(0xffffffffu, hi.y, o);
        lo.x += __shfl_down_sync(0xffffffffu, lo.x, o) + two_sum(hi.x, hx);
        lo.y += __shfl_down_sync(0xffffffffu, lo.y, o) + two_sum(hi.y, hy);
      }
      if (sub == 0 && v < nv) {
        Vc[2 * v] = (double)hi.x + (double)lo.x;
        Vc[2 * v + 1] = (double)hi.y + (double)lo.y;
      }
    }
    if (threadIdx.x >= LM_SOLVE_THREADS - 32) {
      double l = 0.0;
      for (int k = threadIdx.x & 31; k < nblk; k += 32) l += ls[k];
      for (int o = 16; o > 0; o >>= 1) l += __shfl_xor_sync(0xffffffffu, l, o);
      if ((threadIdx.x & 31) == 0) Vc[2 * nv] = l;
    }
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    const int cand = 1 - st->cur;
    const double l0 = sets[(st->cur + 1) * ns - 1], l1 = sets[(cand + 1) * ns - 1];
    const int ok = step == 0 || (l1 < l0 && isfinite(l1));
    if (hist) hist[step] = ok ? l1 : l0;
    if (step > 0) {
      st->lambda = ok ? fmax(st->lambda * (1.0 / 3.0), 1e-12) : fmin(st->lambda * 4.0, 1e12);
      st->accepted += ok;
    }
    if (ok) st->cur = cand;
    s_ok = ok;
    s_cur = st->cur;
  }
  __syncthreads();
  if (s_ok && step > 0) {
    for (int q = threadIdx.x; q < m * d; q += blockDim.x) t[q] = tc[q];
    for (int q = threadIdx.x; q < m; q += blockDim.x) c[q] = cc[q];
  }
  if (!solve) return;
  const double lam = st->lambda;
  const double* H = sets + s_cur * ns;
  const double* V = H + (long long)P * P;
  for (int q = threadIdx.x; q < m; q += blockDim.x) cs[q] = (s_ok && step > 0) ? cc[q] : c[q];
  // the diagonal first (for the scaling)
  for (int p = threadIdx.x; p < P; p += blockDim.x) {
    const double v = H[(long long)p * P + p] * (1.0 + lam) + 1e-30;
    const int h = exponent_of(v) >> 1;
    const float f = scaled_float(v, 2 * h), r = rsqrtf(f);        // f in [1, 4)
    sh[p] = h;
    sc[p] = r;
    A[p * ld + p] = f * r * r;
  }
  __syncthreads();
#pragma unroll 4
  for (int idx = threadIdx.x; idx < P * (P - 1) / 2; idx += LM_SOLVE_THREADS) {   // entries below the diagonal
    int p = (int)((sqrtf(8.f * idx + 1.f) + 1.f) * 0.5f);
    if (p * (p - 1) / 2 > idx) --p;
    if (p * (p + 1) / 2 <= idx) ++p;
    const int q = idx - p * (p - 1) / 2;
    A[p * ld + q] = scaled_float(H[(long long)p * P + q], sh[p] + sh[q]) * sc[p] * sc[q];
  }
  for (int p = threadIdx.x; p < P; p += blockDim.x) {
    const int a = p / (d + 2), al = p % (d + 2);
    int wi;
    const double2 s = sigma_of(al, d, cs[a], wi);
    const double* v = V + 2 * (wi * m + a);
    const double re = s.x * v[0] + s.y * v[1];        // Re( conj(s) v )
    A[P * ld + p] = scaled_float(-re, sh[p]) * sc[p];
  }
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  for (int k0 = 0; k0 < P; k0 += LM_NB) {
    const int nb = min(LM_NB, P - k0);
    __syncthreads();
    if (warp == 0) {
      float row[LM_NB];
#pragma unroll
      for (int x = 0; x < LM_NB; ++x) row[x] = (lane < nb && x <= lane) ? A[(k0 + lane) * ld + k0 + x] : 0.f;
#pragma unroll
      for (int j = 0; j < LM_NB; ++j) {
        const float dj = __shfl_sync(0xffffffffu, row[j], j);
        const float dv = fmaxf(dj, 1e-20f), inv = rsqrtf(dv), root = dv * inv;
        const float l = lane == j ? root : row[j] * inv;
        row[j] = l;
        if (lane == j && j < nb) dinv[k0 + j] = inv;
#pragma unroll
        for (int x = j + 1; x < LM_NB; ++x) row[x] -= l * __shfl_sync(0xffffffffu, l, x);
      }
      if (lane < LM_NB) {
#pragma unroll
        for (int x = 0; x < LM_NB; ++x) {
          const float v = (lane < nb && x < nb && x <= lane) ? row[x] : 0.f;
          Ld[lane][x] = v;
          if (lane < nb && x <= lane) A[(k0 + lane) * ld + k0 + x] = v;
        }
      }
    }
    __syncthreads();
    const int r0 = k0 + nb, nr = P + 1 - r0;         // rows below, the right-hand side among them
    for (int i = threadIdx.x; i < nr; i += blockDim.x) {
      float* Ai = A + (r0 + i) * ld + k0;
      float x[LM_NB];
#pragma unroll
      for (int j = 0; j < LM_NB; j += 4) *(float4*)(x + j) = *(const float4*)(Ai + j);
#pragma unroll
      for (int j = 0; j < LM_NB; ++j) {
        x[j] = j < nb ? x[j] * dinv[k0 + j] : 0.f;
#pragma unroll
        for (int e = j + 1; e < LM_NB; ++e) x[e] -= x[j] * Ld[e][j];
        Pt[j * ld + i] = x[j];
      }
#pragma unroll
      for (int j = 0; j < LM_NB; ++j)
        if (j < nb) Ai[j] = x[j];
    }
    if (r0 >= P) break;
    __syncthreads();
    // trailing block: rows r0 + 4 ti .., columns r0 + 4 tj .., tj <= ti (what lies above the diagonal or
    // past row P is never read)
    const int nt = (nr + 3) / 4;
    for (int tile = threadIdx.x; tile < nt * (nt + 1) / 2; tile += blockDim.x) {
      int ti = (int)((sqrtf(8.f * tile + 1.f) - 1.f) * 0.5f);
      if (ti * (ti + 1) / 2 > tile) --ti;
      if ((ti + 1) * (ti + 2) / 2 <= tile) ++ti;
      const int tj = tile - ti * (ti + 1) / 2;
      float acc[4][4] = {};
#pragma unroll 4
      for (int j = 0; j < LM_NB; ++j) {
        const float4 x4 = *(const float4*)(Pt + j * ld + 4 * ti), z4 = *(const float4*)(Pt + j * ld + 4 * tj);
        const float x[4] = {x4.x, x4.y, x4.z, x4.w}, z[4] = {z4.x, z4.y, z4.z, z4.w};
#pragma unroll
        for (int u = 0; u < 4; ++u)
#pragma unroll
          for (int v = 0; v < 4; ++v) acc[u][v] += x[u] * z[v];
      }
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        float4* at = (float4*)(A + (r0 + 4 * ti + u) * ld + r0 + 4 * tj);
        float4 o = *at;
        o.x -= acc[u][0];
        o.y -= acc[u][1];
        o.z -= acc[u][2];
        o.w -= acc[u][3];
        *at = o;
      }
    }
  }
  __syncthreads();
  // L^T x = z (row P) by one warp: lane l keeps the running residuals of the entries l + 32 q
  if (warp == 0) {
    constexpr int NQ = PRONY_LM_PMAX / 32;
    float r[NQ];
#pragma unroll
    for (int q = 0; q < NQ; ++q) r[q] = lane + 32 * q < P ? A[P * ld + lane + 32 * q] : 0.f;
#pragma unroll
    for (int q = NQ - 1; q >= 0; --q)
#pragma unroll 4
      for (int jj = min(31, P - 1 - 32 * q); jj >= 0; --jj) {
        const int j = 32 * q + jj;
        const float xj = __shfl_sync(0xffffffffu, r[q], jj) * dinv[j];
#pragma unroll
        for (int e = 0; e <= q; ++e)
          if (lane + 32 * e < j) r[e] -= A[j * ld + lane + 32 * e] * xj;
        if (lane == jj) r[q] = xj;
      }
#pragma unroll
    for (int q = 0; q < NQ; ++q)
      if (lane + 32 * q < P) A[P * ld + lane + 32 * q] = r[q];
  }
  __syncthreads();
  for (int p = threadIdx.x; p < P; p += blockDim.x) {
    const int a = p / (d + 2), al = p % (d + 2);
    // sc 2^(-sh) in FP64
    const double delta = (double)(A[P * ld + p] * sc[p]) * __longlong_as_double((long long)(1023 - sh[p]) << 52);
    if (al < d) {
      // tc holds the accepted point if the last candidate was taken, t always does
      double v = ((s_ok && step > 0) ? tc[a * d + al] : t[a * d + al]) + delta;
      v -= floor(v);                                   // f is 1-periodic in each t_a(l)
      tc[a * d + al] = v;
    } else if (al == d) {
      cc[a].x = cs[a].x + delta;
    } else {
      cc[a].y = cs[a].y + delta;
    }
  }
}

// The starting point as the first candidate, empty accumulators.
__global__ void k_lm_init(LmState* st, double lambda0, const double* t, const double2* c, double* tc,
                          double2* cc, float4* circle, int m, int d) {
  if (threadIdx.x == 0) {
    st->lambda = lambda0;
    st->accepted = 0;
    st->cur = 1;
  }
  for (int q = threadIdx.x; q < LM_SEG; q += blockDim.x) {     // exp(-2 pi i q / LM_SEG)
    double sn, cn;
    sincospi(2.0 * q / LM_SEG, &sn, &cn);
    const float cf = (float)cn, sf = (float)-sn;
    circle[q] = make_float4(cf, sf, (float)(cn - cf), (float)(-sn - sf));
  }
  for (int q = threadIdx.x; q < m * d; q += blockDim.x) tc[q] = t[q];
  for (int q = threadIdx.x; q < m; q += blockDim.x) cc[q] = c[q];
}

// Every point CTA adds a slot to the sums of k_lm_step, one CTA's work, so there are few; from 32 tiles each (1.2
// million points) the pass over the points outweighs that, and four CTAs per SM hide more of its latency (2^22
// points on one axis: m = 1 428 -> 300 us a step, m = 20 942 -> 617).
inline int lm_point_ctas(long long K) {
  const long long tiles = (K + LM_TILE - 1) / LM_TILE;
  return (int)std::min<long long>(tiles, tiles < 32 * LM_CTA ? LM_CTA : LM_MAXCTA);
}
size_t lm_points_smem(int m, int d) {
  return sizeof(float4) * (size_t)m * LM_SEG + sizeof(float2) * ((size_t)m * LM_EP + 2 * LM_TILE) +
         sizeof(float) * (size_t)d * LM_TILE;
}
size_t lm_step_smem(int m, int d) {
  const size_t ld = lm_ld(m * (d + 2));
  return sizeof(float) * (ld * ld + LM_NB * ld + 2 * ld);
}

}  // namespace

// ----------------------------------------------------------------------------- host side
long long lm_workspace_bytes(int m, int d) {
  return 16LL * (LM_SEG + m) + 8LL * LM_MAXCTA * ((long long)m * (d + 1) + 1) +
         8 * (2 * lm_set_elems(m, d) + (long long)m * d) + sizeof(LmState) + 64;
}

// Dynamic shared-memory limits of the refinement kernels.
cudaError_t lm_set_attributes(int m, int d) {
  const cudaError_t e = allow_smem(k_lm_points, lm_points_smem(m, d));
  return e == cudaSuccess ? allow_smem(k_lm_step, lm_step_smem(m, d)) : e;
}

// The whole refinement, enqueued on `s`: 2 iters + 3 launches (the host stays ahead of the device,
// so no graph is kept).
void launch_refine_lm(double* t, double2* c, int m, int d, const int* lo, const int* len, long long K,
                      const float2* y, int iters, double lambda0, double* hist, void* ws, cudaStream_t s) {
  float4* circle = (float4*)ws;
  double2* cc = (double2*)(circle + LM_SEG);
  double* tc = (double*)(cc + m);
  double* ls = tc + m * d;
  float2* vs = (float2*)(ls + LM_MAXCTA);
  double* sets = (double*)(vs + (long long)LM_MAXCTA * m * (d + 1));
  LmState* st = (LmState*)(sets + 2 * lm_set_elems(m, d));
  const Box B = make_box(d, lo, len);
  const size_t sp = lm_points_smem(m, d), ss = lm_step_smem(m, d);
  const int npt = lm_point_ctas(K), npair = m * (m + 1) / 2;
  note_launch();
  k_lm_init<<<1, 256, 0, s>>>(st, lambda0, t, c, tc, cc, circle, m, d);
  for (int it = 0; it <= iters; ++it) {
    note_launch();
    chain_launch(k_lm_points, npt + npair, LM_TILE, sp, s, tc, cc, m, d, B, K, npt, y, st, circle, sets, vs, ls);
    note_launch();
    chain_launch(k_lm_step, 1, LM_SOLVE_THREADS, ss, s, t, c, tc, cc, m, d, st, sets, vs, ls, npt, hist, it, it < iters);
  }
}
