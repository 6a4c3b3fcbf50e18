// Data-parallel kernels over the rows of one or many problems: grid preparation,
// Philox starting block, tall-skinny Gram and products of the block power method
// (Algorithm 3), the Vandermonde right-hand side conj(A) f and the LS residual
// (Eq. ls_probl), and the exponential sum of Eq. 1 with its vector-Jacobian product.
#include "common.cuh"

#include <algorithm>
#include <map>
#include <mutex>

namespace {

__device__ inline const ProbDesc& prob(const Dev& D, int p) { return D.P[p]; }

__device__ inline float2* buf_base(const Dev& D, int buf, const ProbDesc& p, int& ld) {
  switch (buf) {
    case BUF_V: ld = p.N; return D.V + p.xoff;
    case BUF_U: ld = p.N; return D.U + p.xoff;
    case BUF_B1: ld = p.N; return D.B1 + p.xoff;
    case BUF_B2: ld = p.N; return D.B2 + p.xoff;
    default: ld = p.Next; return D.Y + p.yoff;
  }
}

__device__ inline int width_of(const ProbState& s, const ProbDesc& p, int sel) { return sel_width(s, p, sel); }

// Row of buffer `buf` holding row r of I_n (Y is laid out over the box {0..n+1}^d).
__device__ inline int buf_row(int buf, const ProbDesc& p, int r, int shift) {
  return buf == BUF_Y ? map_row(r, p.n, p.d, p.n + 2, shift) : r;
}

template <typename T>
__device__ inline T block_sum(T v, T* sh) {
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  int w = threadIdx.x >> 5, l = threadIdx.x & 31;
  __syncthreads();
  if (l == 0) sh[w] = v;
  __syncthreads();
  T r = 0;
  if (threadIdx.x < 32) {
    r = (l < (int)(blockDim.x >> 5)) ? sh[l] : (T)0;
    for (int o = 16; o > 0; o >>= 1) r += __shfl_xor_sync(0xffffffffu, r, o);
  }
  return r;  // valid in thread 0
}

// ----------------------------------------------------------------------------- grid prep
__global__ void k_state_init(Dev D) {
  int p = blockIdx.x * blockDim.x + threadIdx.x;
  if (p >= D.nprob) return;
  ProbState s = {};
  s.wu = D.P[p].r0;
  s.wv = D.P[p].r0;
  s.rank_det = -1;
  s.rank_used = D.P[p].m;
  s.resid2_prev = -1.0;
  D.st[p] = s;
}

// gF = f, gH(x) = conj f(-x) (zero where -x leaves the grid); ||T||_F^2 by the
// multiplicity of each difference (prod_l (n+1-|x_l|)), ||f||^2 over I_n, finiteness.  A product on
// its own needs the copies only (NORMS = false: no FP64 sums).
template <bool NORMS>
__global__ void k_prep(Dev D) {
  __shared__ double sh[32];
  const int pi = blockIdx.y;
  const ProbDesc& p = D.P[pi];
  double accT = 0.0, accF = 0.0;
  int bad = 0;
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < p.Gd; i += gridDim.x * blockDim.x) {
    int rem = i, mir = 0, mul = 1;
    double w = 1.0;
    bool inT = true, inI = true, mvalid = true;
    for (int l = p.d - 1; l >= 0; --l) {
      int dig = rem % p.G;
      rem /= p.G;
      int x = dig - p.n;
      int ax = x < 0 ? -x : x;
      if (ax > p.n) inT = false; else w *= (double)(p.n + 1 - ax);
      if (x < 0 || x > p.n) inI = false;
      int md = 2 * p.n - dig;  // digit of -x
      if (md < 0) mvalid = false;
      mir += md * mul;
      mul *= p.G;
    }
    double2 f = D.grid64[p.grid + i];
    if (!isfinite(f.x) || !isfinite(f.y)) bad = 1;
    D.gF[p.grid + i] = make_float2((float)f.x, (float)f.y);
    float2 h = make_float2(0.f, 0.f);
    if (mvalid) {
      double2 fm = D.grid64[p.grid + mir];
      h = make_float2((float)fm.x, -(float)fm.y);
    }
    D.gH[p.grid + i] = h;
    if (!NORMS) continue;
    double a2 = f.x * f.x + f.y * f.y;
    if (inT) accT += w * a2;
    if (inI) accF += a2;
  }
  if (bad) atomicOr(&D.st[pi].nonfinite, 1);
  if (!NORMS) return;
  double sT = block_sum(accT, sh);
  double sF = block_sum(accF, sh);
  // block sums in fixed block order
  double2* slot = (double2*)red_region(D, pi);
  if (threadIdx.x == 0 && ws_ok(D, 16LL * (blockIdx.x + 1) <= D.red_stride, 11)) slot[blockIdx.x] = make_double2(sT, sF);
  if (red_arrive(D, pi, gridDim.x) && threadIdx.x == 0) {
    double t2 = 0.0, f2 = 0.0;
    for (int b = 0; b < (int)gridDim.x; ++b) {
      const double2 v = __ldcg(slot + b);
      t2 += v.x;
      f2 += v.y;
    }
    D.st[pi].normT2 = t2;
    D.st[pi].normf2 = f2;
  }
}

// V_0 entry (i, j) = complex normal from Philox counter i*r0 + j (Algorithm 3 start block).
__global__ void k_init_v0(Dev D, unsigned long long seed) {
  const int pi = blockIdx.y;
  const ProbDesc& p = D.P[pi];
  // a thread takes rows, the threads of a warp neighbouring rows of one column at a time
  // (coalesced stores); the counter of entry (row, col) is row * r0 + col
  for (int row = blockIdx.x * blockDim.x + threadIdx.x; row < p.N; row += gridDim.x * blockDim.x)
  for (int col = 0; col < p.r0; ++col) {
    const long long q = (long long)row * p.r0 + col;
    uint64_t c[4] = {(uint64_t)q, 0, 0, 0};
    philox4x64(c, seed, PRONY_STREAM_V0);
    // u = ((w >> 11) + 1/2) 2^-53 rounded to FP32 without FP64 operations (they took most of this kernel:
    // 0.61 ms for 64 blocks of 8000 x 80, now 0.48; 0.41 -> 0.34 for 4096 blocks of d=2, n 7..31)
    float u0 = __ull2float_rn((c[0] >> 11) * 2 + 1) * 5.5511151231257827e-17f;      // 2^-54
    float u1 = __ull2float_rn((c[1] >> 11) * 2 + 1) * 5.5511151231257827e-17f;
    float r = sqrtf(-logf(u0)), sn, cs;
    sincospif(2.0f * u1, &sn, &cs);
    D.V[p.xoff + (long long)col * p.N + row] = make_float2(r * cs, r * sn);
  }
}

// Clears a block of the small workspace of every problem still iterating.
__global__ void k_zero_small(Dev D, long long off, long long bytes) {
  if (D.st[blockIdx.y].done) return;
  const ProbDesc& p = D.P[blockIdx.y];
  unsigned int* b = (unsigned int*)(D.small + p.soff + off);
  for (long long i = blockIdx.x * blockDim.x + threadIdx.x; i < bytes / 4; i += gridDim.x * blockDim.x) b[i] = 0u;
}

// ----------------------------------------------------------------------------- tall-skinny Gram
// out[a][b] = sum_r conj(X[r, a]) Z[r, b] over a block of `chunk` rows (chosen by the launcher so that the
// batch fills the resident blocks: few blocks per problem means few partial Grams to add).
//
// Rows are staged RS at a time through three shared-memory buffers filled by cp.async (two passes in flight while
// one is multiplied; rows past the end are zeros).  A buffer holds the values as they are in memory, column-major,
// with a row pitch of RS + 2: a pair of rows is one 16-byte load, and consecutive columns lie in different banks.
// The products are paired FP32 FMAs on whole values: acc1 += (Re x Re z, Im x Im z) and
// acc2 += (Re x Im z, Im x Re z), with conj(x) z = (acc1.lo + acc1.hi) + i (acc2.lo - acc2.hi) at the end, so that
// nothing but a swap of z is rearranged.  What bounds a 4 x 4 tile is then shared memory and the FP32 pipe about
// equally; values stored as the four floats of two paired operands took twice the loads (64 blocks of 8000 x 80:
// 0.69 ms, now 0.39; a solve of 4096 problems with n 7..31: 5.3 -> 1.9 ms of Gram sums, with blocks of 128 threads).
// Output ownership is interleaved: thread (ti, tj) owns the entries (ti + NA i, tj + NB j),
// i, j < 4, so the threads of a warp read consecutive columns (different banks) or the same one
// (broadcast).  When there are fewer 4x4 tiles than threads, threads split the staged row pairs into
// row groups whose partial sums are added in shared memory; when there are more, the tiles are
// processed in batches (every batch re-stages the rows).  Each block stores its partial Gram; the
// last block of the problem (or k_gram_sum) adds the partials (FP32, a fixed order) and writes the FP64 output.
constexpr int GRAM_T = 4;           // register tile (GRAM_T x GRAM_T entries, two packed sums each)
constexpr int GRAM_STAGES = 3;      // staging buffers
constexpr int GRAM_RED = GRAM_T * GRAM_T + 1;        // pitch of a thread's sums in the group reduction

__host__ __device__ inline int gram_rows(int LR) { return LR <= 40 ? 32 : 16; }
// float2 entries of one staging buffer (sized by the widest blocks of the batch, LR columns)
__host__ __device__ inline int gram_buf_elems(int LR) { return 2 * LR * (gram_rows(LR) + 2); }
// Rows staged per pass for a block of `cols` staged columns: the most (128 down to 8) that fit the buffer.
__device__ inline int gram_rows_for(int cols, int LR) {
  const int cap = gram_buf_elems(LR);
  int rs = 128;
  while (rs > 8 && cols * (rs + 2) > cap) rs >>= 1;
  return rs;
}
// Threads of a block: narrow blocks have few tiles and are bound by latency, so more and smaller blocks per SM
inline int gram_threads(int LR) { return LR <= 24 ? 128 : 256; }

__device__ __forceinline__ unsigned long long pk2(float lo, float hi) {
  unsigned long long r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
  return r;
}
__device__ __forceinline__ float2 upk2(unsigned long long v) {
  float lo, hi;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(v));
  return make_float2(lo, hi);
}
__device__ __forceinline__ unsigned long long swap2(unsigned long long v) {
  unsigned long long r;
  asm("{ .reg .b32 lo, hi; mov.b64 {lo, hi}, %1; mov.b64 %0, {hi, lo}; }" : "=l"(r) : "l"(v));
  return r;
}
__device__ __forceinline__ void ffma2(unsigned long long& acc, unsigned long long a, unsigned long long b) {
  asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(acc) : "l"(a), "l"(b));
}
__device__ __forceinline__ void cp_async8(void* dst, const void* src, bool valid) {   // (zeros when not valid)
  asm volatile("cp.async.ca.shared.global [%0], [%1], 8, %2;"
               ::"r"((unsigned)__cvta_generic_to_shared(dst)), "l"(src), "r"(valid ? 8 : 0)
               : "memory");
}

__global__ void __launch_bounds__(256, 2) k_gram(Dev D, int xbuf, int xshift, int xw, int zbuf, int zshift, int zw,
                                              long long out_off, int out_ld, int chunk, int own_sum) {
  extern __shared__ float4 smem4[];
  const int pi = blockIdx.y;
  const ProbDesc& p = D.P[pi];
  const ProbState& s = D.st[pi];
  if (s.done) return;
  const int a = width_of(s, p, xw), b = width_of(s, p, zw);
  const int r_begin = blockIdx.x * chunk;
  if (r_begin >= p.N || a <= 0 || b <= 0) return;
  const int r_end = min(p.N, r_begin + chunk);
  const int LR = D.L.LDR;
  // X^* X (same buffer, shift and width): the rows are staged once and only the tiles on and
  // above the diagonal are computed, the others written as their conjugate mirrors
  const bool sym = xbuf == zbuf && xshift == zshift && a == b;
  const int ncols = sym ? a : a + b, ZC = sym ? 0 : a;   // staged columns: of X, then of Z
  const int RS = gram_rows_for(ncols, LR), PR = RS + 2;
  const int buf_elems = gram_buf_elems(LR);
  float2* stage = (float2*)smem4;
  float2* red = (float2*)smem4;                    // [RG][per_batch][GRAM_RED], over the buffers once the rows are done
  int ldx, ldz;
  const float2* X = buf_base(D, xbuf, p, ldx);
  const float2* Z = buf_base(D, zbuf, p, ldz);
  const int NA = (a + GRAM_T - 1) / GRAM_T, NB = (b + GRAM_T - 1) / GRAM_T;
  const int ntile = sym ? NA * (NA + 1) / 2 : NA * NB;
  const int nthr = blockDim.x;
  const int per_batch = min(ntile, nthr);
  const int RG = max(1, min(RS / 2, nthr / per_batch));   // row groups (1 when tiles >= threads)
  const int nbatch = (ntile + per_batch - 1) / per_batch;
  double2* out = (double2*)(D.small + p.soff + out_off);
  float2* mine = (float2*)red_region(D, pi) + (size_t)blockIdx.x * a * b;   // this block's partial Gram
  const bool mine_ok = ws_ok(D, 8LL * a * b * (blockIdx.x + 1) <= D.red_stride, 12);
  // staging role: one row, columns c0, c0 + cstep, ...
  const int my_rr = threadIdx.x % RS, c0 = threadIdx.x / RS, cstep = nthr / RS;
  auto issue = [&](int r0, int buf) {
    if (r0 < r_end) {
      const int r = r0 + my_rr;
      const bool ok = r < r_end;
      const float2* x = X + (ok ? buf_row(xbuf, p, r, xshift) : 0);
      const float2* z = Z + (ok && !sym ? buf_row(zbuf, p, r, zshift) : 0);
      float2* dst = stage + (size_t)buf * buf_elems + my_rr;
      for (int col = c0; col < ncols; col += cstep)
        cp_async8(dst + col * PR, col < a ? x + (long long)col * ldx : z + (long long)(col - a) * ldz, ok);
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
  for (int batch = 0; batch < nbatch; ++batch) {
    const int tl = threadIdx.x % per_batch, tile = batch * per_batch + tl, grp = threadIdx.x / per_batch;
    const bool active = grp < RG && tile < ntile;
    int ti = tile / NB, tj = tile % NB;
    if (sym) {                                    // tile -> (ti, tj), ti <= tj, row by row
      ti = 0;
      int rest = min(tile, ntile - 1);
      while (rest >= NA - ti) {
        rest -= NA - ti;
        ++ti;
      }
      tj = ti + rest;
    }
    // offsets of the owned columns in a buffer (entries past a or b read a valid column; their
    // sums are never stored)
    int xo[GRAM_T], zo[GRAM_T];
#pragma unroll
    for (int i = 0; i < GRAM_T; ++i) {
      xo[i] = min(ti + NA * i, a - 1) * PR;
      zo[i] = (min(tj + NB * i, b - 1) + ZC) * PR;
    }
    unsigned long long acc1[GRAM_T][GRAM_T], acc2[GRAM_T][GRAM_T];
#pragma unroll
    for (int i = 0; i < GRAM_T; ++i)
#pragma unroll
      for (int j = 0; j < GRAM_T; ++j) acc1[i][j] = acc2[i][j] = 0ull;
    __syncthreads();                              // the buffers are free (previous batch done)
    issue(r_begin, 0);
    issue(r_begin + RS, 1);
    int buf = 0;
    for (int r0 = r_begin; r0 < r_end; r0 += RS) {
      asm volatile("cp.async.wait_group 1;" ::: "memory");
      __syncthreads();                            // these rows are there; the buffer of the pass before is free
      issue(r0 + 2 * RS, buf == 0 ? 2 : buf - 1);
      const float2* Bs = stage + (size_t)buf * buf_elems;
      if (active) {
        const int npair = (min(RS, r_end - r0) + 1) / 2;
        for (int rp = grp; rp < npair; rp += RG) {
          ulonglong2 xa[GRAM_T], zb[GRAM_T];
#pragma unroll
          for (int i = 0; i < GRAM_T; ++i) xa[i] = *(const ulonglong2*)(Bs + xo[i] + 2 * rp);
#pragma unroll
          for (int j = 0; j < GRAM_T; ++j) zb[j] = *(const ulonglong2*)(Bs + zo[j] + 2 * rp);
#pragma unroll
          for (int j = 0; j < GRAM_T; ++j) {
            const unsigned long long s0 = swap2(zb[j].x), s1 = swap2(zb[j].y);
#pragma unroll
            for (int i = 0; i < GRAM_T; ++i) {
              ffma2(acc1[i][j], xa[i].x, zb[j].x);
              ffma2(acc2[i][j], xa[i].x, s0);
              ffma2(acc1[i][j], xa[i].y, zb[j].y);
              ffma2(acc2[i][j], xa[i].y, s1);
            }
          }
        }
      }
      buf = buf == GRAM_STAGES - 1 ? 0 : buf + 1;
    }
    asm volatile("cp.async.wait_group 0;" ::: "memory");
    // one entry of the block's sums: the tile's (i, j)-th
    auto put = [&](int ti, int tj, int i, int j, float2 v) {
      const int ia = ti + NA * i, jb = tj + NB * j;
      if (mine_ok && ia < a && jb < b) {
        mine[ia * b + jb] = v;
        if (sym && ti != tj) mine[jb * b + ia] = make_float2(v.x, -v.y);   // mirror of a tile above the diagonal
      }
    };
    auto sum_of = [&](int i, int j) {
      const float2 u = upk2(acc1[i][j]), v = upk2(acc2[i][j]);
      return make_float2(u.x + u.y, v.x - v.y);
    };
    if (RG == 1) {
      if (active)
#pragma unroll
        for (int i = 0; i < GRAM_T; ++i)
#pragma unroll
          for (int j = 0; j < GRAM_T; ++j) put(ti, tj, i, j, sum_of(i, j));
    } else {
      // row groups: their sums meet in shared memory and are added in the order of the groups, an entry per
      // thread (there is one batch then)
      __shared__ int s_tile[256];
      __syncthreads();                            // every group is done with the staged rows
      if (active) {
        if (grp == 0) s_tile[tl] = ti | tj << 16;
        float2* dst = red + (size_t)(grp * per_batch + tl) * GRAM_RED;
#pragma unroll
        for (int i = 0; i < GRAM_T; ++i)
#pragma unroll
          for (int j = 0; j < GRAM_T; ++j) dst[i * GRAM_T + j] = sum_of(i, j);
      }
      __syncthreads();
      for (int q = threadIdx.x; q < per_batch * 16; q += nthr) {
        const int t = q >> 4, e = q & 15;
        float2 v = red[(size_t)t * GRAM_RED + e];
        for (int g = 1; g < RG; ++g) {
          const float2 u = red[(size_t)(g * per_batch + t) * GRAM_RED + e];
          v.x += u.x;
          v.y += u.y;
        }
        put(s_tile[t] & 0xffff, s_tile[t] >> 16, e >> 2, e & 3, v);
      }
    }
  }
  // The blocks' partial Grams (one slot of a x b each) added in FP32 in a fixed order: slot k
  // goes to the partial sum k mod 4 of its entry, and the four are combined pairwise.  Each thread
  // takes GR entries at a time, so that 4 GR loads are in flight.  (FP32 sums of at most 64
  // partials add less rounding than each partial already carries from its own rows; FP64
  // additions, at a small fraction of the FP32 rate here, made this one block per problem the
  // longest part of the launch.)
  const int nblk = (p.N + chunk - 1) / chunk;
  if (own_sum && red_arrive(D, pi, nblk)) {
    constexpr int GR = 2;
    const float2* slots = (const float2*)red_region(D, pi);
    const int ss = a * b;
    for (int e0 = threadIdx.x; e0 < ss; e0 += GR * blockDim.x) {
      float2 acc[GR][4];
#pragma unroll
      for (int g = 0; g < GR; ++g)
#pragma unroll
        for (int u = 0; u < 4; ++u) acc[g][u] = make_float2(0.f, 0.f);
      int k = 0;
      for (; k + 4 <= nblk; k += 4) {
        float2 v[GR][4];
#pragma unroll
        for (int g = 0; g < GR; ++g)
#pragma unroll
          for (int u = 0; u < 4; ++u) {
            const int e = e0 + g * blockDim.x;
            v[g][u] = e < ss ? __ldcg(slots + (size_t)(k + u) * ss + e) : make_float2(0.f, 0.f);
          }
#pragma unroll
        for (int g = 0; g < GR; ++g)
#pragma unroll
          for (int u = 0; u < 4; ++u) {
            acc[g][u].x += v[g][u].x;
            acc[g][u].y += v[g][u].y;
          }
      }
#pragma unroll
      for (int u = 0; u < 3; ++u) {                 // the last nblk mod 4 slots
        if (k + u < nblk) {
#pragma unroll
          for (int g = 0; g < GR; ++g) {
            const int e = e0 + g * blockDim.x;
            const float2 v = e < ss ? __ldcg(slots + (size_t)(k + u) * ss + e) : make_float2(0.f, 0.f);
            acc[g][u].x += v.x;
            acc[g][u].y += v.y;
          }
        }
      }
#pragma unroll
      for (int g = 0; g < GR; ++g) {
        const int e = e0 + g * blockDim.x;
        if (e < ss) {
          const float tx = (acc[g][0].x + acc[g][1].x) + (acc[g][2].x + acc[g][3].x);
          const float ty = (acc[g][0].y + acc[g][1].y) + (acc[g][2].y + acc[g][3].y);
          out[(e / b) * out_ld + e % b] = make_double2((double)tx, (double)ty);
        }
      }
    }
  }
}

// The sum of the partial Grams as a launch of its own (k_gram without own_sum): one entry per thread,
// the same order of additions.  With one problem on the GPU and 64 partials, one block took longer over
// them than all blocks over the rows (w = 40: 20 of 28 us; now 3 us in 7 blocks).
__global__ void __launch_bounds__(256) k_gram_sum(Dev D, int xw, int zw, long long out_off, int out_ld, int chunk) {
  const int pi = blockIdx.y;
  const ProbDesc& p = D.P[pi];
  const ProbState& s = D.st[pi];
  if (s.done) return;
  const int a = width_of(s, p, xw), b = width_of(s, p, zw), ss = a * b;
  const int e = blockIdx.x * blockDim.x + threadIdx.x;
  if (a <= 0 || b <= 0 || e >= ss) return;
  const int nblk = (p.N + chunk - 1) / chunk;
  const float2* slots = (const float2*)red_region(D, pi) + e;
  float2 acc[4] = {make_float2(0.f, 0.f), make_float2(0.f, 0.f), make_float2(0.f, 0.f), make_float2(0.f, 0.f)};
  for (int k = 0; k < nblk; k += 16) {               // sixteen loads in flight
    float2 v[16];
#pragma unroll
    for (int u = 0; u < 16; ++u) v[u] = __ldcg(slots + (size_t)min(k + u, nblk - 1) * ss);
#pragma unroll
    for (int u = 0; u < 16; ++u)
      if (k + u < nblk) {
        acc[u & 3].x += v[u].x;
        acc[u & 3].y += v[u].y;
      }
  }
  const float tx = (acc[0].x + acc[1].x) + (acc[2].x + acc[3].x);
  const float ty = (acc[0].y + acc[1].y) + (acc[2].y + acc[3].y);
  ((double2*)(D.small + p.soff + out_off))[(e / b) * out_ld + e % b] = make_double2((double)tx, (double)ty);
}

// ----------------------------------------------------------------------------- X M products
// OUT[r, j] = sum_i X[r, i] M[i][j] (- Z[r, j] with OUT = Z - X M for the residual).  A block
// takes `rows` rows (128, or 64 when the blocks are wide), stages them and M in shared memory
// once, then each thread computes one row and four columns at a time (one X value and four
// broadcast M values per four complex products).  X and OUT may be the same buffer: every
// block reads its rows before writing them.
__global__ void __launch_bounds__(256) k_apply(Dev D, int xbuf, int xw, int outw, long long m_off, int m_double,
                                               int zbuf, int outbuf, int norm_only, int rows) {
  extern __shared__ float2 smem[];
  __shared__ double shr[32];
  const int pi = blockIdx.y;
  const ProbDesc& p = D.P[pi];
  ProbState& s = D.st[pi];
  if (s.done) return;
  const int a = width_of(s, p, xw), b = width_of(s, p, outw);
  const int r0 = blockIdx.x * rows;
  if (r0 >= p.N || b <= 0) return;
  const int ldm = (b + 3) & ~3;                   // M rows padded to whole groups of four columns
  float2* Ms = smem;                              // [a][ldm]
  float2* Xs = smem + (size_t)D.L.LDR * ((D.L.LDR + 3) & ~3);   // [a][rows]
  for (int idx = threadIdx.x; idx < a * ldm; idx += blockDim.x) {
    const int i = idx / ldm, j = idx % ldm;
    float2 v = make_float2(0.f, 0.f);
    if (j < b) {
      if (m_double) {
        const double2 dv = ((const double2*)(D.small + p.soff + m_off))[i * D.L.LDM + j];
        v = make_float2((float)dv.x, (float)dv.y);
      } else {
        v = ((const float2*)(D.small + p.soff + m_off))[i * D.L.LDR + j];
      }
    }
    Ms[idx] = v;
  }
  int ldx;
  const float2* X = buf_base(D, xbuf, p, ldx);
  // a thread stages one row (blockDim.x is a multiple of rows) and every cstep-th column, eight
  // loads in flight at a time
  const int rr = threadIdx.x % rows, cg = threadIdx.x / rows;
  const int ngrp = blockDim.x / rows;
  const int r = r0 + rr;
  {
    const bool ok = r < p.N;
    const int gx = ok ? buf_row(xbuf, p, r, -1) : 0;
    for (int cb = cg; cb < a; cb += 8 * ngrp) {
      float2 v[8];
#pragma unroll
      for (int u = 0; u < 8; ++u) {
        const int col = cb + u * ngrp;
        v[u] = (ok && col < a) ? X[(long long)col * ldx + gx] : make_float2(0.f, 0.f);
      }
#pragma unroll
      for (int u = 0; u < 8; ++u) {
        const int col = cb + u * ngrp;
        if (col < a) Xs[col * rows + rr] = v[u];
      }
    }
  }
  __syncthreads();
  int ldz = 0, ldo = 0;
  const float2* Z = zbuf >= 0 ? buf_base(D, zbuf, p, ldz) : nullptr;
  float2* O = norm_only ? nullptr : buf_base(D, outbuf, p, ldo);
  // squares of a row summed in FP32 (the entries are FP32 values; b <= 128 terms), blocks in FP64
  float nrm = 0.f;
  if (r < p.N) {
    const int gz = Z ? buf_row(zbuf, p, r, -1) : 0;
    const int go = O ? buf_row(outbuf, p, r, -1) : 0;
    for (int j0 = 4 * cg; j0 < b; j0 += 4 * ngrp) {
      float2 zv[4];
#pragma unroll
      for (int e = 0; e < 4; ++e)      // issued before the products so that their latency overlaps them
        zv[e] = (Z && j0 + e < b) ? Z[(long long)(j0 + e) * ldz + gz] : make_float2(0.f, 0.f);
      // x m as paired FP32 FMAs on M as stored: p1 += (Re x, Re x)(Re m, Im m),
      // p2 += (Im x, Im x)(Re m, Im m); then x m = (p1.x - p2.y, p1.y + p2.x)
      unsigned long long p1[4] = {0ull, 0ull, 0ull, 0ull}, p2[4] = {0ull, 0ull, 0ull, 0ull};
      for (int i = 0; i < a; ++i) {
        const float2 x = Xs[i * rows + rr];
        const unsigned long long xr = pk2(x.x, x.x), xi = pk2(x.y, x.y);
        const unsigned long long* mrow = (const unsigned long long*)(Ms + i * ldm + j0);
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          const unsigned long long mm = mrow[e];
          ffma2(p1[e], xr, mm);
          ffma2(p2[e], xi, mm);
        }
      }
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        const int j = j0 + e;
        if (j >= b) break;
        const float2 q1 = upk2(p1[e]), q2 = upk2(p2[e]);
        float2 v = make_float2(q1.x - q2.y, q1.y + q2.x);
        if (Z) {
          v.x = zv[e].x - v.x;
          v.y = zv[e].y - v.y;
        }
        if (norm_only) nrm = fmaf(v.x, v.x, fmaf(v.y, v.y, nrm));
        else O[(long long)j * ldo + go] = v;
      }
    }
  }
  if (norm_only) {
    double t = block_sum((double)nrm, shr);
    double* slot = (double*)red_region(D, pi);
    if (threadIdx.x == 0 && ws_ok(D, 8LL * (blockIdx.x + 1) <= D.red_stride, 13)) slot[blockIdx.x] = t;
    const int nblk = (p.N + rows - 1) / rows;
    if (red_arrive(D, pi, nblk)) {
      // the block sums in a fixed order: thread i adds slots i, i + 256, ..., then a block sum
      double r2 = 0.0;
      for (int k = threadIdx.x; k < nblk; k += blockDim.x) r2 += __ldcg(slot + k);
      r2 = block_sum(r2, shr);
      if (threadIdx.x == 0) s.resid2 = r2;
    }
  }
}

// Largest-modulus row of each of the first m columns (lowest row on ties).
__global__ void k_argmax(Dev D, int buf) {
  const int pi = blockIdx.y;
  const ProbDesc& p = D.P[pi];
  const ProbState& s = D.st[pi];
  int ld;
  const float2* X = buf_base(D, buf, p, ld);
  unsigned long long* am = (unsigned long long*)(D.small + p.soff + D.L.argmx);
  if (s.done) return;
  const int w = min(s.wv, p.m);                 // argmx holds LDM >= m entries
  for (int j = 0; j < w; ++j) {
    unsigned long long best = 0ull;
    for (int r = blockIdx.x * blockDim.x + threadIdx.x; r < p.N; r += gridDim.x * blockDim.x) {
      float2 v = X[(long long)j * ld + r];
      float a2 = v.x * v.x + v.y * v.y;
      unsigned long long key = ((unsigned long long)__float_as_uint(a2) << 32) | (0xFFFFFFFFull - (unsigned)r);
      best = key > best ? key : best;
    }
    for (int o = 16; o > 0; o >>= 1) {
      unsigned long long oth = __shfl_xor_sync(0xffffffffu, best, o);
      best = oth > best ? oth : best;
    }
    if ((threadIdx.x & 31) == 0) atomicMax(&am[j], best);
  }
}

// ----------------------------------------------------------------------------- Vandermonde right-hand side
// The sums of Eq. ls_probl factorise over the axes.  k_powers tabulates E_l[x][i] = e^{2 pi i t_i(l) x}
// (or conj(z~_i(l))^x with the raw eigenvalues) for x in {0..n}, FP64, once per problem.  A unit of work
// is a piece of at most RHS_SEG points of a line of the last axis:
//   k_rhs<false>  conj(A) f: a thread sums f(k) E_{d-1}[k_{d-1}][i] over the points of a unit for one term i and
//                 multiplies by the powers of the other axes once;
//   k_rhs<true>   ||A^T c - f||: a block forms c_i times the conjugate powers of the other axes per unit, and a
//                 thread sums the terms at one point.
// Either way a point and term take four FP64 FMAs instead of 4 d (the FP64 pipe, two FMAs per clock and
// SM, bounds both), and the powers come without a chain of n dependent products per block: 64 problems
// d = 3, n = 19, m = 40: 0.69 ms each before, now 0.32 (floor of the FP64 operations 0.14); one problem of
// n = 63, m = 20: 100 us each before, now 16.
constexpr int RHS_SEG = 16;             // points of a unit
constexpr int RHS_THREADS = 128;

// The same launch evaluates the Gram matrix conj(A) A^T (its lower triangle) over the whole GPU for k_solve_c
// (there, one CTA per problem computed all m^2 entries: FP64 sincospi is what it spent its time on):
//   G_ij = prod_l sum_{x=0}^{n} exp(2 pi i (t_i(l) - t_j(l)) x), or with the raw eigenvalues
//   prod_l sum_x (conj(z_i(l)) z_j(l))^x (summed term by term: |q| need not be 1).
__global__ void k_powers(Dev D) {
  const int pi = blockIdx.y;
  const ProbDesc& p = D.P[pi];
  const ProbState& s = D.st[pi];
  const int m = s.rank_used, n1 = p.n + 1;
  if (s.done || m <= 0 || m > p.m) return;
  double2* E = D.zpow + pi * D.zpow_stride;
  double2* G = (double2*)(D.small + p.soff + D.L.gram);              // packed: i (i + 1) / 2 + j, j <= i
  const double2* zr = (const double2*)(D.small + p.soff + D.L.zraw);
  const double* t = (const double*)(D.small + p.soff + D.L.t);
  const int ntri = m * (m + 1) / 2, npow = D.vand ? p.d * m : p.d * n1 * m;
  for (int q = blockIdx.x * blockDim.x + threadIdx.x; q < ntri + npow; q += gridDim.x * blockDim.x) {
    if (q < ntri) {
      int i = (int)((sqrtf(8.f * q + 1.f) - 1.f) * 0.5f);
      if (i * (i + 1) / 2 > q) --i;
      if ((i + 1) * (i + 2) / 2 <= q) ++i;
      const int j = q - i * (i + 1) / 2;
      double2 g = make_double2(1.0, 0.0);
      for (int l = 0; l < p.d; ++l) {
        double2 term;
        if (D.vand) {
          const double2 w = cmulc(zr[i * PRONY_DMAX + l], zr[j * PRONY_DMAX + l]);
          double2 pw = make_double2(1.0, 0.0);
          term = make_double2(1.0, 0.0);
          for (int x = 1; x <= p.n; ++x) {
            pw = cmul(pw, w);
            term = cadd(term, pw);
          }
        } else {
          double dl = t[i * PRONY_DMAX + l] - t[j * PRONY_DMAX + l];
          dl -= rint(dl);
          if (dl == 0.0) {
            term = make_double2((double)n1, 0.0);
          } else {
            const double num = sinpi(dl * n1), den = sinpi(dl);
            double sn, cs;
            sincospi(dl * p.n, &sn, &cs);
            term = cscale(make_double2(cs, sn), num / den);
          }
        }
        g = cmul(g, term);
      }
      G[q] = g;
      continue;
    }
    const int e = q - ntri;
    if (D.vand) {
      const int l = e / m, i = e % m;
      const double2 e1 = cconj(zr[i * PRONY_DMAX + l]);
      double2 v = make_double2(1.0, 0.0);
      for (int x = 0; x < n1; ++x) {
        E[((size_t)l * n1 + x) * m + i] = v;
        v = cmul(v, e1);
      }
    } else {
      const int i = e % m, x = e / m % n1, l = e / m / n1;
      double ph = t[i * PRONY_DMAX + l] * x, sn, cs;
      ph = fma(t[i * PRONY_DMAX + l], (double)x, -rint(ph));       // reduced with one rounding
      sincospi(2.0 * ph, &sn, &cs);
      E[e] = make_double2(cs, sn);
    }
  }
}

// Unit u of a problem: line and first point of the last axis (nseg pieces per line).
__device__ inline long long rhs_unit(const ProbDesc& p, int u, int nseg, int& line, int& x0) {
  line = u / nseg;
  x0 = (u - line * nseg) * RHS_SEG;
  long long g = 0, mul = 1;
  int rem = line;
  g = x0 + p.n;
  mul = p.G;
  for (int l = p.d - 2; l >= 0; --l) {
    g += (long long)(rem % (p.n + 1) + p.n) * mul;
    rem /= p.n + 1;
    mul *= p.G;
  }
  return p.grid + g;                                  // grid index of the unit's first sample
}

// `upb` units per block.
template <bool RESID>
__global__ void __launch_bounds__(RHS_THREADS) k_rhs(Dev D, int upb) {
  __shared__ double2 sh[PRONY_MMAX * (RHS_THREADS / RHS_SEG) + RHS_THREADS];
  __shared__ double shr[32];
  const int pi = blockIdx.y;
  const ProbDesc& p = D.P[pi];
  ProbState& s = D.st[pi];
  const int m = s.rank_used;
  if (s.done || m <= 0 || m > p.m) return;
  const int n1 = p.n + 1, nseg = (n1 + RHS_SEG - 1) / RHS_SEG, nunit = p.N / n1 * nseg;
  const int u0 = blockIdx.x * upb, u1 = min(nunit, u0 + upb);
  if (u0 >= nunit) return;
  const int nblk = (nunit + upb - 1) / upb;
  const double2* E = D.zpow + pi * D.zpow_stride;
  const double2* last = E + (size_t)(p.d - 1) * n1 * m;
  // product over the leading axes of the powers of term i at a line
  auto lead = [&](int line, int i) {
    double2 e = make_double2(1.0, 0.0);
    for (int l = p.d - 2; l >= 0; --l) {
      const double2 v = E[((size_t)l * n1 + line % n1) * m + i];
      e = l == p.d - 2 ? v : cmul(e, v);
      line /= n1;
    }
    return e;
  };
  if (!RESID) {
    const int groups = RHS_THREADS / m;               // m <= 64: at least two
    const int i = threadIdx.x % m, grp = threadIdx.x / m;
    double2 b = make_double2(0.0, 0.0);
    if (grp < groups)
      for (int u = u0 + grp; u < u1; u += groups) {
        int line, x0;
        const double2* f = D.grid64 + rhs_unit(p, u, nseg, line, x0);
        const double2* w = last + (size_t)x0 * m + i;
        const int nx = min(RHS_SEG, n1 - x0);
        double2 a = make_double2(0.0, 0.0);
#pragma unroll 4
        for (int x = 0; x < nx; ++x) {
          const double2 fv = f[x], wv = w[(size_t)x * m];
          a.x = fma(fv.x, wv.x, fma(-fv.y, wv.y, a.x));
          a.y = fma(fv.x, wv.y, fma(fv.y, wv.x, a.y));
        }
        b = cadd(b, p.d > 1 ? cmul(a, lead(line, i)) : a);
      }
    sh[threadIdx.x] = b;
    __syncthreads();
    double2* out = (double2*)(D.small + p.soff + D.L.rhs);
    double2* slots = (double2*)red_region(D, pi);
    if (grp == 0 && ws_ok(D, 16LL * m * (blockIdx.x + 1) <= D.red_stride, 14)) {
      for (int g = 1; g < groups; ++g) b = cadd(b, sh[g * m + i]);
      slots[(size_t)blockIdx.x * m + i] = b;
    }
    // block sums in block order
    if (red_arrive(D, pi, nblk) && threadIdx.x < m) {
      double2 sum = make_double2(0.0, 0.0);
#pragma unroll 4
      for (int k = 0; k < nblk; ++k) sum = cadd(sum, __ldcg(slots + (size_t)k * m + threadIdx.x));
      out[threadIdx.x] = sum;
    }
  } else {
    const double2* c = (const double2*)(D.small + p.soff + D.L.rhs);   // in the order of the powers (k_solve_c)
    constexpr int PER = RHS_THREADS / RHS_SEG;        // units at a time
    double r2 = 0.0;
    for (int v0 = u0; v0 < u1; v0 += PER) {
      const int nv = min(PER, u1 - v0);
      __syncthreads();
      for (int q = threadIdx.x; q < nv * m; q += RHS_THREADS) {   // c_i conj(powers of the leading axes)
        const int line = (v0 + q / m) / nseg, i = q % m;
        sh[q] = p.d > 1 ? cmulc(lead(line, i), c[i]) : c[i];
      }
      __syncthreads();
      const int v = threadIdx.x / RHS_SEG, dx = threadIdx.x % RHS_SEG;
      if (v < nv) {
        int line, x0;
        const double2* f = D.grid64 + rhs_unit(p, v0 + v, nseg, line, x0);
        if (x0 + dx < n1) {
          const double2* w = last + (size_t)(x0 + dx) * m;
          const double2* cu = sh + v * m;
          const double2 fv = f[dx];
          double2 a = make_double2(-fv.x, -fv.y), a1 = make_double2(0.0, 0.0);   // two chains over the terms
#pragma unroll 2
          for (int i = 0; i < m; i += 2) {
            const double2 c0 = cu[i], w0 = w[i];
            a.x = fma(c0.x, w0.x, fma(c0.y, w0.y, a.x));          // c conj(w)
            a.y = fma(c0.y, w0.x, fma(-c0.x, w0.y, a.y));
            if (i + 1 < m) {
              const double2 c1 = cu[i + 1], w1 = w[i + 1];
              a1.x = fma(c1.x, w1.x, fma(c1.y, w1.y, a1.x));
              a1.y = fma(c1.y, w1.x, fma(-c1.x, w1.y, a1.y));
            }
          }
          r2 += cabs2(cadd(a, a1));
        }
      }
    }
    const double tot = block_sum(r2, shr);
    double* slot = (double*)red_region(D, pi);
    if (threadIdx.x == 0 && ws_ok(D, 8LL * (blockIdx.x + 1) <= D.red_stride, 15)) slot[blockIdx.x] = tot;
    if (red_arrive(D, pi, nblk)) {
      double sum = 0.0;                               // lane sums in lane order, then a fixed tree
      for (int k = threadIdx.x; k < nblk; k += RHS_THREADS) sum += __ldcg(slot + k);
      sum = block_sum(sum, shr);
      if (threadIdx.x == 0) s.ls_num2 = sum;
    }
  }
}

// Packed outputs: t_out[(ooff + j) d + l], c_out[ooff + j]; entries past rank_used are zero.
__global__ void k_gather_out(Dev D, double* t_out, double2* c_out) {
  const int pi = blockIdx.x;
  const ProbDesc& p = D.P[pi];
  const ProbState& s = D.st[pi];
  const double* t = (const double*)(D.small + p.soff + D.L.t);
  const double2* c = (const double2*)(D.small + p.soff + D.L.c);
  for (int q = threadIdx.x; q < p.m * p.d; q += blockDim.x) {
    int j = q / p.d, l = q % p.d;
    t_out[(p.ooff + j) * D.maxD + l] = j < s.rank_used ? t[j * PRONY_DMAX + l] : 0.0;
  }
  for (int j = threadIdx.x; j < p.m; j += blockDim.x)
    c_out[p.ooff + j] = j < s.rank_used ? c[j] : make_double2(0.0, 0.0);
}

__global__ void k_copy_cols(Dev D, int buf, int wsel, double2* out) {
  const ProbDesc& p = D.P[0];
  const ProbState& s = D.st[0];
  int ld;
  const float2* X = buf_base(D, buf, p, ld);
  const int w = width_of(s, p, wsel);
  for (long long q = blockIdx.x * (long long)blockDim.x + threadIdx.x; q < (long long)p.N * p.m;
       q += (long long)gridDim.x * blockDim.x) {
    int col = (int)(q / p.N), r = (int)(q % p.N);
    float2 v = col < w ? X[(long long)col * ld + r] : make_float2(0.f, 0.f);
    out[q] = make_double2(v.x, v.y);
  }
}

// ----------------------------------------------------------------------------- exponential sum (Eq. 1)
__global__ void __launch_bounds__(256) k_expsum_fwd(const double* t, const float2* c, int m, int d, Box B,
                                                    long long K, float2* f) {
  __shared__ uint64_t T[PRONY_MMAX * PRONY_DMAX];
  __shared__ float2 cs[PRONY_MMAX];
  for (int q = threadIdx.x; q < m * d; q += blockDim.x) T[q] = frac64(t[q]);
  for (int q = threadIdx.x; q < m; q += blockDim.x) cs[q] = c[q];
  __syncthreads();
  for (long long q = blockIdx.x * (long long)blockDim.x + threadIdx.x; q < K; q += (long long)gridDim.x * blockDim.x) {
    int k[PRONY_DMAX];
    box_point(B, d, q, k);
    float2 acc = make_float2(0.f, 0.f);
    for (int j = 0; j < m; ++j) {
      float u = centred_phase(T + j * d, k, d), sn, cn;
      sincospif(2.0f * u, &sn, &cn);                  // e = cn - i sn
      float2 cj = cs[j];
      acc.x += cj.x * cn + cj.y * sn;
      acc.y += cj.y * cn - cj.x * sn;
    }
    f[q] = acc;
  }
}

// acc[j][0..1] += sum_k g_k conj(e_jk);  acc[j][2+l] += sum_k k_l Im(conj(g_k) c_j e_jk)
__global__ void __launch_bounds__(256) k_expsum_bwd(const double* t, const float2* c, int m, int d, Box B,
                                                    long long K, const float2* g, double* acc) {
  __shared__ uint64_t T[PRONY_MMAX * PRONY_DMAX];
  __shared__ float2 cs[PRONY_MMAX];
  __shared__ float blk[PRONY_MMAX * (2 + PRONY_DMAX)];
  const int W = 2 + d;
  for (int q = threadIdx.x; q < m * d; q += blockDim.x) T[q] = frac64(t[q]);
  for (int q = threadIdx.x; q < m; q += blockDim.x) cs[q] = c[q];
  for (int q = threadIdx.x; q < m * W; q += blockDim.x) blk[q] = 0.f;
  __syncthreads();
  for (long long base = blockIdx.x * (long long)blockDim.x; base < K; base += (long long)gridDim.x * blockDim.x) {
    long long q = base + threadIdx.x;
    int k[PRONY_DMAX] = {0, 0, 0, 0};
    float2 gk = make_float2(0.f, 0.f);
    if (q < K) {
      box_point(B, d, q, k);
      gk = g[q];
    }
    for (int j = 0; j < m; ++j) {
      float u = centred_phase(T + j * d, k, d), sn, cn;
      sincospif(2.0f * u, &sn, &cn);
      float2 e = make_float2(cn, -sn);
      float gcx = gk.x * e.x + gk.y * e.y;            // g conj(e)
      float gcy = gk.y * e.x - gk.x * e.y;
      float2 ce = make_float2(cs[j].x * e.x - cs[j].y * e.y, cs[j].x * e.y + cs[j].y * e.x);
      float im = gk.x * ce.y - gk.y * ce.x;           // Im(conj(g) c e)
      float v[2 + PRONY_DMAX] = {gcx, gcy, im * k[0], im * k[1], im * k[2], im * k[3]};
#pragma unroll
      for (int w = 0; w < 2 + PRONY_DMAX; ++w) {
        if (w >= W) break;
        float x = v[w];
        for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
        if ((threadIdx.x & 31) == 0) atomicAdd(&blk[j * W + w], x);
      }
    }
  }
  __syncthreads();
  for (int q = threadIdx.x; q < m * W; q += blockDim.x) atomicAdd(&acc[q], (double)blk[q]);
}

__global__ void k_expsum_bwd_finish(const double* acc, int m, int d, double* gt, float2* gc) {
  const int W = 2 + d;
  const double two_pi = 6.283185307179586;
  for (int j = threadIdx.x; j < m; j += blockDim.x) {
    gc[j] = make_float2((float)acc[j * W], (float)acc[j * W + 1]);
    for (int l = 0; l < d; ++l) gt[j * d + l] = two_pi * acc[j * W + 2 + l];
  }
}

__global__ void k_eval_points(const double* t, const double2* c, int m, int d, const int* k, int K, double2* f) {
  for (long long q = blockIdx.x * blockDim.x + threadIdx.x; q < K; q += gridDim.x * blockDim.x) {   // (K up to 2^31 - 1)
    double2 acc = make_double2(0.0, 0.0);
    for (int j = 0; j < m; ++j) {
      uint64_t a = 0;
      for (int l = 0; l < d; ++l) a += frac64(t[j * d + l]) * (uint64_t)(long long)k[q * d + l];
      double u = (double)(long long)a * 5.421010862427522e-20;   // 2^-64
      double sn, cn;
      sincospi(2.0 * u, &sn, &cn);
      acc = cadd(acc, cmul(c[j], make_double2(cn, -sn)));
    }
    f[q] = acc;
  }
}

// The same for many points, with fewer FP64 operations per term (GB300 does ~2 FP64 FMAs per clock
// and SM, and sincospi takes a few dozen): exp(-2 pi i u) = T64[hi] T14[mid] (1 + eps) with the 14 leading
// bits of the phase (rounded) as hi and mid and |eps| <= 2 pi 2^-15 from two short Taylor polynomials
// (the terms left out are below 1e-20).  c_j T64 and T14 come from k_eval_tables; 14 FP64 operations per
// term.  65536 points, m = 40: 338 us with sincospi per term, now 109 us and 3.5 us for the tables (the
// FP64 pipe's floor for 14 operations a term is about 60 us), the whole host call 408 -> 179 us.
constexpr int EV_HI = 64, EV_MID = 256;
constexpr int EV_MANY = 12;           // terms from which the tables serve few points too
// tab: c_j exp(-2 pi i q / 64) at j * 64 + q, then exp(-2 pi i q / 2^14), q < 256
__global__ void k_eval_tables(const double2* c, int m, double2* tab) {
  for (int q = blockIdx.x * blockDim.x + threadIdx.x; q < m * EV_HI + EV_MID; q += gridDim.x * blockDim.x) {
    const bool hi = q < m * EV_HI;
    double sn, cn;
    sincospi(hi ? 2.0 * (q % EV_HI) / EV_HI : 2.0 * (q - m * EV_HI) / (EV_HI * EV_MID), &sn, &cn);
    const double2 e = make_double2(cn, -sn);
    tab[q] = hi ? cmul(c[q / EV_HI], e) : e;
  }
}
__global__ void __launch_bounds__(128) k_eval_many(const double* t, const double2* tab, int m, int d, const int* k,
                                                   int K, double2* f) {
  extern __shared__ double2 ev_tab[];
  __shared__ uint64_t T[PRONY_MMAX * PRONY_DMAX];
  for (int q = threadIdx.x; q < m * EV_HI + EV_MID; q += blockDim.x) ev_tab[q] = tab[q];
  for (int q = threadIdx.x; q < m * d; q += blockDim.x) T[q] = frac64(t[q]);
  __syncthreads();
  const double2* mid = ev_tab + m * EV_HI;
  for (long long q = blockIdx.x * blockDim.x + threadIdx.x; q < K; q += gridDim.x * blockDim.x) {
    uint64_t kq[PRONY_DMAX];
#pragma unroll
    for (int l = 0; l < PRONY_DMAX; ++l) kq[l] = l < d ? (uint64_t)(long long)k[q * d + l] : 0;
    double2 acc[2] = {make_double2(0.0, 0.0), make_double2(0.0, 0.0)};   // even and odd terms
#pragma unroll 2
    for (int j = 0; j < m; ++j) {
      uint64_t ph = 0;
#pragma unroll
      for (int l = 0; l < PRONY_DMAX; ++l)
        if (l < d) ph += T[j * d + l] * kq[l];
      const uint64_t seg = (ph + (1ull << 49)) >> 50;                       // 14 bits, mod 2^14
      const double x = (double)(long long)(ph - (seg << 50)) * 3.4061215800865545e-19;   // 2 pi 2^-64
      const double x2 = x * x;
      const double sn = x * fma(x2, -1.0 / 6.0, 1.0), cm = x2 * fma(x2, 1.0 / 24.0, -0.5);
      const double2 b = mid[seg & 255], a = ev_tab[j * EV_HI + (int)((seg >> 8) & 63)];
      const double2 w = make_double2(b.x + fma(b.x, cm, b.y * sn), b.y + fma(b.y, cm, -b.x * sn));   // b (1 + cm - i sn)
      double2& s = acc[j & 1];
      s.x = fma(a.x, w.x, fma(-a.y, w.y, s.x));
      s.y = fma(a.x, w.y, fma(a.y, w.x, s.y));
    }
    f[q] = cadd(acc[0], acc[1]);
  }
}

inline int blocks_for(long long n, int per) { return (int)std::min<long long>((n + per - 1) / per, 1 << 16); }

}  // namespace

#include <algorithm>

void launch_prep(const Dev& D, bool norms, cudaStream_t s) {
  note_launch();
  k_state_init<<<(D.nprob + 127) / 128, 128, 0, s>>>(D);
  note_launch();
  dim3 g(blocks_per_problem(std::min((D.maxGd + 255) / 256, 64), D.nprob), D.nprob);
  if (norms) k_prep<true><<<g, 256, 0, s>>>(D);
  else k_prep<false><<<g, 256, 0, s>>>(D);
}

void launch_init_v0(const Dev& D, unsigned long long seed, cudaStream_t s) {
  dim3 g(blocks_per_problem(std::min((D.maxN + 255) / 256, 256), D.nprob), D.nprob);
  note_launch();
  k_init_v0<<<g, 256, 0, s>>>(D, seed);
}

void launch_zero_small(const Dev& D, long long off, long long bytes, cudaStream_t s) {
  dim3 g(blocks_per_problem(std::min<long long>((bytes / 4 + 255) / 256, 32), D.nprob), D.nprob);
  note_launch();
  k_zero_small<<<g, 256, 0, s>>>(D, off, bytes);
}

// Blocks of k_gram resident on the current device with `sm` bytes of shared memory each.
static int gram_slots(int nthr, size_t sm) {
  static std::mutex lock;
  static std::map<std::pair<int, size_t>, int> known;   // (device, shared memory)
  int dev = 0, occ = 1, sms = 1;
  cudaGetDevice(&dev);
  std::lock_guard<std::mutex> hold(lock);
  int& slots = known[{dev, sm}];
  if (slots) return slots;
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  allow_smem(k_gram, sm);
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, k_gram, nthr, sm) != cudaSuccess) {
    cudaGetLastError();
    occ = 2;
  }
  return slots = std::max(1, occ) * sms;
}

// Launch geometry of k_gram for a batch: dynamic shared memory, rows per block and blocks per
// problem (the batch fills the resident blocks once or twice, at least RS rows per block).
static void gram_geometry(const Dev& D, size_t& sm, int& chunk, int& nblk) {
  // the staging buffers (float2 per value); afterwards the same space holds the sums of the row groups, at most
  // one thread's per thread
  const int RS = gram_rows(D.L.LDR), nthr = gram_threads(D.L.LDR);
  sm = sizeof(float2) * std::max<size_t>((size_t)GRAM_STAGES * gram_buf_elems(D.L.LDR), (size_t)nthr * GRAM_RED);
  // at most 64 blocks per problem: the last block of a problem adds every block's partial Gram
  const int np = std::max(1, D.nprob), slots = gram_slots(nthr, sm);
  int per_prob = std::max(1, std::min(64, slots / np));
  // (a whole number per problem that leaves over a tenth of the resident blocks empty: two rounds of half the rows)
  if ((long long)np * per_prob * 10 < 9LL * slots && per_prob < 64) per_prob = std::min(64, 2 * slots / np);
  chunk = std::max(RS, (D.maxN + per_prob - 1) / per_prob);
  chunk = (chunk + RS - 1) / RS * RS;
  nblk = (D.maxN + chunk - 1) / chunk;
}

// Units of the largest problem, and units per block: about eight blocks per SM over the batch, at most
// 256 blocks per problem (the last one adds their sums).
static int rhs_units_per_block(const Dev& D) {
  const long long total = (long long)D.maxUnits * D.nprob;
  const long long want = std::max<long long>(1, total / (8 * 152));
  return (int)std::max<long long>(std::max<long long>(RHS_THREADS / RHS_SEG, want), (D.maxUnits + 255) / 256);
}
int rhs_units(const ProbDesc& p) { return p.N / (p.n + 1) * ((p.n + RHS_SEG) / RHS_SEG); }

long long red_bytes_per_problem(const Dev& D) {
  size_t sm;
  int chunk, nblk;
  gram_geometry(D, sm, chunk, nblk);
  long long b = (long long)nblk * D.L.LDR * D.L.LDR * (long long)sizeof(float2);           // k_gram
  b = std::max<long long>(b, 64LL * sizeof(double2));                                         // k_prep (<= 64 blocks)
  b = std::max<long long>(b, (D.maxN + 63) / 64 * (long long)sizeof(double));                // k_apply norms
  b = std::max<long long>(b, (D.maxUnits + rhs_units_per_block(D) - 1) / rhs_units_per_block(D) *
                                 (long long)std::max(1, D.L.LDM) * (long long)sizeof(double2));   // k_rhs
  return (b + 255) / 256 * 256;
}

void launch_gram(const Dev& D, int xbuf, int xshift, int xw, int zbuf, int zshift, int zw, long long out_off,
                 int out_ld, cudaStream_t s) {
  size_t sm;
  int chunk, nblk;
  gram_geometry(D, sm, chunk, nblk);
  allow_smem(k_gram, sm);
  dim3 g(nblk, D.nprob);
  note_launch();
  const int own_sum = nblk <= 8;                 // few partials: the last block adds them
  k_gram<<<g, gram_threads(D.L.LDR), sm, s>>>(D, xbuf, xshift, xw, zbuf, zshift, zw, out_off, out_ld, chunk, own_sum);
  if (!own_sum) {
    note_launch();
    k_gram_sum<<<dim3((D.L.LDR * D.L.LDR + 255) / 256, D.nprob), 256, 0, s>>>(D, xw, zw, out_off, out_ld, chunk);
  }
}

void launch_apply(const Dev& D, int xbuf, int xw, int outw, long long m_off, int m_double, int zbuf, int outbuf,
                  int norm_only, cudaStream_t s) {
  const int rows = D.L.LDR <= 64 ? 128 : 64;
  const size_t sm = sizeof(float2) * ((size_t)D.L.LDR * ((D.L.LDR + 3) & ~3) + (size_t)D.L.LDR * rows);
  allow_smem(k_apply, sm);
  dim3 g((D.maxN + rows - 1) / rows, D.nprob);
  note_launch();
  k_apply<<<g, 256, sm, s>>>(D, xbuf, xw, outw, m_off, m_double, zbuf, outbuf, norm_only, rows);
}

void launch_argmax(const Dev& D, int buf, cudaStream_t s) {
  dim3 g(std::max(1, std::min((D.maxN + 255) / 256, 64)), D.nprob);
  note_launch();
  k_argmax<<<g, 256, 0, s>>>(D, buf);
}

void launch_powers(const Dev& D, cudaStream_t s) {
  note_launch();
  const int ntri = D.maxM * (D.maxM + 1) / 2;
  const int want = (int)(((D.vand ? (long long)D.maxD * D.maxM : D.zpow_stride) + ntri + 127) / 128);
  k_powers<<<dim3(blocks_per_problem(want, D.nprob), D.nprob), 128, 0, s>>>(D);
}
void launch_rhs(const Dev& D, int resid, cudaStream_t s) {
  const int upb = rhs_units_per_block(D);
  dim3 g((D.maxUnits + upb - 1) / upb, D.nprob);
  note_launch();
  if (resid) k_rhs<true><<<g, RHS_THREADS, 0, s>>>(D, upb);
  else k_rhs<false><<<g, RHS_THREADS, 0, s>>>(D, upb);
}

void launch_gather_out(const Dev& D, double* t_out, double2* c_out, cudaStream_t s) {
  note_launch();
  k_gather_out<<<D.nprob, 128, 0, s>>>(D, t_out, c_out);
}

void launch_copy_cols(const Dev& D, int buf, int w_sel, double2* out, cudaStream_t s) {
  note_launch();
  k_copy_cols<<<64, 256, 0, s>>>(D, buf, w_sel, out);
}

void launch_expsum_fwd(const double* t, const float2* c, int m, int d, const int* lo, const int* len, long long K,
                       float2* f, cudaStream_t s) {
  note_launch();
  k_expsum_fwd<<<blocks_for(K, 256), 256, 0, s>>>(t, c, m, d, make_box(d, lo, len), K, f);
}

void launch_expsum_bwd(const double* t, const float2* c, int m, int d, const int* lo, const int* len, long long K,
                       const float2* g, double* acc, cudaStream_t s) {
  int nb = std::min(blocks_for(K, 256), 4 * 152);
  note_launch();
  k_expsum_bwd<<<nb, 256, 0, s>>>(t, c, m, d, make_box(d, lo, len), K, g, acc);
}

void launch_expsum_bwd_finish(const double* acc, int m, int d, double* gt, float2* gc, cudaStream_t s) {
  note_launch();
  k_expsum_bwd_finish<<<1, 64, 0, s>>>(acc, m, d, gt, gc);
}

size_t eval_table_bytes(int m) { return sizeof(double2) * ((size_t)m * EV_HI + EV_MID); }

// tab: eval_table_bytes(m) of scratch.  The tables cost a launch more, m * 64 exponentials and their copy into shared
// memory, 5 to 8 us in all; what they save is half of the FP64 work and, for many terms, a chain of m exponentials per
// point.  Few terms therefore take them from 65536 exponentials on (K = 65536, m = 1: 111 us directly, 105 with
// tables; half as many points: 74 and 77), twelve and more from 8192 (K = 512, m = 16: 66 and 52 us).
cudaError_t launch_eval_points(const double* t, const double2* c, int m, int d, const int* k, int K, double2* f,
                               double2* tab, cudaStream_t s) {
  if ((long long)K * m < (m >= EV_MANY ? 8192 : 65536)) {
    note_launch();
    k_eval_points<<<blocks_for(K, 128), 128, 0, s>>>(t, c, m, d, k, K, f);
    return cudaGetLastError();
  }
  const size_t sm = eval_table_bytes(m);
  const cudaError_t e = allow_smem(k_eval_many, sm);
  if (e != cudaSuccess) return e;
  note_launch();
  k_eval_tables<<<(m * EV_HI + EV_MID + 63) / 64, 64, 0, s>>>(c, m, tab);
  note_launch();
  k_eval_many<<<std::min(blocks_for(K, 128), 4 * 152), 128, sm, s>>>(t, tab, m, d, k, K, f);
  return cudaGetLastError();
}
