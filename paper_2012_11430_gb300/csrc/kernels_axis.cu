// Toeplitz block products with the leading axis diagonalised by a DFT.
//
// T = [f(k - h)] is block Toeplitz in the leading axis: with f(x_0, x') placed at x_0 mod L,
// L = 2n + 2, the differences k_0 - h_0 of rows k_0 in {0..n+1} and columns h_0 in {0..n} land on
// points of their own, so
//   Y[k_0, k'] = (1/L) sum_w e^{2 pi i w k_0 / L} sum_h' F^(w; k' - h') X^(w; h'),
// F^(w; x') = sum_x0 f(x_0, x') e^{-2 pi i w x_0 / L},  X^(w; h') = sum_h0 X[h_0, h'] e^{-2 pi i w h_0 / L}.
// For each of the L frequencies the inner sum is a Toeplitz product of d - 1 dimensions, which the
// product kernels compute as they compute the full one, on sub-problems (one per problem and
// frequency, the samples F^(w; .) in place of f): L (n+1)^(2(d-1)) multiply-adds per column instead
// of (n+1)^(2d), that is (n+1)/2 times fewer, and dot products (n+1) times shorter, so the FP32
// accumulations round less.  The transforms are FP32 with twiddles rounded from FP64.
//   k_axis_tables  F^(w; .) of every sub-problem, in the table format of the product kernel
//   k_axis_in      X^ in the operand format of the product kernel (BF16 / TF32 planes in the
//                  shared-memory image of a B' tile, or complex64)
//   k_axis_out     the inverse transform of the sub-products
// With w, -w, w + H and H - w (H = n + 1 = L / 2) taken together, a class of four outputs needs the
// sums of x cos and x sin over the even and the odd h_0 only: 8 real FMAs per h_0 instead of
// 32.  k_axis_out uses the same symmetry on its inputs.  A direct sum is preferred to an FFT
// stage network: it serves every n without padding L to a product of small radices.
// Measured, 64 problems of d = 3, n = 19 (N = 8000), BF16x3, T V over the row box: 80 columns 10.4 ms
// directly, now 2.6 ms (k_axis_in 0.62, the 10240 CTAs of the product kernel 1.54, k_axis_out 0.43);
// 40 columns 8.5 ms and 1.8 ms (0.33, 1.25, 0.25).  k_axis_in writes 1.97 GB at 80 columns (0.29 ms at
// 6.8 TB/s), k_axis_out moves 1.1 GB (0.16 ms): both within 2.7 times their traffic, the rest is issue of
// the splits and of the sums.  Error of one product against FP64: 3.4e-6 directly, 7e-7 now.
#include "common.cuh"
#include "tc_ptx.cuh"

#include <algorithm>

namespace {

__device__ inline float2* ax_buf(const Dev& D, int buf, const ProbDesc& p, int& ld) {
  switch (buf) {
    case BUF_V: ld = p.N; return D.V + p.xoff;
    case BUF_U: ld = p.N; return D.U + p.xoff;
    case BUF_B1: ld = p.N; return D.B1 + p.xoff;
    case BUF_B2: ld = p.N; return D.B2 + p.xoff;
    default: ld = p.Next; return D.Y + p.yoff;
  }
}

typedef unsigned long long u64;
__device__ __forceinline__ u64 ax_pack(float lo, float hi) {
  u64 r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
  return r;
}
__device__ __forceinline__ float2 ax_unpack(u64 v) {
  float lo, hi;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(v));
  return make_float2(lo, hi);
}
__device__ __forceinline__ void ax_fma(u64& acc, u64 a, u64 b) { asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(acc) : "l"(a), "l"(b)); }

// One 16-bit BF16 plane entry.
__device__ __forceinline__ uint16_t ax_bf16(float a) { return (uint16_t)(pack_bf16x2(a, 0.f) & 0xFFFFu); }

// Entry x of a sub-problem's sample table (both sides share the format): complex64 for the FP32
// products, else the split planes of Re and Im as the tensor-core kernel reads them (TF32: word x
// of each table; BF16: entries in reverse order, wide or compact).
template <int MODE, int FMT>
__device__ __forceinline__ void ax_put(float2* grid, uint32_t* tab, int Gd4, int x, float2 v) {
  if (MODE == AX_FP32) {
    grid[x] = v;
  } else if (MODE == AX_TF32X3) {
    uint32_t wr[2], wi[2];
    split_tf32(v.x, wr);
    split_tf32(v.y, wi);
#pragma unroll
    for (int pl = 0; pl < 2; ++pl) {
      tab[(long long)pl * Gd4 + x] = wr[pl];
      tab[(long long)(2 + pl) * Gd4 + x] = wi[pl];
    }
  } else {
    uint16_t* t16 = (uint16_t*)tab;
    const float r[2] = {v.x, v.y};
#pragma unroll
    for (int part = 0; part < 2; ++part) {
      float rest = r[part];
#pragma unroll
      for (int pl = 0; pl < 3; ++pl) {
        const uint16_t h = ax_bf16(rest);
        const int r = Gd4 - 1 - x;
        uint16_t* t = t16 + 2LL * (part * 3 + pl) * Gd4;
        if (FMT == TT_WIDE) {                     // low half of word r, high half of the word before
          t[2 * r] = h;
          if (r > 0) t[2 * r - 1] = h;
        } else {
          t[r] = h;
        }
        rest -= __uint_as_float((uint32_t)h << 16);
      }
    }
  }
}

// F^(w; x') for four frequencies per thread (or per `parts` threads, each summing a piece of the line), and the tables of T^* from them: the samples conj f(-x)
// transform to conj F^(w; -x'), zero where -x' leaves the grid.  The difference x_0 = n + 1 occurs
// in the products over the row box {0..n+1}^d only; `trim` leaves those samples out where a caller
// asks for a product over I_n alone (whatever they hold, they do not enter it).
template <int MODE, int FMT>
__global__ void __launch_bounds__(64) k_axis_tables(Dev D, Dev S, int trim, int parts) {
  extern __shared__ float2 ax_tw[];
  const ProbDesc& p = D.P[blockIdx.y];
  const int G = p.G, Gs = p.Gd / G;
  {
    const float2* tw = S.ftw + S.P[p.sub].foff;
    for (int j = threadIdx.x; j < G; j += blockDim.x) ax_tw[j] = tw[j];
  }
  __syncthreads();
  const int groups = (G + 3) / 4;
  const long long total = (long long)Gs * groups;
  const int part = threadIdx.x & (parts - 1), per_block = blockDim.x / parts;
  const int last = trim ? G - 1 : G;
  const int seg = (last + 8 * parts - 1) / (8 * parts) * 8, i_begin = min(part * seg, last), i_end = min(i_begin + seg, last);
  // (the loop runs for whole warps: items past the end repeat the last one and write nothing)
  for (long long q0 = blockIdx.x * (long long)per_block; q0 < total; q0 += (long long)gridDim.x * per_block) {
    const long long q = min(q0 + threadIdx.x / parts, total - 1);
    const bool mine = q0 + threadIdx.x / parts < total;
    const int x = (int)(q % Gs), w0 = 4 * (int)(q / Gs);
    const float2* f = D.gF + p.grid + x;
    float2 acc[2][4];                             // two interleaved partial sums per frequency
    int at[4], step[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      acc[0][u] = acc[1][u] = make_float2(0.f, 0.f);
      step[u] = min(w0 + u, G - 1);
      at[u] = (int)((long long)step[u] * (G - p.n + i_begin) % G);          // twiddle of x_0 = -n + i_begin
    }
    for (int i0 = i_begin; i0 < i_end; i0 += 8) {  // eight loads in flight
      float2 v[8];
#pragma unroll
      for (int e = 0; e < 8; ++e) v[e] = i0 + e < i_end ? f[(long long)(i0 + e) * Gs] : make_float2(0.f, 0.f);
#pragma unroll
      for (int e = 0; e < 8; ++e)
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          const float2 t = ax_tw[at[u]];
          float2& a = acc[e & 1][u];
          a.x = fmaf(v[e].x, t.x, fmaf(v[e].y, t.y, a.x));        // v e^{-i theta}
          a.y = fmaf(v[e].y, t.x, fmaf(-v[e].x, t.y, a.y));
          at[u] += step[u];
          if (at[u] >= G) at[u] -= G;
        }
    }
    // mirror -x' of x' on the sub-grid
    int rem = x, mir = 0, mul = 1;
    bool mvalid = true;
    for (int l = 1; l < p.d; ++l) {
      const int md = 2 * p.n - rem % G;
      rem /= G;
      if (md < 0) mvalid = false;
      mir += md * mul;
      mul *= G;
    }
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      float2 v = make_float2(acc[0][u].x + acc[1][u].x, acc[0][u].y + acc[1][u].y);
      for (int o = 1; o < parts; o <<= 1) {
        v.x += __shfl_xor_sync(0xffffffffu, v.x, o);
        v.y += __shfl_xor_sync(0xffffffffu, v.y, o);
      }
      if (!mine || w0 + u >= G || (u & (parts - 1)) != part) continue;
      const ProbDesc& ps = S.P[p.sub + w0 + u];
      ax_put<MODE, FMT>(S.gF + ps.grid, S.tabF + ps.toff, ps.Gd4, x, v);
      ax_put<MODE, FMT>(S.gH + ps.grid, S.tabH + ps.toff, ps.Gd4, mvalid ? mir : x,
                   mvalid ? make_float2(v.x, -v.y) : make_float2(0.f, 0.f));
      if (MODE != AX_FP32 && x == Gs - 1)                         // padding of the tables
        for (int y = Gs; y < ps.Gd4; ++y) {
          ax_put<MODE, FMT>(nullptr, S.tabF + ps.toff, ps.Gd4, y, make_float2(0.f, 0.f));
          ax_put<MODE, FMT>(nullptr, S.tabH + ps.toff, ps.Gd4, y, make_float2(0.f, 0.f));
        }
    }
  }
}

// X^(w; h') of column j by the lane of point h' (one of the 32 of a K chunk), into the operand of the
// product kernel.  BF16 tiles: rows 2j = (Re | -Im) and 2j + 1 = (Im | Re) of a plane hold 64 K
// values of 2 bytes; the lanes of a pair exchange their values, the even lane writes its row's
// words (two points each), the odd lane the other row's.  TF32: one word per value.
template <int MODE>
__device__ __forceinline__ void ax_emit(const Dev& S, const ProbDesc& ps, unsigned char* tile, int NT, int j, int hp,
                                        bool valid, int Np, int lane, float2 v) {
  if (MODE == AX_FP32) {
    if (valid) S.V[ps.xoff + (long long)j * Np + hp] = v;
  } else if (MODE == AX_TF32X3) {
    uint32_t re[2], im[2], ng[2];
    split_tf32(v.x, re);
    split_tf32(v.y, im);
    split_tf32(-v.y, ng);
#pragma unroll
    for (int pl = 0; pl < 2; ++pl)
#pragma unroll
      for (int odd = 0; odd < 2; ++odd) {
        const int R = pl * NT + 2 * j + odd;
        unsigned char* at = tile + (size_t)R * 128 + (((lane >> 2) ^ (R & 7)) << 4) + ((lane & 3) << 2);
        *(uint32_t*)at = odd ? im[pl] : re[pl];
        *(uint32_t*)(at + (size_t)2 * NT * 128) = odd ? re[pl] : ng[pl];
      }
  } else {
    constexpr int NPL = MODE == AX_BF16X3 ? 3 : 2;
    uint32_t own[3];
    split_pair<NPL>(v.x, v.y, own);
    const bool odd = lane & 1;
    const int row = 2 * j + (lane & 1);
#pragma unroll
    for (int pl = 0; pl < NPL; ++pl) {
      const uint32_t oth = __shfl_xor_sync(0xffffffffu, own[pl], 1);
      const uint32_t lo = odd ? oth : own[pl], hi = odd ? own[pl] : oth;
      const uint32_t rew = __byte_perm(lo, hi, 0x5410), imw = __byte_perm(lo, hi, 0x7632);
      const int R = pl * NT + row, g = lane >> 3;
      unsigned char* at = tile + (size_t)R * 128 + (((lane & 7) >> 1) << 2);
      *(uint32_t*)(at + ((g ^ (R & 7)) << 4)) = odd ? imw : rew;
      *(uint32_t*)(at + (((4 + g) ^ (R & 7)) << 4)) = odd ? rew : imw ^ 0x80008000u;
    }
  }
}

// A warp takes 32 points h', NC columns and CL frequency classes at a time; the items of a
// problem are spread over its warps, the classes of a line next to each other (the line's n + 1
// values then come from L1 for all but the first).  Large batches take four classes and two
// columns (each twiddle read serves two lines), bound by HBM writes: 24 bytes per transformed
// value of a BF16x3 operand.  Few lines (one problem) take one class and one column, eight times
// the warps: there the loads' latency counts.
template <int MODE, int CL, int NC>
__global__ void __launch_bounds__(256, 2) k_axis_in(Dev D, Dev S, int xbuf, int wsel, unsigned char* xb,
                                                 long long xb_stride) {
  extern __shared__ float4 ax_tab[];              // [class][h_0] = (cos, cos, sin, sin)
  const ProbDesc& p = D.P[blockIdx.y];
  const ProbState& st = D.st[p.st];
  if (st.done) return;
  const int w = sel_width(st, p, wsel);
  if (w <= 0) return;
  const int H = p.n + 1, L = p.G, Hs = H + (H & 1), Np = p.N / H;
  const int ncls = H / 2 + 1, ngrp = (ncls + CL - 1) / CL, nc = (Np + 31) / 32;
  const int NT = ((2 * w + 15) / 16) * 16;
  const int ncol = MODE == AX_FP32 ? (w + NC - 1) / NC : NT / (2 * NC);
  {
    const float2* tw = S.ftw + S.P[p.sub].foff;
    for (int q = threadIdx.x; q < ncls * Hs; q += blockDim.x) {
      const int c = q / Hs, h = q % Hs;
      const float2 t = h < H ? tw[(c * h) % L] : make_float2(0.f, 0.f);
      ax_tab[q] = make_float4(t.x, t.x, t.y, t.y);
    }
  }
  __syncthreads();
  int ldx;
  const float2* X = ax_buf(D, xbuf, p, ldx);
  const int lane = threadIdx.x & 31;
  constexpr int NPL = MODE == AX_BF16X3 ? 3 : 2;
  constexpr int HU = CL * NC == 8 ? 2 : 8;        // h_0 per pass (their loads are in flight together)
  const size_t tile_bytes = (size_t)(MODE == AX_TF32X3 ? 2 : 1) * NPL * NT * 128;
  const long long items = (long long)nc * ncol * ngrp, xchunk = S.P[p.sub].xchunk;
  for (long long it = blockIdx.x * (long long)(blockDim.x >> 5) + (threadIdx.x >> 5); it < items;
       it += (long long)gridDim.x * (blockDim.x >> 5)) {
    const int grp = (int)(it % ngrp), c = (int)(it / ngrp / ncol), j0 = NC * (int)(it / ngrp % ncol);
    const int hp = 32 * c + lane;
    const bool valid = hp < Np;
    const float2* x0 = X + (long long)j0 * ldx + hp;
    u64 acc[CL][NC][4];                           // class, column, (cos even, sin even, cos odd, sin odd)
#pragma unroll
    for (int u = 0; u < CL; ++u)
#pragma unroll
      for (int k = 0; k < NC; ++k)
#pragma unroll
        for (int z = 0; z < 4; ++z) acc[u][k][z] = 0ull;
    const ulonglong2* tb[CL];
#pragma unroll
    for (int u = 0; u < CL; ++u) tb[u] = (const ulonglong2*)ax_tab + min(CL * grp + u, ncls - 1) * Hs;
    if (j0 < w) {
      for (int h = 0; h < H; h += HU) {
        u64 x[HU][NC];
#pragma unroll
        for (int e = 0; e < HU; ++e)
#pragma unroll
          for (int k = 0; k < NC; ++k) {
            const bool ok = valid && h + e < H && j0 + k < w;
            const float2 v = ok ? x0[(long long)k * ldx + (long long)(h + e) * Np] : make_float2(0.f, 0.f);
            x[e][k] = ax_pack(v.x, v.y);
          }
#pragma unroll
        for (int e = 0; e < HU; ++e) {
          if (h + e >= Hs) break;
#pragma unroll
          for (int u = 0; u < CL; ++u) {
            const ulonglong2 t = tb[u][h + e];
#pragma unroll
            for (int k = 0; k < NC; ++k) {
              ax_fma(acc[u][k][2 * (e & 1)], x[e][k], t.x);
              ax_fma(acc[u][k][2 * (e & 1) + 1], x[e][k], t.y);
            }
          }
        }
      }
    }
#pragma unroll
    for (int u = 0; u < CL; ++u) {
      const int cls = CL * grp + u;
      if (cls >= ncls) break;
      const bool four = cls != 0 && 2 * cls != H;
#pragma unroll
      for (int k = 0; k < NC; ++k) {
        if (MODE == AX_FP32 && j0 + k >= w) break;
        const float2 ce = ax_unpack(acc[u][k][0]), se = ax_unpack(acc[u][k][1]);
        const float2 co = ax_unpack(acc[u][k][2]), so = ax_unpack(acc[u][k][3]);
        const float2 a = make_float2(ce.x + co.x, ce.y + co.y), b = make_float2(se.x + so.x, se.y + so.y);
        const float2 c2 = make_float2(ce.x - co.x, ce.y - co.y), d2 = make_float2(se.x - so.x, se.y - so.y);
        auto put = [&](int f, float2 v) {
          ax_emit<MODE>(S, S.P[p.sub + f], xb + xb_stride * (xchunk + f * nc) + (size_t)c * tile_bytes, NT, j0 + k, hp, valid,
                        Np, lane, v);
        };
        put(cls, make_float2(a.x + b.y, a.y - b.x));              // cos - i sin
        put(cls + H, make_float2(c2.x + d2.y, c2.y - d2.x));
        if (four) {
          put(L - cls, make_float2(a.x - b.y, a.y + b.x));
          put(H - cls, make_float2(c2.x - d2.y, c2.y + d2.x));
        }
      }
    }
  }
}

// The inverse transform of one line (k', column j) by a lane, KB rows k_0 at a time:
//   y[k] = (1/L) sum over the classes of P cos + i Q sin,  P = A + A', Q = A - A' for even k with
// A = y^(w) + y^(w+H), A' = y^(-w) + y^(H-w), and the differences instead of the sums for odd k.
template <int KB, int SP>
__global__ void __launch_bounds__(256) k_axis_out(Dev D, Dev S, int wsel, int ybuf, int y_ext) {
  extern __shared__ float4 ax_tab[];              // [class][k_0] = (cos, cos, sin, sin)
  const ProbDesc& p = D.P[blockIdx.y];
  const ProbState& st = D.st[p.st];
  if (st.done) return;
  const int w = sel_width(st, p, wsel);
  if (w <= 0) return;
  const int H = p.n + 1, L = p.G, K = y_ext ? H + 1 : H;
  const int Np = y_ext ? p.Next / (p.n + 2) : p.N / H;            // rows of a sub-product
  const int ncls = H / 2 + 1, nblk = (K + KB - 1) / KB, Kt = nblk * KB, nt = (Np + 31) / 32;
  const ProbDesc& ps = S.P[p.sub];
  {
    const float2* tw = S.ftw + ps.foff;
    for (int q = threadIdx.x; q < ncls * Kt; q += blockDim.x) {
      const int c = q / Kt, k = q % Kt;
      const float2 t = k < K ? tw[(c * k) % L] : make_float2(0.f, 0.f);
      ax_tab[q] = make_float4(t.x, t.x, t.y, t.y);
    }
  }
  __syncthreads();
  const long long fstride = (long long)Np * p.r0;                 // one frequency of the sub-products
  const float2* src0 = y_ext ? S.Y + ps.yoff : S.B2 + ps.xoff;
  int ldy;
  float2* Y = ax_buf(D, ybuf, p, ldy);
  const float scale = 1.0f / (float)L;
  const int lane = threadIdx.x & 31;
  const long long items = (long long)nt * w * nblk;
  constexpr int PER = 8 / SP;                     // items of a block at a time
  const int warp = threadIdx.x >> 5, sub = warp % SP;
  for (long long it0 = blockIdx.x * (long long)PER; it0 < items; it0 += (long long)gridDim.x * PER) {
    const bool mine = it0 + warp / SP < items;
    if (SP == 1 && !mine) break;
    const long long it = mine ? it0 + warp / SP : items - 1;
    const int blk = (int)(it % nblk), t = (int)(it / nblk % nt), j = (int)(it / nblk / nt);
    const int kp = 32 * t + lane, k0 = blk * KB;
    const bool valid = mine && kp < Np;
    const float2* src = src0 + (long long)j * Np + (valid ? kp : 0);
    u64 acc[KB];
#pragma unroll
    for (int k = 0; k < KB; ++k) acc[k] = 0ull;
#pragma unroll(KB <= 8 ? 4 : 2)
    for (int c = sub; c < ncls; c += SP) {
      const bool four = c != 0 && 2 * c != H;
      const float2 zero = make_float2(0.f, 0.f);
      const float2 y0 = src[c * fstride], y2 = src[(c + H) * fstride];
      const float2 y1 = four ? src[(L - c) * fstride] : zero, y3 = four ? src[(H - c) * fstride] : zero;
      const float2 ap = make_float2(y0.x + y2.x, y0.y + y2.y), am = make_float2(y0.x - y2.x, y0.y - y2.y);
      const float2 bp = make_float2(y1.x + y3.x, y1.y + y3.y), bm = make_float2(y1.x - y3.x, y1.y - y3.y);
      const u64 pe = ax_pack(ap.x + bp.x, ap.y + bp.y), qe = ax_pack(bp.y - ap.y, ap.x - bp.x);   // i (A - A')
      const u64 po = ax_pack(am.x + bm.x, am.y + bm.y), qo = ax_pack(bm.y - am.y, am.x - bm.x);
      const ulonglong2* tb = (const ulonglong2*)ax_tab + c * Kt + k0;
#pragma unroll
      for (int k = 0; k < KB; k += 2) {
        const ulonglong2 t0 = tb[k], t1 = tb[k + 1];
        ax_fma(acc[k], pe, t0.x);
        ax_fma(acc[k], qe, t0.y);
        ax_fma(acc[k + 1], po, t1.x);
        ax_fma(acc[k + 1], qo, t1.y);
      }
    }
    if (SP > 1) {                                 // the warps of an item: sums over their classes, in order
      __shared__ u64 part[SP > 1 ? 8 : 1][SP > 1 ? KB : 1][32];
      __syncthreads();
#pragma unroll
      for (int k = 0; k < KB; ++k) part[warp][k][lane] = acc[k];
      __syncthreads();
      constexpr int OWN = KB / SP;
      if (valid) {
        float2* dst = Y + (long long)j * ldy + (long long)k0 * Np + kp;
#pragma unroll
        for (int e = 0; e < OWN; ++e) {
          const int k = sub * OWN + e;
          float2 v = ax_unpack(part[warp - sub][k][lane]);
#pragma unroll
          for (int g = 1; g < SP; ++g) {
            const float2 u = ax_unpack(part[warp - sub + g][k][lane]);
            v.x += u.x;
            v.y += u.y;
          }
          if (k0 + k < K) dst[(long long)k * Np] = make_float2(v.x * scale, v.y * scale);
        }
      }
    } else if (valid) {
      float2* dst = Y + (long long)j * ldy + (long long)k0 * Np + kp;
#pragma unroll
      for (int k = 0; k < KB; ++k)
        if (k0 + k < K) {
          const float2 v = ax_unpack(acc[k]);
          dst[(long long)k * Np] = make_float2(v.x * scale, v.y * scale);
        }
    }
  }
}

// S.fLT holds the largest n of the batch, S.maxN / S.maxNext / S.maxGd its largest sub-problem.
inline int max_axis_n(const Dev& S) { return S.fLT; }

}  // namespace

template <int MODE, int FMT>
static cudaError_t axis_tables(const Dev& D, const Dev& S, int trim, cudaStream_t s) {
  const int G = 2 * max_axis_n(S) + 2;
  const long long items = (long long)S.maxGd * ((G + 3) / 4);
  // eight threads a sum where that leaves at most two warps per scheduler: a single small problem has a few thousand
  // sums of 2 n + 2 terms, each a chain of loads and twiddle steps (d = 2, n = 50: 44 -> 13 us)
  const int parts = 8 * items * D.nprob <= 152LL * 256 ? 8 : 1;
  note_launch();
  k_axis_tables<MODE, FMT><<<dim3(blocks_per_problem((parts * items + 63) / 64, D.nprob), D.nprob), 64, sizeof(float2) * G, s>>>(
      D, S, trim, parts);
  return cudaGetLastError();
}

cudaError_t launch_axis_tables(const Dev& D, const Dev& S, int mode, int fmt, int trim, cudaStream_t s) {
  if (mode == AX_FP32) return axis_tables<AX_FP32, TT_TF32>(D, S, trim, s);
  if (mode == AX_TF32X3) return axis_tables<AX_TF32X3, TT_TF32>(D, S, trim, s);
  return fmt == TT_WIDE ? axis_tables<AX_BF16X3, TT_WIDE>(D, S, trim, s)              // three planes written, two or three read
                        : axis_tables<AX_BF16X3, TT_COMPACT>(D, S, trim, s);
}

template <int MODE, int CL, int NC>
static cudaError_t axis_in_as(const Dev& D, const Dev& S, int xbuf, int wsel, long long items, void* xb,
                              long long xb_stride, cudaStream_t s) {
  const int H = max_axis_n(S) + 1;
  const size_t sm = sizeof(float4) * (size_t)(H / 2 + 1) * (H + (H & 1));
  cudaError_t e = allow_smem(k_axis_in<MODE, CL, NC>, sm);
  if (e != cudaSuccess) return e;
  const long long per = items * D.nprob > 152LL * 64 ? 2 : 1;     // items per warp (one twiddle table per block)
  note_launch();
  k_axis_in<MODE, CL, NC><<<dim3(blocks_per_problem((items + 8 * per - 1) / (8 * per), D.nprob), D.nprob), 256, sm, s>>>(
      D, S, xbuf, wsel, (unsigned char*)xb, xb_stride);
  return cudaGetLastError();
}

template <int MODE>
static cudaError_t axis_in(const Dev& D, const Dev& S, int xbuf, int wsel, int maxw, void* xb, long long xb_stride,
                           cudaStream_t s) {
  // items of the largest problem; the wide form from about eight of its warps per SM on
  const int ncls = (max_axis_n(S) + 1) / 2 + 1;
  const long long lines = (long long)((S.maxN + 31) / 32) * ((2 * maxw + 15) / 16 * 8);
  if (lines * ncls / 8 * D.nprob >= 152LL * 8)
    return axis_in_as<MODE, 4, 2>(D, S, xbuf, wsel, (lines + 1) / 2 * ((ncls + 3) / 4), xb, xb_stride, s);
  return axis_in_as<MODE, 1, 1>(D, S, xbuf, wsel, lines * ncls, xb, xb_stride, s);
}

cudaError_t launch_axis_in(const Dev& D, const Dev& S, int mode, int xbuf, int wsel, int maxw, void* xb,
                           long long xb_stride, cudaStream_t s) {
  switch (mode) {
    case AX_FP32: return axis_in<AX_FP32>(D, S, xbuf, wsel, maxw, xb, xb_stride, s);
    case AX_TF32X3: return axis_in<AX_TF32X3>(D, S, xbuf, wsel, maxw, xb, xb_stride, s);
    case AX_BF16X2: return axis_in<AX_BF16X2>(D, S, xbuf, wsel, maxw, xb, xb_stride, s);
    default: return axis_in<AX_BF16X3>(D, S, xbuf, wsel, maxw, xb, xb_stride, s);
  }
}

template <int KB, int SP>
static cudaError_t axis_out(const Dev& D, const Dev& S, int wsel, int ybuf, int y_ext, int maxw, cudaStream_t s) {
  const int H = max_axis_n(S) + 1, K = y_ext ? H + 1 : H, nblk = (K + KB - 1) / KB;
  // (H / 2 + 1) x Kt grows with n: the largest problem's table is the largest of the batch
  const size_t sm = sizeof(float4) * (size_t)(H / 2 + 1) * nblk * KB;
  cudaError_t e = allow_smem(k_axis_out<KB, SP>, sm);
  if (e != cudaSuccess) return e;
  const long long items = (long long)(((y_ext ? S.maxNext : S.maxN) + 31) / 32) * maxw * nblk;
  note_launch();
  k_axis_out<KB, SP><<<dim3(blocks_per_problem((items * SP + 7) / 8, D.nprob), D.nprob), 256, sm, s>>>(D, S, wsel, ybuf, y_ext);
  return cudaGetLastError();
}

cudaError_t launch_axis_out(const Dev& D, const Dev& S, int wsel, int ybuf, int y_ext, int maxw, cudaStream_t s) {
  // 22 rows a pass re-read the sub-products least: the most that leave two blocks of 256 threads per SM (109 registers,
  // 24 rows take 146).  A last pass computes rows past the end: none at n = 19, a fifth of the work at n = 50.  Few lines (a
  // single small problem) take 8 rows a pass, which gives three times the warps, and with fewer than eight warps per SM four warps share a line's
  // classes (d = 2, n = 50, 37 columns: 25 -> 11 us; with 11 warps per SM, d = 3, n = 19, 40 columns, 3 us slower)
  const long long lines = (long long)(((y_ext ? S.maxNext : S.maxN) + 31) / 32) * maxw * D.nprob;
  if (lines >= 152LL * 16) return axis_out<22, 1>(D, S, wsel, ybuf, y_ext, maxw, s);
  const int nblk = (max_axis_n(S) + (y_ext ? 2 : 1) + 7) / 8;
  return lines * nblk < 152LL * 8 ? axis_out<8, 4>(D, S, wsel, ybuf, y_ext, maxw, s)
                                  : axis_out<8, 1>(D, S, wsel, ybuf, y_ext, maxw, s);
}
