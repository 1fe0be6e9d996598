// Device parts of the transform solve (boxpoisson.cu) that its own kernels and
// the closing kernel of the step's solve (poisson.cu) share.
#pragma once

#include <cuda_runtime.h>

#include "internal.cuh"

namespace picgb {

constexpr int kBoxThreads = 512;       // of the solve and the closing kernel
constexpr int kKB = 4;                 // modes per CTA of the solve


struct BoxArgs {
  BoxBlock b[2];           // slab, slot
  int nblk[2];             // CTAs of the solve per block
  int pitch;               // nodes per grid row
  int slot, xs, singular;
  const float *sinv;       // [wc][wc] inverse of the interface's Schur complement
  float *fh, *sh;          // spectra of the interface values in the slab's and the slot's basis
  unsigned int *ticket;
  const float *r;
  float2 *pot;
  PoissonState *ps;
};

// tridiag(-1, d, -1) x = y in place for one warp: y_i <- w_i (y_i + y_{i-1}),
// then x_i = y_i + w_i x_{i+1} (Thomas, w_i = 1 / (d - w_{i-1})).  Each lane
// takes a run of rows; both recurrences are linear in the value carried into
// the run, so a first pass gives every run's result for a zero carry and the
// product of its factors, a scan over the lanes the carries, and a second pass
// the values.  An odd run length keeps the lanes on different banks.
__device__ __forceinline__ void tri_warp(float *y, const float *w, int m) {
  const int lane = threadIdx.x & 31, L = ((m + 31) / 32) | 1;
  const int lo = min(m, lane * L), hi = min(m, lo + L);
  float v = 0.f, p = 1.f;
  for (int i = lo; i < hi; ++i) {
    v = w[i] * (y[i] + v);
    p *= w[i];
  }
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const float v0 = __shfl_up_sync(0xffffffffu, v, o), p0 = __shfl_up_sync(0xffffffffu, p, o);
    if (lane >= o) {
      v = fmaf(p, v0, v);
      p *= p0;
    }
  }
  float c = __shfl_up_sync(0xffffffffu, v, 1);
  if (lane == 0) c = 0.f;
  for (int i = lo; i < hi; ++i) {
    c = w[i] * (y[i] + c);
    y[i] = c;
  }
  __syncwarp();
  v = 0.f;
  p = 1.f;
  for (int i = hi - 1; i >= lo; --i) {
    v = fmaf(w[i], v, y[i]);
    p *= w[i];
  }
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const float v0 = __shfl_down_sync(0xffffffffu, v, o), p0 = __shfl_down_sync(0xffffffffu, p, o);
    if (lane + o < 32) {
      v = fmaf(p, v0, v);
      p *= p0;
    }
  }
  c = __shfl_down_sync(0xffffffffu, v, 1);
  if (lane == 31) c = 0.f;
  for (int i = hi - 1; i >= lo; --i) {
    c = fmaf(w[i], c, y[i]);
    y[i] = c;
  }
  __syncwarp();
}

// The interface, in the last CTA to finish: g = r_G + v_R(row m) + v_S(first
// slot row), u_G = S^-1 g added to the potential, and the spectra of u_G that
// the inverse transform applies.
__device__ __forceinline__ void box_interface(const BoxArgs &f, float *sm) {
  const BoxBlock &R = f.b[0], &S = f.b[1];
  const int wc = S.n, nk = R.n, lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
  float *vm = sm, *vs = vm + nk, *g = vs + wc, *u = g + wc;
  for (int k = threadIdx.x; k < nk; k += blockDim.x) vm[k] = __ldcg(R.c + size_t(k) * R.mp + R.m - 1);
  for (int k = threadIdx.x; k < wc; k += blockDim.x) vs[k] = __ldcg(S.c + size_t(k) * S.mp);
  __syncthreads();
  const int c0 = S.col0 - R.col0;   // the slot's first column in the slab's numbering
  for (int c = warp; c < wc; c += nw) {
    const float *vr = R.v + size_t(c0 + c) * R.ldv, *vc = S.v + size_t(c) * S.ldv;
    float a = 0.f;
    for (int k = lane; k < nk; k += 32) a = fmaf(vm[k], __ldg(vr + k), a);
    for (int k = lane; k < wc; k += 32) a = fmaf(vs[k], __ldg(vc + k), a);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) a += __shfl_xor_sync(0xffffffffu, a, o);
    if (lane == 0) g[c] = __ldcg(f.r + size_t(f.xs) * f.pitch + S.col0 + c) + a;
  }
  __syncthreads();
  for (int c = warp; c < wc; c += nw) {
    float a = 0.f;
    for (int q = lane; q < wc; q += 32) a = fmaf(__ldg(f.sinv + size_t(c) * wc + q), g[q], a);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) a += __shfl_xor_sync(0xffffffffu, a, o);
    if (lane == 0) {
      u[c] = a;
      const size_t n = size_t(f.xs) * f.pitch + S.col0 + c;
      f.pot[n] = pair_add_f(f.pot[n], a);
    }
  }
  __syncthreads();
  for (int k = threadIdx.x; k < nk; k += blockDim.x) {
    float a = 0.f;
#pragma unroll 8
    for (int c = 0; c < wc; ++c) a = fmaf(u[c], __ldg(R.v + size_t(c0 + c) * R.ldv + k), a);
    f.fh[k] = a;
  }
  for (int k = threadIdx.x; k < wc; k += blockDim.x) {
    float a = 0.f;
#pragma unroll 8
    for (int c = 0; c < wc; ++c) a = fmaf(u[c], __ldg(S.v + size_t(c) * S.ldv + k), a);
    f.sh[k] = a;
  }
}

// Group g of a block's modes (kKB of them; the slab's groups come first):
// c[k][i] = sum_j r[i][j] V[j][k] over all rows i, then each mode's tridiagonal
// system in one warp.  box_stage brings the static tables (basis columns, Thomas
// factors) into sm; box_modes takes four rows a warp at a time, lanes along j.
__device__ __forceinline__ void box_stage(const BoxArgs &f, int g, float *sm) {
  const int which = g < f.nblk[0] ? 0 : 1;
  const BoxBlock &B = f.b[which];
  const int k0 = (g - (which ? f.nblk[0] : 0)) * kKB, n = B.n, mp = B.mp;
  float4 *vs = reinterpret_cast<float4 *>(sm);   // [n] the group's basis columns
  float *ws = sm + 4 * n;                        // [kKB][mp] Thomas factors
  for (int j = threadIdx.x; j < n; j += blockDim.x)
    vs[j] = __ldg(reinterpret_cast<const float4 *>(B.v + size_t(j) * B.ldv + k0));
  for (int t = threadIdx.x; t < kKB * mp; t += blockDim.x) {
    const int kk = t / mp;
    ws[t] = k0 + kk < n ? __ldg(B.w + size_t(k0) * mp + t) : 0.f;
  }
}
__device__ __forceinline__ void box_modes(const BoxArgs &f, int g, float *sm) {
  const int which = g < f.nblk[0] ? 0 : 1;
  const BoxBlock &B = f.b[which];
  const int k0 = (g - (which ? f.nblk[0] : 0)) * kKB, n = B.n, m = B.m, mp = B.mp;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
  const float4 *vs = reinterpret_cast<const float4 *>(sm);
  const float *ws = sm + 4 * n;
  float *cs = sm + 4 * n + kKB * mp;             // [kKB][mp] spectra
  for (int i0 = 4 * warp; i0 < m; i0 += 4 * nw) {
    float a[16];
#pragma unroll
    for (int q = 0; q < 16; ++q) a[q] = 0.f;
    const float *r0 = f.r + size_t(B.row0 + i0) * f.pitch + B.col0;
#pragma unroll 4
    for (int j = lane; j < n; j += 32) {
      const float4 v = vs[j];
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const float rv = i0 + q < m ? __ldcg(r0 + size_t(q) * f.pitch + j) : 0.f;
        a[4 * q + 0] = fmaf(rv, v.x, a[4 * q + 0]);
        a[4 * q + 1] = fmaf(rv, v.y, a[4 * q + 1]);
        a[4 * q + 2] = fmaf(rv, v.z, a[4 * q + 2]);
        a[4 * q + 3] = fmaf(rv, v.w, a[4 * q + 3]);
      }
    }
    // sums over the lanes: each exchange halves the values a lane still holds,
    // lane l ends with value l >> 1 (both lanes of a pair hold half of it)
#pragma unroll
    for (int h = 8, o = 16; h >= 1; h >>= 1, o >>= 1) {
      const bool upper = (lane & o) != 0;
#pragma unroll
      for (int q = 0; q < h; ++q) {
        const float keep = upper ? a[q + h] : a[q], give = upper ? a[q] : a[q + h];
        a[q] = keep + __shfl_xor_sync(0xffffffffu, give, o);
      }
    }
    a[0] += __shfl_xor_sync(0xffffffffu, a[0], 1);
    const int q = lane >> 1, i = i0 + (q >> 2);
    if (!(lane & 1) && i < m) cs[(q & 3) * mp + i] = a[0];
  }
  __syncthreads();
  if (warp < kKB && k0 + warp < n) {
    const int k = k0 + warp;
    float *y = cs + warp * mp;
    const float *w = ws + warp * mp;
    if (!B.ring) {
      tri_warp(y, w, m);
    } else {
      // a ring of m rows: rows 1 .. m - 1 with row 0 held, then row 0 from
      // its own equation and its response z on the others; the singular
      // system (a doubly periodic box's constant mode) keeps row 0 at 0 and
      // loses its mean
      tri_warp(y + 1, w + 1, m - 1);
      const float x0 = (y[0] + y[1] + y[m - 1]) * __ldg(B.ring + k);
      __syncwarp();
      const float *z = B.z + size_t(k) * mp;
      float s = 0.f;
      for (int i = 1 + lane; i < m; i += 32) {
        const float x = fmaf(x0, __ldg(z + i), y[i]);
        y[i] = x;
        s += x;
      }
      __syncwarp();
      if (lane == 0) y[0] = x0;
      if (f.singular && k == 0) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
        s /= float(m);
        __syncwarp();
        for (int i = lane; i < m; i += 32) y[i] -= s;
      }
      __syncwarp();
    }
    for (int i = lane; i < m; i += 32) B.c[size_t(k) * mp + i] = y[i];
  }
}

// Inverse transform of rows i0 .. i0 + 7 of block B, added to the potential:
// e[i][j] = sum_k (c[k][i] + z[k][i] h[k]) V[j][k].  The CTA's threads are
// spread over the columns and, where those are few, over the eight rows.
template <int NR>
__device__ __forceinline__ void box_add_columns(const BoxArgs &f, const BoxBlock &B, const float *cs, int i0, int j0,
                                                int step, int row, int rg) {
  for (int j = j0; j < B.n; j += step) {
    float e[NR];
    float2 p[NR];
#pragma unroll
    for (int q = 0; q < NR; ++q) {
      e[q] = 0.f;
      const int i = i0 + row + q * rg;
      p[q] = i < B.m ? __ldcg(f.pot + size_t(B.row0 + i) * f.pitch + B.col0 + j) : make_float2(0.f, 0.f);
    }
    const float *v = B.vt + j;
#pragma unroll 16
    for (int k = 0; k < B.n; ++k) {
      const float vv = __ldg(v + size_t(k) * B.n);
#pragma unroll
      for (int q = 0; q < NR; ++q) e[q] = fmaf(cs[8 * k + row + q * rg], vv, e[q]);
    }
#pragma unroll
    for (int q = 0; q < NR; ++q) {
      const int i = i0 + row + q * rg;
      if (i < B.m) f.pot[size_t(B.row0 + i) * f.pitch + B.col0 + j] = pair_add_f(p[q], e[q]);
    }
  }
}
// the rows of every block, eight at a time, shared out over ncta CTAs; sm: 8 n floats
__device__ __forceinline__ void box_add_rows(const BoxArgs &f, float *sm, int rank, int ncta) {
  for (int which = 0; which <= f.slot; ++which) {
    const BoxBlock &B = f.b[which];
    const float *h = f.slot ? (which ? f.sh : f.fh) : nullptr;
    const int cw = min(int(blockDim.x), (B.n + 31) & ~31), fit = int(blockDim.x) / cw;
    const int rg = fit >= 8 ? 8 : fit >= 4 ? 4 : fit >= 2 ? 2 : 1;
    const int row = int(threadIdx.x) / cw, j0 = int(threadIdx.x) - row * cw;
    for (int i0 = 8 * rank; i0 < B.m; i0 += 8 * ncta) {
      for (int t = threadIdx.x; t < 2 * B.n; t += blockDim.x) {
        const int k = t >> 1, q = (t & 1) * 4;
        float4 c = __ldcg(reinterpret_cast<const float4 *>(B.c + size_t(k) * B.mp + i0 + q));
        if (h) {
          const float4 z = __ldg(reinterpret_cast<const float4 *>(B.z + size_t(k) * B.mp + i0 + q));
          const float hk = __ldcg(h + k);
          c = make_float4(fmaf(z.x, hk, c.x), fmaf(z.y, hk, c.y), fmaf(z.z, hk, c.z), fmaf(z.w, hk, c.w));
        }
        *reinterpret_cast<float4 *>(sm + 8 * k + q) = c;
      }
      __syncthreads();
      if (row < rg) {
        if (rg == 8) box_add_columns<1>(f, B, sm, i0, j0, cw, row, 8);
        else if (rg == 4) box_add_columns<2>(f, B, sm, i0, j0, cw, row, 4);
        else if (rg == 2) box_add_columns<4>(f, B, sm, i0, j0, cw, row, 2);
        else box_add_columns<8>(f, B, sm, i0, j0, cw, row, 1);
      }
      __syncthreads();
    }
  }
}

inline size_t box_solve_smem(const BoxBlock &b) { return (4 * size_t(b.n) + 2 * kKB * size_t(b.mp)) * 4; }
// Where the captured step's solve ends in a cluster (k_box_tail) instead of a
// conditional node: grids whose checking pass 16 SMs do in no more than the
// node's cost beyond what all of them take (384 x 384: the same step time, 512 x
// 512: 123 -> 131 us).
constexpr int kTailNodes = 81920;
// Its further passes are transforms by a dense basis on 16 SMs, which grow with the
// columns squared.  Two passes a step against multigrid (1e-8): 128 x 512 between walls
// 237 against 494 us, 64 x 1024 547 against 483 (1e-6 from a guess of 0: 547 against 428);
// so a box of more than kTailCols columns repeats its two kernels on all SMs under the node.
constexpr int kTailCols = 512;
// On a grid of the FFT solve a conditional node runs the FFT kernels on all SMs instead.
// With one pass a step the cluster gains on every such grid (128 x 64: 57 -> 35 us a step,
// 312 x 256: 67 -> 55, 72 x 1024: 80 -> 64), with two only on the smaller ones (640 x 32: 87
// -> 67, 128 x 64: 80 -> 64, 160 x 128: 88 -> 88; but 1248 x 64: 105 -> 134, 312 x 256: 99
// -> 196, 72 x 1024: 118 -> 522).  So the FFT grids have it up to kFftTailNodes nodes and
// kFftTailCols columns, and beyond where a second pass is rare: up to kFftOnceRows rows
// and kFftOnceCols columns, a tolerance of kFftOnceRtol or more and a guess from the
// steps before (passes a step on 320 rows: 1.00 to 1.08 from the potential of the step
// before, 2.00 from 0; on 640 rows up to 1.42; on 1248 up to 1.77).
constexpr int kFftTailNodes = 21504, kFftTailCols = 128;
constexpr int kFftOnceRows = 320, kFftOnceCols = 256;
constexpr double kFftOnceRtol = 1e-6;
// launch arguments for a context's transform solve of A e = r (its tables set up)
BoxArgs box_args(pic_ctx *c, const float *r, float2 *pot, PoissonState *ps);

}  // namespace picgb
