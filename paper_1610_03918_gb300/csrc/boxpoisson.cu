// Transform solve of the Poisson correction equation A e = r, A = -Delta_h on
// the free nodes, for the boxes that the FFT solve of fastpoisson.cu does not
// take: y periodic with any node count, or bounded; x bounded (with or without
// the trench's slot under the slab) or periodic.
//
// The slab rows are diagonalised along y by a dense orthonormal real basis V
// (cosines and sines where y is periodic, sines between two walls), which
// leaves per mode k the system tridiag(-1, 2 + lambda_k, -1) along x, with
// Dirichlet ends or, x periodic, closed into a ring.  Interface row and slot
// are eliminated as in fastpoisson.cu, with V in place of the Fourier basis:
//   v_R = A_RR^-1 r_R,   v_S = A_SS^-1 r_S,
//   (A_GG - G_R - G_S) u_G = r_G + v_R(row m) + v_S(row xs + 1),
//   u_R = v_R + A_RR^-1 (u_G on row m),   u_S = v_S + A_SS^-1 (u_G on row xs + 1).
// Slab and slot are the same kind of block (rows x columns, a basis, a
// tridiagonal system per mode), so both run through the same two kernels:
//   k_box_solve  forward transform of a few modes over all rows, their
//                tridiagonal systems; the last CTA to finish solves the interface
//   k_box_add    inverse transform, added to the double-float potential
// Arithmetic is FP32; the iterative refinement around it certifies the result.
//
// What bounds it: latency.  These grids hold 2k to 300k nodes (0.01 to 1.2 MB,
// L2-resident), so a pass is two kernels of a few microseconds, where the
// multigrid PCG took 4 to 14 iterations of 3 to 11 launches, and where a size
// had few factors of two, a coarsest level of hundreds of nodes swept in one
// CTA.  A dense basis costs m n^2 multiply-adds per transform (17M on 256 x
// 256, 157M on 600 x 512), which the FP32 pipes do in 1 to 10 us; an FFT of
// general length would save operations that are not the bound here.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <vector>

#include "boxpoisson.cuh"
#include "internal.cuh"

namespace picgb {
namespace {

constexpr int kAddThreads = 128;       // one column per thread
constexpr int kChunkK = 32;            // modes staged per round of the inverse transform
constexpr int kMaxCols = 1024;         // columns of the basis (V is n x n)
constexpr int kMaxRows = 4096;
constexpr int kMaxSlot = 512;          // interface columns (their Schur complement is inverted on the host)

// Multiply-adds of a transform (rows x columns^2) above which multigrid is the faster
// one.  A pass here grows with that product, a V-cycle with the nodes; one, two and
// three passes stand against 5, 7 to 9 and 10 to 12 V-cycles at tolerances of 1e-6, 1e-8
// to 1e-10 and 1e-12, two against 6 at 1e-6 from a guess of 0.  Four walls, us a step
// here : there at 1e-6, 1e-8, 1e-12 and from 0: 1024 x 1024 553 : 779, 908 : 1018, 1258 :
// 1385, 917 : 919; 2048 x 1024 1044 : 1153, 1675 : 1485, 2328 : 2094, 1669 : 1354.  A
// coarsest level of more than 160 unknowns is swept in one CTA, 0.06 us a node and
// V-cycle: the line rises with it.  Doubly periodic boxes' V-cycles take longer (1024 x
// 1024 539 : 817, 869 : 1055, 1190 : 1423, 871 : 964; 2048 x 1024 979 : 1238, 1573 : 1588,
// 2170 : 2194, 1581 : 1447); with such a coarsest level multigrid is slow on any box
// periodic in y (4096 x 960 between plates 1427 : 4970).
constexpr double kMaxWorkWalls = 1.1e9, kMaxWorkCoarsest = 1.2e6, kMaxWorkPeriodic = 1.7e9;

int pad4(int n) { return (n + 3) & ~3; }
int pad8(int n) { return (n + 7) & ~7; }

// one group of modes per CTA (the tables staged before the wait for the
// preceding kernel); the last CTA to finish solves the interface
__global__ void __launch_bounds__(kBoxThreads, 1) k_box_solve(BoxArgs f) {
  extern __shared__ __align__(16) float sm[];
  __shared__ bool last;
  box_stage(f, blockIdx.x, sm);
  pdl_enter();
  __syncthreads();
  box_modes(f, blockIdx.x, sm);
  if (!f.slot) return;
  __syncthreads();   // the CTA's stores, then its arrival
  if (threadIdx.x == 0) {
    __threadfence();
    last = atomicAdd(f.ticket, 1u) == gridDim.x - 1;
  }
  __syncthreads();
  if (!last) return;
  __threadfence();
  box_interface(f, sm);
  if (threadIdx.x == 0) *f.ticket = 0u;
}

// e[i][j] = sum_k (c[k][i] + z[k][i] h[k]) V[j][k] (h: the spectrum of the
// interface values, z the mode's response to them), added to the potential.
// A CTA takes BM rows of 128 columns; the basis comes through shared memory
// kChunkK modes at a time, double-buffered, the first two rounds requested
// before the wait for the preceding kernel (they are static).
template <int BM>
__global__ void __launch_bounds__(kAddThreads) k_box_add(BoxArgs f, int split) {
  extern __shared__ __align__(16) float sm[];
  const int which = int(blockIdx.x) < split ? 0 : 1;
  const BoxBlock &B = f.b[which];
  const int t = int(blockIdx.x) - (which ? split : 0);
  const int n = B.n, m = B.m, mp = B.mp, ncb = (n + kAddThreads - 1) / kAddThreads;
  const int j0 = (t % ncb) * kAddThreads, i0 = (t / ncb) * BM, j = j0 + int(threadIdx.x);
  float *vb = sm;                                  // [2][kChunkK][kAddThreads]
  float *cs = sm + 2 * kChunkK * kAddThreads;      // [n][BM]
  const int rounds = (n + kChunkK - 1) / kChunkK;
  auto fetch = [&](int q) {
    float *d = vb + (q & 1) * kChunkK * kAddThreads;
    const int kk1 = min(kChunkK, n - q * kChunkK);
    if (j < n)
      for (int kk = 0; kk < kk1; ++kk)
        asm volatile("cp.async.ca.shared.global [%0], [%1], 4;\n" ::"r"(
                         unsigned(__cvta_generic_to_shared(d + kk * kAddThreads + threadIdx.x))),
                     "l"(B.vt + size_t(q * kChunkK + kk) * n + j)
                     : "memory");
    asm volatile("cp.async.commit_group;\n" ::: "memory");
  };
  fetch(0);
  if (rounds > 1) fetch(1);
  pdl_enter();
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    f.ps->outer_iters += 1;   // this pass's correction is in the potential once this kernel is done
    f.ps->inner_iters += 1;
    f.ps->total_iters += 1;
  }
  float2 pot[BM];
#pragma unroll
  for (int q = 0; q < BM; ++q)
    pot[q] = j < n && i0 + q < m ? f.pot[size_t(B.row0 + i0 + q) * f.pitch + B.col0 + j] : make_float2(0.f, 0.f);
  const float *h = f.slot ? (which ? f.sh : f.fh) : nullptr;
  for (int u = threadIdx.x; u < n * (BM / 4); u += kAddThreads) {
    const int k = u / (BM / 4), q = (u - k * (BM / 4)) * 4;
    float4 c = *reinterpret_cast<const float4 *>(B.c + size_t(k) * mp + i0 + q);
    if (h) {
      const float4 z = __ldg(reinterpret_cast<const float4 *>(B.z + size_t(k) * mp + i0 + q));
      const float hk = h[k];
      c = make_float4(fmaf(z.x, hk, c.x), fmaf(z.y, hk, c.y), fmaf(z.z, hk, c.z), fmaf(z.w, hk, c.w));
    }
    *reinterpret_cast<float4 *>(cs + k * BM + q) = c;
  }
  float e[BM];
#pragma unroll
  for (int q = 0; q < BM; ++q) e[q] = 0.f;
  for (int r = 0; r < rounds; ++r) {
    if (r + 1 < rounds) asm volatile("cp.async.wait_group 1;\n" ::: "memory");
    else asm volatile("cp.async.wait_group 0;\n" ::: "memory");
    __syncthreads();
    const float *v = vb + (r & 1) * kChunkK * kAddThreads + threadIdx.x;
    const float4 *c4 = reinterpret_cast<const float4 *>(cs + r * kChunkK * BM);
    const int kk1 = min(kChunkK, n - r * kChunkK);
#pragma unroll 8
    for (int kk = 0; kk < kk1; ++kk) {
      const float vv = v[kk * kAddThreads];
#pragma unroll
      for (int q = 0; q < BM / 4; ++q) {
        const float4 c = c4[kk * (BM / 4) + q];
        e[4 * q + 0] = fmaf(c.x, vv, e[4 * q + 0]);
        e[4 * q + 1] = fmaf(c.y, vv, e[4 * q + 1]);
        e[4 * q + 2] = fmaf(c.z, vv, e[4 * q + 2]);
        e[4 * q + 3] = fmaf(c.w, vv, e[4 * q + 3]);
      }
    }
    __syncthreads();
    if (r + 2 < rounds) fetch(r + 2);
  }
  if (j >= n) return;
#pragma unroll
  for (int q = 0; q < BM; ++q)
    if (i0 + q < m) f.pot[size_t(B.row0 + i0 + q) * f.pitch + B.col0 + j] = pair_add_f(pot[q], e[q]);
}

size_t add_smem(const BoxBlock &b, int bm) { return (2 * size_t(kChunkK) * kAddThreads + size_t(b.n) * bm) * 4; }
int add_ctas(const BoxBlock &b, int bm) {
  return ((b.n + kAddThreads - 1) / kAddThreads) * ((b.m + bm - 1) / bm);
}

template <typename T>
T *upload(pic_ctx *c, const std::vector<T> &v) {
  T *d = static_cast<T *>(dev_alloc(c, std::max<size_t>(v.size(), 1) * sizeof(T)));
  if (d && !v.empty() && cudaMemcpy(d, v.data(), v.size() * sizeof(T), cudaMemcpyHostToDevice) != cudaSuccess)
    return nullptr;
  return d;
}

// The basis of a block's columns, its eigenvalues lambda, and the tables of
// its tridiagonal systems.  unit_row: the row whose unit response is kept in
// z (-1: none); ring: the rows close into a ring.
struct BlockTables {
  std::vector<double> basis, lambda, zrow;   // V [n][n], lambda [n], the response at unit_row
};

cudaError_t build_block(pic_ctx *c, BoxBlock &b, bool periodic, int unit_row, bool ring, BlockTables &t) {
  const int n = b.n, m = b.m;
  const double pi = 3.14159265358979323846;
  b.mp = pad8(m);
  b.ldv = pad4(n);
  t.basis.assign(size_t(n) * n, 0.0);
  t.lambda.assign(n, 0.0);
  if (periodic) {
    // orthonormal real Fourier basis: column 0 constant, then cos, sin pairs,
    // and for even n the alternating column
    std::vector<double> cs(n), sn(n);
    for (int q = 0; q < n; ++q) {
      cs[q] = std::cos(2 * pi * q / n);
      sn[q] = std::sin(2 * pi * q / n);
    }
    for (int k = 0; k < n; ++k) {
      const int f = (k + 1) / 2;
      t.lambda[k] = 2.0 - 2.0 * std::cos(2 * pi * f / n);
      const bool single = k == 0 || (n % 2 == 0 && k == n - 1);
      const double s = std::sqrt((single ? 1.0 : 2.0) / n);
      for (int j = 0; j < n; ++j) {
        const int q = int((int64_t(f) * j) % n);
        t.basis[size_t(j) * n + k] = s * ((k % 2 == 0 && k > 0) ? sn[q] : cs[q]);
      }
    }
  } else {
    std::vector<double> sn(2 * (n + 1));
    for (int q = 0; q < 2 * (n + 1); ++q) sn[q] = std::sin(pi * q / (n + 1));
    for (int k = 0; k < n; ++k) {
      t.lambda[k] = 2.0 - 2.0 * std::cos(pi * (k + 1) / (n + 1));
      for (int j = 0; j < n; ++j)
        t.basis[size_t(j) * n + k] =
            std::sqrt(2.0 / (n + 1)) * sn[size_t((int64_t(k + 1) * (j + 1)) % (2 * (n + 1)))];
    }
  }
  std::vector<float> v(size_t(n) * b.ldv, 0.f), vt(size_t(n) * n), w(size_t(n) * b.mp, 0.f), z;
  for (int j = 0; j < n; ++j)
    for (int k = 0; k < n; ++k) {
      const float x = float(t.basis[size_t(j) * n + k]);
      v[size_t(j) * b.ldv + k] = x;
      vt[size_t(k) * n + j] = x;
    }
  // Thomas factors (of rows 1 .. m - 1 for a ring) and the unit response
  const int r0 = ring ? 1 : 0, mr = m - r0;
  if (ring || unit_row >= 0) z.assign(size_t(n) * b.mp, 0.f);
  std::vector<float> rg(n, 0.f);
  std::vector<double> wk(m), y(m);
  t.zrow.assign(n, 0.0);
  for (int k = 0; k < n; ++k) {
    const double d = 2.0 + t.lambda[k];
    double p = 0.0;
    for (int i = 0; i < mr; ++i) {
      p = 1.0 / (d - p);
      wk[i] = p;
      w[size_t(k) * b.mp + r0 + i] = float(p);
    }
    if (z.empty()) continue;
    std::fill(y.begin(), y.end(), 0.0);
    if (ring) y[0] = 1.0, y[mr - 1] += 1.0;
    else y[unit_row] = 1.0;
    for (int i = 0; i < mr; ++i) y[i] = wk[i] * (y[i] + (i > 0 ? y[i - 1] : 0.0));
    for (int i = mr - 2; i >= 0; --i) y[i] += wk[i] * y[i + 1];
    for (int i = 0; i < mr; ++i) z[size_t(k) * b.mp + r0 + i] = float(y[i]);
    if (ring) {
      const double den = d - y[0] - y[mr - 1];
      rg[k] = (c->singular && k == 0) ? 0.f : float(1.0 / den);
    } else {
      t.zrow[k] = y[unit_row];
    }
  }
  b.v = upload(c, v);
  b.vt = upload(c, vt);
  b.w = upload(c, w);
  b.z = z.empty() ? nullptr : upload(c, z);
  b.ring = ring ? upload(c, rg) : nullptr;
  b.c = static_cast<float *>(dev_alloc(c, size_t(n) * b.mp * sizeof(float)));
  if (!b.v || !b.vt || !b.w || !b.c || (!z.empty() && !b.z) || (ring && !b.ring)) return cudaErrorMemoryAllocation;
  return cudaMemsetAsync(b.c, 0, size_t(n) * b.mp * sizeof(float), c->stream);
}

bool invert_spd(std::vector<double> &A, int n) {   // in place, Gauss-Jordan (diagonally dominant enough: no pivoting)
  for (int p = 0; p < n; ++p) {
    const double d = A[size_t(p) * n + p];
    if (!(std::fabs(d) > 1e-300)) return false;
    A[size_t(p) * n + p] = 1.0;
    for (int k = 0; k < n; ++k) A[size_t(p) * n + k] /= d;
    for (int r = 0; r < n; ++r) {
      if (r == p) continue;
      const double q = A[size_t(r) * n + p];
      A[size_t(r) * n + p] = 0.0;
      for (int k = 0; k < n; ++k) A[size_t(r) * n + k] -= q * A[size_t(p) * n + k];
    }
  }
  return true;
}

}  // namespace

BoxArgs box_args(pic_ctx *c, const float *r, float2 *pot, PoissonState *ps) {
  const BoxPoisson &p = c->box;
  BoxArgs a;
  for (int q = 0; q < 2; ++q) {
    a.b[q] = p.b[q];
    a.nblk[q] = q == 0 || p.slot ? (p.b[q].n + kKB - 1) / kKB : 0;
  }
  a.pitch = c->g.nyn;
  a.slot = p.slot;
  a.xs = p.xs;
  a.singular = c->singular;
  a.sinv = p.sinv;
  a.fh = p.fh;
  a.sh = p.sh;
  a.ticket = c->red.ticket + 4;   // spare word
  a.r = r;
  a.pot = pot;
  a.ps = ps;
  return a;
}

// Enabled (automatic method only) for free nodes that form a full slab --
// rows 1 .. m of a bounded x, or every row of a periodic one, all columns of a
// periodic y or all between the walls of a bounded one -- and, below a bounded
// slab, at most one interface row and a slot of at least one row on the same
// run of columns.
cudaError_t box_poisson_setup(pic_ctx *c) {
  BoxPoisson &p = c->box;
  p = BoxPoisson();
  const Geom &g = c->g;
  if (c->cfg.poisson_method != 0) return cudaSuccess;
  // beside the FFT solve only for the passes its closing kernel may add
  if (c->fp.enabled && (c->g.nxn * c->g.nyn > kTailNodes || c->g.nyn > kFftOnceCols)) return cudaSuccess;
  const int nyn = g.nyn, nxn = g.nxn, col0 = g.py ? 0 : 1, n = g.py ? nyn : nyn - 2;
  if (n < 2 || n > kMaxCols) return cudaSuccess;
  auto free_at = [&](int i, int j) { return (c->h_nodeflags[size_t(i) * nyn + j] & kFree) != 0; };
  auto row_count = [&](int i) {
    int q = 0;
    for (int j = 0; j < nyn; ++j) q += free_at(i, j);
    return q;
  };
  auto too_large = [&](int m) {
    const MGLevel &L = c->lev.back();
    return double(m) * n * n > (!g.py           ? kMaxWorkWalls + kMaxWorkCoarsest * L.nxn * L.nyn
                                : c->ncoarse > 0 ? kMaxWorkPeriodic
                                                 : HUGE_VAL);
  };
  BoxBlock &R = p.b[0], &S = p.b[1];
  R.col0 = col0;
  R.n = n;
  BlockTables tr, ts;
  cudaError_t e;
  if (g.px) {
    if (nxn < 3 || nxn > kMaxRows) return cudaSuccess;
    for (int i = 0; i < nxn; ++i)
      if (row_count(i) != n) return cudaSuccess;
    if (too_large(nxn)) return cudaSuccess;
    R.row0 = 0;
    R.m = nxn;
    if ((e = build_block(c, R, g.py != 0, -1, true, tr)) != cudaSuccess) return e;
  } else {
    if (row_count(0) != 0 || row_count(nxn - 1) != 0) return cudaSuccess;
    int xs = 1;
    while (xs < nxn - 1 && row_count(xs) == n) ++xs;
    const int m = xs - 1;
    if (m < 1 || m > kMaxRows || too_large(m)) return cudaSuccess;
    bool slot = false;
    for (int r = xs; r < nxn; ++r) slot = slot || row_count(r) > 0;
    int first = -1, last = -1, ms = 0;
    if (slot) {
      for (int j = 0; j < nyn; ++j)
        if (free_at(xs, j)) {
          if (first < 0) first = j;
          last = j;
        }
      if (first < 0) return cudaSuccess;
      const int wc = last - first + 1;
      if (wc > kMaxSlot || wc >= n || row_count(xs) != wc || (g.py && (first < 1 || last > nyn - 2)))
        return cudaSuccess;
      int r = xs + 1;
      while (r < nxn - 1 && row_count(r) > 0) {
        if (row_count(r) != wc) return cudaSuccess;
        for (int j = first; j <= last; ++j)
          if (!free_at(r, j)) return cudaSuccess;
        ++r;
      }
      for (int rr = r; rr < nxn; ++rr)
        if (row_count(rr) != 0) return cudaSuccess;
      ms = r - xs - 1;
      if (ms < 1 || ms > kMaxRows) return cudaSuccess;
    }
    R.row0 = 1;
    R.m = m;
    if ((e = build_block(c, R, g.py != 0, slot ? m - 1 : -1, false, tr)) != cudaSuccess) return e;
    if (slot) {
      const int wc = last - first + 1, c0 = first - col0;
      S.col0 = first;
      S.n = wc;
      S.row0 = xs + 1;
      S.m = ms;
      if ((e = build_block(c, S, false, 0, false, ts)) != cudaSuccess) return e;
      // Schur complement on the interface: A_GG - G_R - G_S, G the blocks'
      // Green's functions between interface columns
      std::vector<double> A(size_t(wc) * wc, 0.0), vz(n, 0.0);
      for (int a = 0; a < wc; ++a) {
        const double *va = &tr.basis[size_t(c0 + a) * n], *pa = &ts.basis[size_t(a) * wc];
        for (int k = 0; k < n; ++k) vz[k] = va[k] * tr.zrow[k];
        for (int b = 0; b < wc; ++b) {
          const double *vb = &tr.basis[size_t(c0 + b) * n], *pb = &ts.basis[size_t(b) * wc];
          double s = a == b ? 4.0 : (a - b == 1 || b - a == 1) ? -1.0 : 0.0;
          for (int k = 0; k < n; ++k) s -= vz[k] * vb[k];
          for (int k = 0; k < wc; ++k) s -= pa[k] * ts.zrow[k] * pb[k];
          A[size_t(a) * wc + b] = s;
        }
      }
      if (!invert_spd(A, wc)) return cudaSuccess;
      p.sinv = upload(c, std::vector<float>(A.begin(), A.end()));
      p.fh = static_cast<float *>(dev_alloc(c, size_t(n) * sizeof(float)));
      p.sh = static_cast<float *>(dev_alloc(c, size_t(wc) * sizeof(float)));
      if (!p.sinv || !p.fh || !p.sh) return cudaErrorMemoryAllocation;
      p.slot = 1;
      p.xs = xs;
    }
  }
  // rows per CTA of the inverse transform: 8 halves the basis traffic, 4 gives
  // twice the CTAs where 8 would leave SMs idle
  p.bm = add_ctas(R, 8) >= c->num_sms ? 8 : 4;
  p.solve_smem = std::max(box_solve_smem(R), (size_t(n) + 3 * kMaxSlot) * 4);
  p.add_smem = add_smem(R, p.bm);
  if (p.slot) {
    p.solve_smem = std::max(p.solve_smem, box_solve_smem(S));
    p.add_smem = std::max(p.add_smem, add_smem(S, p.bm));
  }
  constexpr size_t kSmem = 220 * 1024;   // the largest size any context may use
  if (p.solve_smem > kSmem || p.add_smem > kSmem) return cudaSuccess;
  e = cudaFuncSetAttribute(k_box_solve, cudaFuncAttributeMaxDynamicSharedMemorySize, int(kSmem));
  if (e == cudaSuccess) e = cudaFuncSetAttribute(k_box_add<4>, cudaFuncAttributeMaxDynamicSharedMemorySize, int(kSmem));
  if (e == cudaSuccess) e = cudaFuncSetAttribute(k_box_add<8>, cudaFuncAttributeMaxDynamicSharedMemorySize, int(kSmem));
  if (e != cudaSuccess) return e;
  p.enabled = c->fp.enabled ? 0 : 1;
  if ((e = box_tail_setup(c)) != cudaSuccess) return e;
  return cudaGetLastError();
}

void box_poisson_launch(pic_ctx *c, const float *r, float2 *pot, PoissonState *ps) {
  const BoxPoisson &p = c->box;
  const BoxArgs a = box_args(c, r, pot, ps);
  launch(k_box_solve, a.nblk[0] + a.nblk[1], kBoxThreads, p.solve_smem, c->stream, a);
  c->launches += 2;
  const int s0 = add_ctas(p.b[0], p.bm), s1 = p.slot ? add_ctas(p.b[1], p.bm) : 0;
  if (p.bm == 8) launch(k_box_add<8>, s0 + s1, kAddThreads, p.add_smem, c->stream, a, s0);
  else launch(k_box_add<4>, s0 + s1, kAddThreads, p.add_smem, c->stream, a, s0);
}

}  // namespace picgb
