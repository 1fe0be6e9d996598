// Cloud-in-cell deposit that allocates nothing (pic_deposit_static).
//
// Who needs it: code that may not call cudaMalloc / cudaFree at the point
// where it deposits -- for example a host program whose device memory is
// already fully reserved by another runtime's pool, or a latency-critical
// loop that cannot afford the device-wide synchronisation an allocation or
// release can cause.  Such a caller passes its own input and output buffers;
// the only scratch this entry point uses is the fixed-size accumulator below,
// which lives in the library image on every GPU that loads the library,
// until the process exits.
//
// The arithmetic is the one of the context-based deposit: each particle's
// four bilinear shares are quantised to 2^-20 of its weight (three rounded
// to nearest-even, the fourth the remainder) and summed exactly in 64-bit
// integers, so the result does not depend on particle order.
#include <cuda_runtime.h>

#include "picgb.h"

namespace {

constexpr long long kStaticMaxNodes = 1ll << 20;   // 8 MiB of 64-bit accumulators
constexpr int kThreads = 256;

// The scratch.  In host code this name is only a stand-in for the device
// symbol: its device address comes from cudaGetSymbolAddress below.
static __device__ __align__(256) unsigned long long g_deposit_scratch[kStaticMaxNodes];

// Device address of the scratch in the current context.  It is looked up
// on every call (a cheap host-side query): a cached address would go stale
// when the caller switches to another context of the same device (a
// runtime that drives its own, non-primary context) or after the device
// was reset and the module loaded again.
pic_status scratch_address(unsigned long long **out) {
  void *p = nullptr;
  if (cudaGetSymbolAddress(&p, g_deposit_scratch) != cudaSuccess || !p) return PIC_ECUDA;
  *out = static_cast<unsigned long long *>(p);
  return PIC_OK;
}

__global__ void k_clear(unsigned long long *acc, long long nn) {
  for (long long k = blockIdx.x * (long long)blockDim.x + threadIdx.x; k < nn;
       k += (long long)gridDim.x * blockDim.x)
    acc[k] = 0ull;
}

// Cell index and FP32 offset of a coordinate in [0, n), n < 2^21, from the bits of
// the double: the integer part by shifts, the offset as the rounded (to
// nearest) fraction, which is what float(X - floor(X)) gives.  FP64 compares,
// floors, differences and conversions run at a small fraction of the FP32
// rate here: a dozen per particle cost more than its memory traffic.
__device__ __forceinline__ void split_coord(unsigned long long bits, int &i, float &f) {
  const int e = int(bits >> 52) - 1023;                                 // sign 0
  const unsigned long long m = (bits & 0xfffffffffffffull) | 0x10000000000000ull;
  const int sh = 52 - e;                                                // X = m 2^-sh
  i = sh <= 52 ? int(m >> sh) : 0;
  const unsigned long long frac = sh <= 52 ? m & ((1ull << sh) - 1ull) : m;
  // 2^-sh as two factors; an offset below 2^-100 (0.0 and denormals among them) gives no share
  f = sh > 150 ? 0.f
               : __fmul_rn(__ull2float_rn(frac), __int_as_float((127 - (sh >> 1)) << 23)) *
                     __int_as_float((127 - (sh - (sh >> 1))) << 23);
  f = fminf(f, 0x1.fffffep-1f);
}

// a double's bits if it lies in [0, n) (n_bits: those of n; -0.0 counts as
// 0), reduced into it first in a periodic direction; else all ones
__device__ __forceinline__ unsigned long long in_box(double X, int n, unsigned long long n_bits, int periodic) {
  unsigned long long b = (unsigned long long)__double_as_longlong(X);
  if (b == 0x8000000000000000ull) b = 0;
  if (b >= n_bits && periodic) {
    X = fmod(X, double(n));
    if (X < 0) X += n;
    if (X >= n) X -= n;
    b = (unsigned long long)__double_as_longlong(X);
    if (b == 0x8000000000000000ull) b = 0;
  }
  return b < n_bits ? b : ~0ull;
}

// One particle per lane finds its cell and shares; then four lanes at a time
// add one particle's four, so that an instruction's atomics fall on a quarter
// of the particles, each with neighbouring addresses: the L2 takes them a
// 32-byte sector at a time.  With PAIRS the scratch keeps, per cell row i and
// node column j, the sum for node (i, j) and that for node (i + 1, j) side by
// side (k_finish joins the two a node has), which puts all four shares of a
// cell into 32 consecutive bytes, one or two sectors; without, the two rows'
// sums lie apart.  8.4M particles on 1024 x 512: 303 us a call with four
// scattered atomics a lane and FP64 arithmetic, 90 us so (a copy of the
// particles' 134 MB: 20 us; the L2's atomics are the bound).
constexpr int kDepThreads = 256;
template <bool PAIRS>
__global__ void __launch_bounds__(kDepThreads) k_deposit(const double *x, const double *y, long long n, int nx, int ny,
                                                         int px, int py, int nyn, unsigned long long *acc) {
  __shared__ int4 s_w[kDepThreads], s_at[kDepThreads];   // shares; their places (x < 0: dropped)
  const float q = 1048576.0f;   // 2^20
  const int lane = threadIdx.x & 31, w0 = threadIdx.x & ~31;
  const unsigned long long xb = (unsigned long long)__double_as_longlong(double(nx));
  const unsigned long long yb = (unsigned long long)__double_as_longlong(double(ny));
  const int *shares = reinterpret_cast<const int *>(s_w + w0), *places = reinterpret_cast<const int *>(s_at + w0);
  for (long long k0 = blockIdx.x * (long long)blockDim.x + w0; k0 < n; k0 += (long long)gridDim.x * blockDim.x) {
    const long long k = k0 + lane;
    int4 at = make_int4(-1, -1, -1, -1), w = make_int4(0, 0, 0, 0);
    if (k < n) {
      const unsigned long long X = in_box(x[k], nx, xb, px), Y = in_box(y[k], ny, yb, py);
      if (X != ~0ull && Y != ~0ull) {   // else outside the grid: skipped
        int i, j;
        float fx, fy;
        split_coord(X, i, fx);
        split_coord(Y, j, fy);
        const float gx = __fsub_rn(1.0f, fx), gy = __fsub_rn(1.0f, fy);
        w.x = __float2int_rn(__fmul_rn(__fmul_rn(gx, gy), q));   // (i, j)
        w.y = __float2int_rn(__fmul_rn(__fmul_rn(fx, gy), q));   // (i + 1, j)
        w.z = __float2int_rn(__fmul_rn(__fmul_rn(gx, fy), q));   // (i, j + 1)
        w.w = int(1u << 20) - w.x - w.y - w.z;                   // (i + 1, j + 1)
        int j1 = j + 1;
        if (py && j1 == ny) j1 = 0;
        if (PAIRS) {
          const int r = 2 * i * nyn;
          at = make_int4(r + 2 * j, r + 2 * j + 1, r + 2 * j1, r + 2 * j1 + 1);
        } else {
          int i1 = i + 1;
          if (px && i1 == nx) i1 = 0;
          at = make_int4(i * nyn + j, i1 * nyn + j, i * nyn + j1, i1 * nyn + j1);
        }
      }
    }
    s_w[threadIdx.x] = w;
    s_at[threadIdx.x] = at;
    __syncwarp();
#pragma unroll
    for (int r = 0; r < 4; ++r) {
      const int p = places[32 * r + lane], v = shares[32 * r + lane];   // particle 8 r + lane / 4, share lane mod 4
      if (p >= 0) atomicAdd(&acc[p], (unsigned long long)(long long)v);
    }
    __syncwarp();
  }
}

// rho from the sums; with pairs, node (i, j) has one from cell row i (none
// above the last) and one from cell row i - 1 (the last row of a box periodic in x)
__global__ void k_finish(const unsigned long long *acc, int nxn, int nyn, int nx, int px, int pairs, double scale,
                         double *rho) {
  const long long nn = (long long)nxn * nyn;
  for (long long k = blockIdx.x * (long long)blockDim.x + threadIdx.x; k < nn;
       k += (long long)gridDim.x * blockDim.x) {
    unsigned long long v;
    if (pairs) {
      const int i = int(k / nyn), j = int(k - (long long)i * nyn), im = i > 0 ? i - 1 : (px ? nx - 1 : -1);
      v = i < nx ? acc[2 * ((long long)i * nyn + j)] : 0ull;
      if (im >= 0) v += acc[2 * ((long long)im * nyn + j) + 1];
    } else {
      v = acc[k];
    }
    rho[k] = scale * double((long long)v);   // two's complement: a sum can be slightly negative
  }
}

int grid_for(long long n) {
  long long b = (n + kThreads - 1) / kThreads;
  if (b < 1) b = 1;
  if (b > 4096) b = 4096;
  return int(b);
}

// Launches one kernel and returns the error of this launch alone (the
// runtime's thread-wide last-error state is neither read nor cleared).
cudaError_t launch1(const void *k, long long work, void **args, cudaStream_t s) {
  return cudaLaunchKernel(k, dim3(unsigned(grid_for(work))), dim3(kThreads), args, 0, s);
}

}  // namespace

extern "C" pic_status pic_deposit_static(int32_t nx, int32_t ny, int32_t periodic_x,
                                         int32_t periodic_y, int64_t n, const double *x,
                                         const double *y, double weight, double *rho,
                                         void *stream) {
  if (nx < 1 || ny < 1 || n < 0 || !rho || (n > 0 && (!x || !y))) return PIC_EINVAL;
  const long long nxn = periodic_x ? nx : (long long)nx + 1;
  const long long nyn = periodic_y ? ny : (long long)ny + 1;
  long long nn = nxn * nyn;
  if (nn > kStaticMaxNodes) return PIC_ESIZE;
  unsigned long long *acc = nullptr;
  const pic_status st = scratch_address(&acc);
  if (st != PIC_OK) return st;
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  int ix = nx, iy = ny, px = periodic_x ? 1 : 0, py = periodic_y ? 1 : 0, inxn = int(nxn), inyn = int(nyn);
  long long np = n;
  double scale = weight / 1048576.0;
  // two sums per cell row and node column where the scratch has room for them and the
  // particles are worth its clearing and reading twice the sums (us with and without
  // pairs: 1024 x 512 with 100 particles 16.6 : 14.6, with 200k 18.7 : 18.6, with 4M 48 : 60;
  // 20 x 20 with 1000 11.0 : 9.5, with 20k 12.9 : 13.5, with 4M 318 : 955)
  int pairs = n >= 8192 && 2 * n >= nn && 2ll * nx * nyn <= kStaticMaxNodes ? 1 : 0;
  long long used = pairs ? 2ll * nx * nyn : nn;
  // the scratch keeps the previous call's sums: clear the part this call uses
  void *a_clear[] = {&acc, &used};
  void *a_dep[] = {&x, &y, &np, &ix, &iy, &px, &py, &inyn, &acc};
  void *a_fin[] = {&acc, &inxn, &inyn, &ix, &px, &pairs, &scale, &rho};
  const void *dep = pairs ? (const void *)k_deposit<true> : (const void *)k_deposit<false>;
  if (launch1((const void *)k_clear, used, a_clear, s) != cudaSuccess) return PIC_ECUDA;
  if (n > 0 && launch1(dep, n, a_dep, s) != cudaSuccess) return PIC_ECUDA;
  if (launch1((const void *)k_finish, nn, a_fin, s) != cudaSuccess) return PIC_ECUDA;
  return PIC_OK;
}
