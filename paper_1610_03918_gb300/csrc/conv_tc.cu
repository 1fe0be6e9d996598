// 3x3 convolutions of the warm-start U-Net on the fifth-generation tensor
// cores: an implicit GEMM whose products run as tcgen05.mma with the FP32
// accumulator in tensor memory (TMEM), operands staged in shared memory by
// the tensor memory accelerator (TMA).
//
// out[b][h][w][n] = act(bias[n] + sum_{dy,dx,c} in[b][h+dy-1][w+dx-1][c] W[n][3 dy + dx][c])
// with BF16 tensors in NHWC (channel slices given by a channel stride and
// offset), FP32 accumulation, act = ReLU or identity, zero padding.
//
// Images at least 128 pixels wide whose channels fit run on the row kernel
// (k_conv_rows), the transposed convolutions and their data gradients on
// k_up_tiles, both persistent; the weight gradients on k_wgrad_rows and
// k_upwgrad_tc, with both operands MN-major; the rest on the tile kernel:
//
// One CTA computes a tile of M = 128 output pixels (a BH x BW block of one
// image, BW = min(W, 128) rounded down to a power of two) for a block of N
// output channels: all of them, or, for layers with fewer pixel tiles than
// SMs, one of the column blocks that the grid's second index selects.  The
// K loop runs over the 9 taps times cin / KB channel blocks.  For each block
// a 4-D TMA box {KB channels, BW, BH, 1} of the input,
// shifted by the tap, lands in shared memory in the swizzled K-major layout
// the MMA reads (zero fill supplies the padding), and a 2-D box {KB, N} of
// the weights [cout][9][cin] beside it.  Warp 0 lane 0 issues the TMA loads
// into a ring of stages (mbarrier expect-tx), warp 1 lane 0 issues KB / 16
// MMAs of 128 x N x 16 per stage and releases the stage by tcgen05.commit;
// then all four warps read their 32 TMEM lanes (one pixel per thread),
// add the bias, apply the activation and store BF16.  Every wait is bounded:
// a wait that gives up sets the error word and the CTA winds down (releasing
// its TMEM) instead of hanging.
//
// The same kernel, in further modes, computes the 2x2 stride-2 transposed
// convolution and its data gradient where the channels are no multiples of 32.
#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <cudaTypedefs.h>

#include <algorithm>
#include <mutex>

#include "internal.cuh"

namespace picgb {
namespace tc {

typedef __nv_bfloat16 bf16;

constexpr int kM = 128;            // output pixels per CTA = TMEM lanes
constexpr int kThreads = 128;      // four warps
constexpr uint64_t kWaitNs = 2000000000ull;   // a wait gives up after 2 s (globaltimer)

// ---------------------------------------------------------------- PTX wrappers
__device__ __forceinline__ uint32_t saddr(const void *p) {
  return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}
__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_expect_tx(uint32_t bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}
__device__ __forceinline__ bool mbar_try(uint32_t bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok)
      : "r"(bar), "r"(parity)
      : "memory");
  return ok != 0;
}
__device__ __forceinline__ uint64_t gtime() {
  uint64_t t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}
// wait for the phase of the given parity to complete, giving up after kWaitNs
// of wall time (one poll may itself suspend for a while, so the number of
// polls alone would not bound the time)
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity) {
  if (mbar_try(bar, parity)) return true;
  const uint64_t t0 = gtime();
  do {
    if (mbar_try(bar, parity)) return true;
  } while (gtime() - t0 < kWaitNs);
  return false;
}
__device__ __forceinline__ void tma_load_4d(uint32_t dst, const CUtensorMap *map, int c0, int c1, int c2,
                                            int c3, uint32_t bar) {
  asm volatile(
      "cp.async.bulk.tensor.4d.shared::cluster.global.tile.mbarrier::complete_tx::bytes "
      "[%0], [%1, {%2, %3, %4, %5}], [%6];" ::"r"(dst),
      "l"(reinterpret_cast<uint64_t>(map)), "r"(c0), "r"(c1), "r"(c2), "r"(c3), "r"(bar)
      : "memory");
}
__device__ __forceinline__ void tma_load_5d(uint32_t dst, const CUtensorMap *map, int c0, int c1, int c2,
                                            int c3, int c4, uint32_t bar) {
  asm volatile(
      "cp.async.bulk.tensor.5d.shared::cluster.global.tile.mbarrier::complete_tx::bytes "
      "[%0], [%1, {%2, %3, %4, %5, %6}], [%7];" ::"r"(dst),
      "l"(reinterpret_cast<uint64_t>(map)), "r"(c0), "r"(c1), "r"(c2), "r"(c3), "r"(c4), "r"(bar)
      : "memory");
}
__device__ __forceinline__ void tma_load_2d(uint32_t dst, const CUtensorMap *map, int c0, int c1,
                                            uint32_t bar) {
  asm volatile(
      "cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes "
      "[%0], [%1, {%2, %3}], [%4];" ::"r"(dst),
      "l"(reinterpret_cast<uint64_t>(map)), "r"(c0), "r"(c1), "r"(bar)
      : "memory");
}
// tcgen05.alloc waits, without a limit, for columns that other CTAs of the SM hold.
// So a kernel here takes its columns in warp 0, waits for the grid before it
// (pdl_wait), and lets the next grid's CTAs in (pdl_release) only after a barrier
// behind the allocation: when they become resident, every CTA of this grid holds its
// columns.  Released earlier, they could take the SM's last columns and wait for
// this grid's end while a CTA of this grid waits for columns.
__device__ __forceinline__ void tmem_alloc(uint32_t slot, uint32_t ncols) {
  asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(slot), "r"(ncols)
               : "memory");
  asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tmem_dealloc(uint32_t taddr, uint32_t ncols) {
  asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(ncols) : "memory");
}
__device__ __forceinline__ void tc_fence_before() {
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
}
__device__ __forceinline__ void tc_fence_after() {
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
}
// D[tmem] (+)= A[smem] . B[smem]^T, M = 128, N from the instruction descriptor, K = 16
__device__ __forceinline__ void mma_bf16(uint32_t tmem_d, uint64_t da, uint64_t db, uint32_t idesc,
                                         uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(tmem_d),
      "l"(da), "l"(db), "r"(idesc), "r"(accumulate)
      : "memory");
}
// the same from the low words of the descriptors; their high words (stride,
// version, swizzle) are one constant
__device__ __forceinline__ void mma_bf16_lo(uint32_t tmem_d, uint32_t da, uint32_t db, uint32_t hi, uint32_t idesc,
                                            uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t.reg .b64 a, b;\n\t"
      "setp.ne.b32 p, %5, 0;\n\t"
      "mov.b64 a, {%1, %3};\n\t"
      "mov.b64 b, {%2, %3};\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], a, b, %4, p;\n\t}" ::"r"(tmem_d),
      "r"(da), "r"(db), "r"(hi), "r"(idesc), "r"(accumulate)
      : "memory");
}
// the same with a high word for each operand
__device__ __forceinline__ void mma_bf16_lo(uint32_t tmem_d, uint32_t da, uint32_t ha, uint32_t db, uint32_t hb,
                                            uint32_t idesc, uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t.reg .b64 a, b;\n\t"
      "setp.ne.b32 p, %6, 0;\n\t"
      "mov.b64 a, {%1, %2};\n\t"
      "mov.b64 b, {%3, %4};\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], a, b, %5, p;\n\t}" ::"r"(tmem_d),
      "r"(da), "r"(ha), "r"(db), "r"(hb), "r"(idesc), "r"(accumulate)
      : "memory");
}
// One lane of a converged warp.  The MMA warps run their loops with all lanes
// and issue from one: control flow and descriptors then stay warp-uniform, in
// uniform registers, where a lone thread's code spent 25 instructions -- about
// 100 cycles -- on moving each MMA's descriptors there (N = 64: 48 cycles of
// tensor core).
__device__ __forceinline__ bool elect_one() {
  uint32_t p;
  asm volatile(
      "{\n\t.reg .pred q;\n\t"
      "elect.sync _|q, 0xffffffff;\n\t"
      "selp.u32 %0, 1, 0, q;\n\t}"
      : "=r"(p));
  return p != 0;
}
// mbar_wait for a whole warp: the answer is warp-uniform
__device__ __forceinline__ bool mbar_wait_warp(uint32_t bar, uint32_t parity) {
  return __all_sync(0xffffffffu, mbar_wait(bar, parity)) != 0;
}
// this thread's warp index, known to the compiler as warp-uniform
__device__ __forceinline__ int warp_index() { return __shfl_sync(0xffffffffu, int(threadIdx.x >> 5), 0); }

// arrives on the mbarrier once every MMA this thread issued before has completed
__device__ __forceinline__ void mma_commit(uint32_t bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar)
               : "memory");
}
// 32 lanes x 16 consecutive 32-bit columns: register k of lane l = TMEM[lane base + l][col + k]
__device__ __forceinline__ void tmem_ld16(uint32_t taddr, uint32_t (&r)[16]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 "
      "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]),
        "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]),
        "=r"(r[14]), "=r"(r[15])
      : "r"(taddr));
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
}

// two floats, BF16-rounded, lo in the low half; with relu, negative values and NaN become 0
__device__ __forceinline__ uint32_t bf16_pair(float lo, float hi, bool relu) {
  __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);
  if (relu) v = __hmax2(v, __floats2bfloat162_rn(0.f, 0.f));
  return *reinterpret_cast<uint32_t *>(&v);
}
// 16 BF16 values as one 32-byte store, or two of 16 bytes.  A thread's pixel is
// 64 bytes or more from its neighbour's, so a 16-byte store fills half a sector:
// with whole ones the transposed convolutions of a 1032 x 512 pass take 47.7
// instead of 55 us, the input convolution 21.8 instead of 24.
__device__ __forceinline__ void store16(bf16 *dst, const uint32_t (&o)[8], bool wide) {
  if (wide) {
    asm volatile("st.global.v8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"l"(dst), "r"(o[0]), "r"(o[1]), "r"(o[2]),
                 "r"(o[3]), "r"(o[4]), "r"(o[5]), "r"(o[6]), "r"(o[7])
                 : "memory");
  } else {
    reinterpret_cast<uint4 *>(dst)[0] = make_uint4(o[0], o[1], o[2], o[3]);
    reinterpret_cast<uint4 *>(dst)[1] = make_uint4(o[4], o[5], o[6], o[7]);
  }
}

// Shared-memory matrix descriptor of a K-major operand tile in the swizzled
// layout TMA wrote: start address, the (unused) leading byte offset, the
// stride between groups of 8 rows (8 x row bytes), the descriptor version of
// this architecture, and the swizzle mode (2: 128 B, 4: 64 B, 6: 32 B rows).
template <int KB>
struct Swz {
  static constexpr uint32_t row_bytes = KB * 2;
  static constexpr uint64_t layout = KB == 64 ? 2 : (KB == 32 ? 4 : 6);
};
template <int KB>
__device__ __forceinline__ uint64_t smem_desc(uint32_t addr) {
  return uint64_t((addr & 0x3FFFF) >> 4) | (uint64_t(1) << 16) |
         (uint64_t((8 * Swz<KB>::row_bytes) >> 4) << 32) | (uint64_t(1) << 46) | (Swz<KB>::layout << 61);
}
// Instruction descriptor of kind::f16: FP32 accumulator, BF16 A and B, both
// K-major, N / 8 and M / 16.
template <int N>
__host__ __device__ constexpr uint32_t instr_desc() {
  return (1u << 4) | (1u << 7) | (1u << 10) | (uint32_t(N >> 3) << 17) | (uint32_t(kM >> 4) << 24);
}

struct TCArgs {
  bf16 *out;
  int out_cs, out_off;
  const float *bias;   // [cout] or null
  int relu;
  int B, H, W, cin, in_off;
  int BW, BH, tiles_w, tiles_h;
  int n_base;          // first GEMM column of this launch; CTA row y of the grid adds y N
  int up_cout;         // transposed convolution: output channels (GEMM column n = (2a + c) up_cout + co)
  int ncols;           // data gradient of the transposed convolution: GEMM columns (weight rows per tap)
  int wide;            // 32-byte stores are aligned
  int *err;            // error word: 1 producer, 2 MMA, 3 epilogue wait gave up
};

constexpr int kHaloPix = kM + 2;   // one image row of the tile and its two neighbours

// Shared memory of one CTA: STAGES A stages, then STAGES B stages, then the
// barriers.  Per stage, A is the 128 x KB input tile of one tap, or (HALO) the
// 130 x KB input row of one vertical tap, and B is the N x KB weight tile of
// one tap, or (HALO) the three horizontal taps' tiles side by side.
template <int N, int KB, int STAGES, bool HALO = false>
struct Layout {
  static constexpr uint32_t B_TILE = N * KB * 2;
  static constexpr uint32_t A_BYTES = HALO ? ((kHaloPix * KB * 2 + 1023) / 1024) * 1024 : kM * KB * 2;
  static constexpr uint32_t A_TX = HALO ? kHaloPix * KB * 2 : kM * KB * 2;   // bytes TMA writes
  static constexpr uint32_t B_BYTES = (HALO ? 3 : 1) * B_TILE;
  static constexpr uint32_t BAR_OFF = STAGES * (A_BYTES + B_BYTES);
  static constexpr uint32_t BYTES = BAR_OFF + (2 * STAGES + 1) * 8 + 16 + 1024;   // + alignment slack
  static constexpr uint32_t NCOLS = N < 32 ? 32 : N;
};

// UP: the 2x2 stride-2 transposed convolution instead of the 3x3 one -- one
// tap (the input pixel itself), GEMM columns n = (2a + c) up_cout + co, and
// the result of input pixel (y, x) written to output pixel (2y + a, 2x + c).
// HALO (tiles of one image row, BW = 128): the K loop runs over the three
// vertical taps times the channel blocks; each step loads the 130-pixel input
// row once and the three horizontal taps read it from rows 0, 1, 2 -- the
// MMA's start address moves by whole swizzled rows, and the swizzle follows
// the shared-memory address, so the shifted operand is the tap's tile.  That
// moves a third of the input bytes of nine shifted tiles.
// UPB: the data gradient of the transposed convolution.  Input pixel (y, x)
// of that convolution gathers, over its four children (2y + a, 2x + c), the
// output gradient's channels: four taps t = 2a + c, each a 5-D box {KB, 1,
// BW, 1, BH} of the gradient viewed as {channels, c, x, a, image rows} -- the
// rows of the tap's 128 pixels, in the same K-major layout as the other
// modes.  B: the weights [4 ncols][cout], rows t ncols + n.
template <int N, int KB, int STAGES, bool UP, bool HALO = false, bool UPB = false>
__global__ void __launch_bounds__(kThreads, 1)
    k_conv3x3_tc(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB, TCArgs a) {
  static_assert(!(UP && HALO), "the transposed convolution has one tap");
  static_assert(!(UPB && (UP || HALO)), "one mode at a time");
  using L = Layout<N, KB, STAGES, HALO>;
  extern __shared__ uint8_t smem_raw[];
  uint8_t *smem = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  const uint32_t sA = saddr(smem), sB = sA + STAGES * L::A_BYTES;
  const uint32_t bar0 = sA + L::BAR_OFF;           // full[s] = bar0 + 8 s, empty[s] = bar0 + 8 (STAGES + s)
  const uint32_t done = bar0 + 16 * STAGES;
  uint32_t *slot = reinterpret_cast<uint32_t *>(smem + L::BAR_OFF + (2 * STAGES + 1) * 8);
  __shared__ int s_fail;

  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  int t = blockIdx.x;
  const int tw = t % a.tiles_w;
  t /= a.tiles_w;
  const int th = t % a.tiles_h;
  const int b = t / a.tiles_h;
  const int w0 = tw * a.BW, h0 = th * a.BH;
  const int nb0 = a.n_base + int(blockIdx.y) * N;   // this CTA's first GEMM column

  if (tid == 0) {
    for (int s = 0; s < STAGES; ++s) {
      mbar_init(bar0 + 8 * s, 1);
      mbar_init(bar0 + 8 * (STAGES + s), 1);
    }
    mbar_init(done, 1);
    s_fail = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 0) tmem_alloc(saddr(slot), L::NCOLS);
  pdl_wait();
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  pdl_release();
  const uint32_t tmem = *slot;
  const int kchunks = a.cin / KB;
  const int nk = (UP ? 1 : (HALO ? 3 : (UPB ? 4 : 9))) * kchunks;

  if (tid == 0) {
    // TMA producer: stage s of round r is reused once the MMAs of round r - 1 released it
    for (int kb = 0; kb < nk; ++kb) {
      const int s = kb % STAGES;
      const uint32_t ph = (kb / STAGES) & 1;
      if (kb >= STAGES && !mbar_wait(bar0 + 8 * (STAGES + s), ph ^ 1)) {
        atomicExch(&s_fail, 1);
        atomicCAS(a.err, 0, 1);
        break;
      }
      if (s_fail) break;
      if (UPB) {
        const int tap = kb / kchunks, c0 = (kb - tap * kchunks) * KB;
        mbar_expect_tx(bar0 + 8 * s, L::A_TX + L::B_BYTES);
        tma_load_5d(sA + s * L::A_BYTES, &tmA, a.in_off + c0, tap & 1, w0, tap >> 1, b * a.H + h0, bar0 + 8 * s);
        tma_load_2d(sB + s * L::B_BYTES, &tmB, c0, tap * a.ncols + nb0, bar0 + 8 * s);
        continue;
      }
      if (HALO) {
        const int dy = kb / kchunks, c0 = (kb - dy * kchunks) * KB;
        mbar_expect_tx(bar0 + 8 * s, L::A_TX + L::B_BYTES);
        tma_load_4d(sA + s * L::A_BYTES, &tmA, a.in_off + c0, w0 - 1, h0 + dy - 1, b, bar0 + 8 * s);
        for (int dx = 0; dx < 3; ++dx)
          tma_load_2d(sB + s * L::B_BYTES + dx * L::B_TILE, &tmB, (3 * dy + dx) * a.cin + c0, nb0, bar0 + 8 * s);
        continue;
      }
      const int tap = UP ? 4 : kb / kchunks, c0 = (kb - (UP ? 0 : tap) * kchunks) * KB;
      const int dy = tap / 3 - 1, dx = tap - 3 * (tap / 3) - 1;
      mbar_expect_tx(bar0 + 8 * s, L::A_TX + L::B_BYTES);
      tma_load_4d(sA + s * L::A_BYTES, &tmA, a.in_off + c0, w0 + dx, h0 + dy, b, bar0 + 8 * s);
      if (UP)
        tma_load_2d(sB + s * L::B_BYTES, &tmB, c0, nb0, bar0 + 8 * s);
      else
        tma_load_2d(sB + s * L::B_BYTES, &tmB, tap * a.cin + c0, nb0, bar0 + 8 * s);
    }
  } else if (tid == 32) {
    // MMA issuer
    constexpr uint32_t idesc = instr_desc<N>();
    for (int kb = 0; kb < nk; ++kb) {
      const int s = kb % STAGES;
      const uint32_t ph = (kb / STAGES) & 1;
      if (!mbar_wait(bar0 + 8 * s, ph)) {
        atomicExch(&s_fail, 1);
        atomicCAS(a.err, 0, 2);
        break;
      }
      tc_fence_after();
      if (HALO) {
#pragma unroll
        for (int dx = 0; dx < 3; ++dx) {
          const uint64_t da = smem_desc<KB>(sA + s * L::A_BYTES + dx * Swz<KB>::row_bytes);   // row dx on
          const uint64_t db = smem_desc<KB>(sB + s * L::B_BYTES + dx * L::B_TILE);
#pragma unroll
          for (int k = 0; k < KB / 16; ++k)
            mma_bf16(tmem, da + 2 * k, db + 2 * k, idesc, (kb | dx | k) != 0 ? 1u : 0u);
        }
      } else {
        const uint64_t da = smem_desc<KB>(sA + s * L::A_BYTES);
        const uint64_t db = smem_desc<KB>(sB + s * L::B_BYTES);
#pragma unroll
        for (int k = 0; k < KB / 16; ++k)   // 16 elements = 32 bytes along the swizzled row
          mma_bf16(tmem, da + 2 * k, db + 2 * k, idesc, (kb | k) != 0 ? 1u : 0u);
      }
      mma_commit(bar0 + 8 * (STAGES + s));
    }
    mma_commit(done);
  }

  // epilogue: thread (warp w, lane l) owns pixel 32 w + l, the accumulator's TMEM lane
  __syncwarp();
  const bool ok = mbar_wait(done, 0);
  tc_fence_after();
  if (!ok) atomicCAS(a.err, 0, 3);
  const int p = 32 * warp + lane;
  const int h = h0 + p / a.BW, w = w0 + p % a.BW;
  const bool inside = h < a.H && w < a.W;
  const uint32_t tl = tmem + (uint32_t(32 * warp) << 16);
#pragma unroll 1
  for (int n0 = 0; n0 < N; n0 += 16) {
    uint32_t r[16];
    tmem_ld16(tl + n0, r);
    if (ok && !s_fail && inside) {
      // destination and bias of these 16 columns (16 divides up_cout: one (a, c) per chunk)
      bf16 *dst;
      int co;
      if (UP) {
        const int n = nb0 + n0, ac = n / a.up_cout;
        co = n - ac * a.up_cout;
        const int oh = 2 * h + (ac >> 1), ow = 2 * w + (ac & 1);
        dst = a.out + ((size_t(b) * 2 * a.H + oh) * 2 * a.W + ow) * a.out_cs + a.out_off + co;
      } else {
        co = nb0 + n0;
        dst = a.out + ((size_t(b) * a.H + h) * a.W + w) * a.out_cs + a.out_off + co;
      }
      uint32_t o[8];
#pragma unroll
      for (int k = 0; k < 8; ++k) {
        const float b0 = a.bias ? __ldg(a.bias + co + 2 * k) : 0.f, b1 = a.bias ? __ldg(a.bias + co + 2 * k + 1) : 0.f;
        o[k] = bf16_pair(__uint_as_float(r[2 * k]) + b0, __uint_as_float(r[2 * k + 1]) + b1, a.relu != 0);
      }
      store16(dst, o, a.wide != 0);
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 0) tmem_dealloc(tmem, L::NCOLS);
}

// ---------------------------------------------------------------- wide images
// The 3x3 convolution on images at least 128 pixels wide, persistent and by
// input rows.  A CTA keeps the weights of its N output channels in shared
// memory and takes a run of output rows of one 128-pixel column block after
// another; every input row of the run (130 pixels: the row's and a neighbour
// on either side) is loaded once, KB channels a unit, and multiplied at once
// into the up to three output rows it belongs to: the three vertical taps'
// weights lie side by side, [dy = 2 | 1 | 0], as one B operand of 3 N columns,
// and the accumulators of consecutive output rows are consecutive column
// blocks of a TMEM ring of kRing rows, so one MMA covers them.  A horizontal
// tap starts one pixel row further into the unit.
//   warps 0-7  epilogue, rows in turn between warps 0-3 and 4-7 (bias, ReLU,
//              BF16, 32-byte stores)
//   warp 8     TMA        warp 9     MMA
// An output row still sums over (dy, chunk, dx), or with TAPS over (dy, dx,
// chunk), the K order of k_conv3x3_tc for the same layer, so the results are
// the same bit for bit.
// What bounds it: an MMA of 128 x N x 16 takes max(N / 2, 44) cycles for N <= 64
// (it reads A at 128 B a cycle), 56 for 96 and 96 for 192 columns: three taps at
// once cost 56 instead of 3 x 45 at N = 32, 96 instead of 3 x 48 at N = 64.  The
// one-tile CTAs before this were bound by their L2 loads (weights and three
// rows a tile) and by the MMA thread's own instructions.  Cold caches, before
// and now: 32 -> 32 at 1032 x 512 41 -> 17 us (a copy's floor 10), 64 -> 32 46 ->
// 22; batch 4, 64 -> 64 at 516 x 256 79 -> 33, 128 -> 64 104 -> 52 (1.51 PFLOP/s),
// at 258 x 128 128 -> 128 54 -> 29 and 256 -> 128 85 -> 70.
struct RowArgs {
  bf16 *out;
  int out_cs, out_off;
  const float *bias;
  int relu;
  int H, W, in_off, cin;
  int col_blocks;          // 128-pixel column blocks per row
  int tiles;               // B x col_blocks x H output rows of 128 pixels
  int wide;                // 32-byte stores are aligned
  int *err;
  // what the epilogue does beside (Epilogue)
  bf16 *pool;              // kPool: [B][H / 2][W / 2][pool_cs]
  int pool_cs;
  const bf16 *y;           // kBack: [B][H][W][y_cs], channels from y_off
  int y_cs, y_off;
  float *db;
  int db_n;                // kSum: the first db_n output channels are summed
};

// kPool: also the 2 x 2 average pool of the output (H and W even).  kBack: the
// output, a gradient, goes through the ReLU that made y (0 where y is not
// positive) and db[c] gains the sum of what is left.  Both spare a pass over the
// output (k_pool_vec, k_relu_back), which is as long as the convolution: batch 4,
// 32 -> 32 at 1032 x 512 46.8 + 42.5 us -> 55.5 and 45.5 + 64.4 -> 62; 64 -> 64 at
// 516 x 256 32.8 + 13.3 -> 36 and 32.7 + 32.5 -> 48.
// kSum: only the sums, of the output's first channels (the bias gradient of the
// transposed convolution whose output they are; k_colsum took 70 us a pass for it).
enum Epilogue { kPlain, kPool, kBack, kSum };

constexpr int kRowThreads = 320;
constexpr int kRing = 8;                     // accumulators (output rows) in TMEM
constexpr uint32_t kRowSmem = 233472;        // shared memory of an SM for CTAs

template <int N, int KB, int KC>
struct RowCfg {
  static constexpr uint32_t UNIT_TX = kHaloPix * KB * 2;
  static constexpr uint32_t UNIT = (UNIT_TX + 1023) / 1024 * 1024;
  static constexpr uint32_t W_TILE = N * KB * 2;
  static constexpr uint32_t W_BYTES = 9 * KC * W_TILE;
  static constexpr int CPS = N == 32 && KC == 1 ? 2 : 1;   // CTAs per SM (TMEM: kRing N columns each)
  static constexpr int ROOM = (int(kRowSmem / CPS) - int(W_BYTES) - 3072) / int(UNIT);
  static constexpr int S = ROOM < 8 ? ROOM : 8;             // units in the ring
  static_assert(S >= KC && S >= 2, "a whole input row beside the weights");
  static constexpr uint32_t BAR_OFF = W_BYTES + S * UNIT;
  static constexpr uint32_t BYTES = BAR_OFF + (2 * S + 1 + 2 * kRing) * 8 + 16 + 1024;
  static constexpr uint32_t NCOLS = kRing * N;
};

__device__ __forceinline__ void mbar_arrive(uint32_t bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void tmem_ld32(uint32_t taddr, uint32_t (&r)[32]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 "
      "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, "
      "%16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
        "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]),
        "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]),
        "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
      : "r"(taddr));
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
}
// the CTA's runs of output rows, pairs of rows with PAIRS (H even): tiles are
// numbered (image, column block, row)
template <bool PAIRS>
struct Runs {
  int t, t1, H, cbs;
  int b, cb, h0, rows;
  __device__ __forceinline__ Runs(const RowArgs &a)
      : t(first(a.tiles, blockIdx.x)), t1(first(a.tiles, blockIdx.x + 1)), H(a.H), cbs(a.col_blocks) {}
  static __device__ __forceinline__ int first(int tiles, unsigned cta) {
    return PAIRS ? int((long long)(tiles / 2) * cta / gridDim.x) * 2 : int((long long)tiles * cta / gridDim.x);
  }
  __device__ __forceinline__ bool next() {
    if (t >= t1) return false;
    const int col = t / H;
    h0 = t - col * H;
    rows = min(t1 - t, H - h0);
    b = col / cbs;
    cb = col - b * cbs;
    t += rows;
    return true;
  }
};

template <int N, int KB, int KC, bool TAPS, int EPI>
__global__ void __launch_bounds__(kRowThreads, RowCfg<N, KB, KC>::CPS)
    k_conv_rows(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB, RowArgs a) {
  using C = RowCfg<N, KB, KC>;
  constexpr uint32_t S = C::S;
  extern __shared__ uint8_t smem_raw[];
  uint8_t *smem = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  const uint32_t sW = saddr(smem), sU = sW + C::W_BYTES, bar0 = sW + C::BAR_OFF;
  // full[s], empty[s] of the units; the weights; accumulators full, accumulators empty
  const uint32_t wbar = bar0 + 16 * S, tfull = wbar + 8, tempty = tfull + 8 * kRing;
  uint32_t *slot = reinterpret_cast<uint32_t *>(smem + C::BAR_OFF + (2 * S + 1 + 2 * kRing) * 8);
  __shared__ int s_fail;
  const int tid = threadIdx.x, warp = warp_index(), lane = tid & 31;
  __shared__ float4 s_bias[N / 4];
  const int n0 = int(blockIdx.y) * N;
  if (tid == 0) {
    for (uint32_t s = 0; s < 2 * S; ++s) mbar_init(bar0 + 8 * s, 1);
    mbar_init(wbar, 1);
    for (int q = 0; q < kRing; ++q) {
      mbar_init(tfull + 8 * q, 1);
      mbar_init(tempty + 8 * q, 4);
    }
    s_fail = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 0) tmem_alloc(saddr(slot), C::NCOLS);
  pdl_wait();
  if (tid < N) reinterpret_cast<float *>(s_bias)[tid] = a.bias ? a.bias[n0 + tid] : 0.f;
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  pdl_release();
  const uint32_t tmem = *slot;
  volatile int *fail = &s_fail;

  if (warp == 8) {
    if (lane == 0) {
      mbar_expect_tx(wbar, C::W_BYTES);
      for (int dx = 0; dx < 3; ++dx)
        for (int c = 0; c < KC; ++c)
          for (int dy = 0; dy < 3; ++dy)
            tma_load_2d(sW + ((dx * KC + c) * 3 + 2 - dy) * C::W_TILE, &tmB, (3 * dy + dx) * a.cin + c * KB, n0, wbar);
      uint32_t s = 0, ph = 1;   // next unit's slot, and the phase its release completes (the first round waits for none)
      bool ok = true;
      Runs<EPI == kPool> r(a);
      while (ok && r.next())
        for (int q = -1; q <= r.rows && ok && !*fail; ++q)
          for (int c = 0; c < KC && ok; ++c) {
            ok = mbar_wait(bar0 + 8 * (S + s), ph);
            if (!ok) break;
            mbar_expect_tx(bar0 + 8 * s, C::UNIT_TX);
            tma_load_4d(sU + s * C::UNIT, &tmA, a.in_off + c * KB, r.cb * kM - 1, r.h0 + q, r.b, bar0 + 8 * s);
            if (++s == S) {
              s = 0;
              ph ^= 1;
            }
          }
      if (!ok) {
        atomicExch(&s_fail, 1);
        atomicCAS(a.err, 0, 1);
      }
    }
  } else if (warp == 9) {
    const bool leader = elect_one();
    constexpr uint32_t idesc1 = instr_desc<N>(), idn = (N >> 3) << 17;   // one row's columns; what each row adds
    // descriptors: only the address field (16-byte units) varies
    const uint64_t dw64 = smem_desc<KB>(sW);
    const uint32_t dw = uint32_t(dw64), du = uint32_t(smem_desc<KB>(sU)), dhi = uint32_t(dw64 >> 32);
    constexpr uint32_t UN = C::UNIT >> 4, WT = C::W_TILE >> 4;
    bool ok = mbar_wait_warp(wbar, 0);
    uint32_t s0 = 0, ph = 0;   // slot of the input row's first unit and its phase
    uint32_t i0 = 0;           // output rows of the runs before
    Runs<EPI == kPool> r(a);
    while (ok && r.next()) {
      for (int q = -1; q <= r.rows && ok; ++q) {
        // output rows lo .. hi of the run take input row q; row q + 1 starts with it
        const int lo = max(q - 1, 0), hi = min(q + 1, r.rows - 1);
        const bool starts = q + 1 < r.rows;
        if (starts) {
          const uint32_t i = i0 + q + 1;
          ok = mbar_wait_warp(tempty + 8 * (i % kRing), ((i / kRing) & 1) ^ 1) && !__any_sync(0xffffffffu, *fail);
        }
        // their accumulators: up to the end of the TMEM ring, and from its start
        const uint32_t r0 = (i0 + lo) % kRing, cnt = hi - lo + 1, ca = min(cnt, kRing - r0), cb = cnt - ca;
        const uint32_t d0 = tmem + r0 * N, ia = idesc1 + (ca - 1) * idn, ib = idesc1 + (cb - 1) * idn;
        const uint32_t b0 = 1 - q + lo;   // first weight block: dy = q + 1 - lo, stored as 2 - dy
        auto unit = [&](int c) { return s0 + c < S ? s0 + c : s0 + c - S; };
        auto need = [&](int c) {
          ok = ok && mbar_wait_warp(bar0 + 8 * unit(c), s0 + c < S ? ph : ph ^ 1);
          tc_fence_after();
        };
        auto mma = [&](int c, int dx) {
          const uint32_t da = du + unit(c) * UN + dx * (Swz<KB>::row_bytes >> 4);
          const uint32_t db = dw + ((dx * KC + c) * 3 + b0) * WT;
          const bool head = starts && dx == 0 && c == 0;
          if (head && leader) {
            // the starting row's first product replaces what its accumulator held
            const uint32_t old = cnt - 1, oa = min(old, ca), ob = old - oa;
            if (oa) mma_bf16_lo(d0, da, db, dhi, idesc1 + (oa - 1) * idn, 1u);
            if (ob) mma_bf16_lo(tmem, da, db + oa * WT, dhi, idesc1 + (ob - 1) * idn, 1u);
            mma_bf16_lo(tmem + (i0 + hi) % kRing * N, da, db + old * WT, dhi, idesc1, 0u);
          }
          const bool first = !head;
          if (cb == 0) {
            if (leader) {
              if (first) mma_bf16_lo(d0, da, db, dhi, ia, 1u);
#pragma unroll
              for (int k = 1; k < KB / 16; ++k) mma_bf16_lo(d0, da + 2 * k, db + 2 * k, dhi, ia, 1u);
            }
          } else if (leader) {
#pragma unroll
            for (int k = 0; k < KB / 16; ++k)
              if (k > 0 || first) {
                mma_bf16_lo(d0, da + 2 * k, db + 2 * k, dhi, ia, 1u);
                mma_bf16_lo(tmem, da + 2 * k, db + ca * WT + 2 * k, dhi, ib, 1u);
              }
          }
        };
        auto release = [&](int c) {
          if (leader) mma_commit(bar0 + 8 * (S + unit(c)));
        };
        if (TAPS) {
#pragma unroll
          for (int dx = 0; dx < 3; ++dx)
#pragma unroll
            for (int c = 0; c < KC; ++c) {
              if (dx == 0) need(c);
              if (!ok) break;
              mma(c, dx);
              if (dx == 2) release(c);
            }
        } else {
#pragma unroll
          for (int c = 0; c < KC; ++c) {
            need(c);
            if (!ok) break;
#pragma unroll
            for (int dx = 0; dx < 3; ++dx) mma(c, dx);
            release(c);
          }
        }
        if (q >= 1 && leader) mma_commit(tfull + 8 * ((i0 + q - 1) % kRing));   // output row q - 1 is complete
        s0 += KC;
        if (s0 >= S) {
          s0 -= S;
          ph ^= 1;
        }
      }
      i0 += r.rows;
    }
    if (!ok && leader) {
      atomicExch(&s_fail, 1);
      atomicCAS(a.err, 0, 2);
    }
  } else {
    // thread (warp w, lane l) owns pixel 32 (w mod 4) + l, the accumulators' TMEM lane
    const int quad = warp & 3, half = warp >> 2;
    const bool relu = a.relu != 0, wide = a.wide != 0;
    uint32_t i = 0;
    bool ok = true;
    Runs<EPI == kPool> r(a);
    constexpr bool SUMS = EPI == kBack || EPI == kSum;
    const bool sums = EPI == kBack || (EPI == kSum && n0 < a.db_n);
    float sum[SUMS ? N : 1];                 // the thread's columns' sums
    uint32_t above[EPI == kPool ? N / 2 : 1];   // kPool: the output above
    if (SUMS)
#pragma unroll
      for (int k = 0; k < N; ++k) sum[SUMS ? k : 0] = 0.f;
    while (ok && r.next()) {
      const int w = r.cb * kM + 32 * quad + lane;
      const size_t p0 = (size_t(r.b) * a.H + r.h0) * a.W + w;
      bf16 *dst = a.out + p0 * a.out_cs + a.out_off + n0;
      const bf16 *y = EPI == kBack ? a.y + p0 * a.y_cs + a.y_off + n0 : nullptr;
      bf16 *pool = EPI == kPool ? a.pool + ((size_t(r.b) * (a.H / 2) + r.h0 / 2) * (a.W / 2) + w / 2) * a.pool_cs + n0
                                : nullptr;
      for (int t = 0; t < r.rows; ++t, ++i, dst += size_t(a.W) * a.out_cs) {
        if (int((EPI == kPool ? i >> 1 : i) & 1) != half) continue;
        uint4 yv[EPI == kBack ? N / 8 : 1];
        if (EPI == kBack) {
          const uint4 *src = reinterpret_cast<const uint4 *>(y + size_t(t) * a.W * a.y_cs);
#pragma unroll
          for (int k = 0; k < N / 8; ++k) yv[EPI == kBack ? k : 0] = w < a.W ? src[k] : make_uint4(0u, 0u, 0u, 0u);
        }
        const uint32_t acc = i % kRing;
        ok = __all_sync(0xffffffffu, mbar_wait(tfull + 8 * acc, (i / kRing) & 1));
        if (!ok) break;
        tc_fence_after();
        const uint32_t tl = tmem + (uint32_t(32 * quad) << 16) + acc * N;
        constexpr int CH = EPI == kPlain ? 32 : 16;   // columns read at once (the others hold more beside)
#pragma unroll
        for (int c = 0; c < N; c += CH) {
          uint32_t v[CH];
          if constexpr (CH == 32) tmem_ld32(tl + c, v);
          else tmem_ld16(tl + c, v);
          if (c + CH == N) {   // read out: the MMA may use the accumulator again
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(tempty + 8 * acc);
          }
#pragma unroll
          for (int q = 0; q < CH; q += 16) {
            uint32_t o[8];
#pragma unroll
            for (int k = 0; k < 8; k += 2) {
              const float4 b = s_bias[(c + q + 2 * k) / 4];
              const float *x = reinterpret_cast<const float *>(v + q + 2 * k);
              o[k] = bf16_pair(x[0] + b.x, x[1] + b.y, relu);
              o[k + 1] = bf16_pair(x[2] + b.z, x[3] + b.w, relu);
            }
            if (EPI == kBack) {
              const uint32_t *yy = reinterpret_cast<const uint32_t *>(yv + (EPI == kBack ? (c + q) / 8 : 0));
#pragma unroll
              for (int k = 0; k < 8; ++k) {
                o[k] &= __hgt2_mask(*reinterpret_cast<const __nv_bfloat162 *>(yy + k), __floats2bfloat162_rn(0.f, 0.f));
              }
            }
            if (sums && (EPI == kBack || w < a.W)) {   // (the mask is 0 off the image)
#pragma unroll
              for (int k = 0; k < 8; ++k) {
                sum[SUMS ? c + q + 2 * k : 0] += __uint_as_float(o[k] << 16);
                sum[SUMS ? c + q + 2 * k + 1 : 0] += __uint_as_float(o[k] & 0xffff0000u);
              }
            }
            if (w < a.W) store16(dst + c + q, o, wide);
            if (EPI == kPool) {
              if (!(i & 1)) {
#pragma unroll
                for (int k = 0; k < 8; ++k) above[EPI == kPool ? (c + q) / 2 + k : 0] = o[k];
              } else {
                // of the pair of pixels the even lane pools channels 0-7, the odd one 8-15:
                // ((above left + above right) + left) + right
                const bool odd = lane & 1;
                uint32_t m[4];
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                  const uint32_t al = above[EPI == kPool ? (c + q) / 2 + k : 0],
                                 ah = above[EPI == kPool ? (c + q) / 2 + 4 + k : 0];
                  const uint32_t am = odd ? ah : al, bm = odd ? o[4 + k] : o[k];
                  const uint32_t ax = __shfl_xor_sync(0xffffffffu, odd ? al : ah, 1);
                  const uint32_t bx = __shfl_xor_sync(0xffffffffu, odd ? o[k] : o[4 + k], 1);
                  const uint32_t bl = odd ? bx : bm, br = odd ? bm : bx;
                  const float lo = 0.25f * (((0.f + __uint_as_float(am << 16)) + __uint_as_float(ax << 16) +
                                             __uint_as_float(bl << 16)) + __uint_as_float(br << 16));
                  const float hi = 0.25f * (((0.f + __uint_as_float(am & 0xffff0000u)) +
                                             __uint_as_float(ax & 0xffff0000u) + __uint_as_float(bl & 0xffff0000u)) +
                                            __uint_as_float(br & 0xffff0000u));
                  m[k] = bf16_pair(lo, hi, false);
                }
                if (w < a.W)
                  *reinterpret_cast<uint4 *>(pool + size_t(t >> 1) * (a.W / 2) * a.pool_cs + c + q + (odd ? 8 : 0)) =
                      make_uint4(m[0], m[1], m[2], m[3]);
              }
            }
          }
          __syncwarp();
        }
      }
    }
    if (sums) {
#pragma unroll
      for (int c = 0; c < N; c += 32) {
        float mine = 0.f;
#pragma unroll
        for (int k = 0; k < 32; ++k) {
          float x = sum[SUMS ? c + k : 0];
#pragma unroll
          for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
          if (lane == k) mine = x;
        }
        if (EPI == kBack || n0 + c + lane < a.db_n) atomicAdd(&a.db[n0 + c + lane], mine);
      }
    }
    if (!ok && lane == 0) {
      atomicExch(&s_fail, 1);
      atomicCAS(a.err, 0, 3);
    }
  }
  __syncwarp();
  tc_fence_before();
  __syncthreads();
  if (warp == 0) tmem_dealloc(tmem, C::NCOLS);
}

// ---------------------------------------------------------------- 2 x 2 transposed convolutions
// The transposed convolution and its data gradient as persistent kernels: CTAs
// of one tile of k_conv3x3_tc spend most of their few MMAs' time on starting, on
// the weights and on an epilogue that nothing overlaps.  A CTA keeps the weights
// of its N GEMM columns in shared memory and takes tiles of 128 pixels of the
// small image one after another, KB channels a unit; units, accumulators and
// epilogue overlap.
//   kUp:      columns (2a + c) up_cout + co of the tile's 128 pixels go to child
//             (2h + a, 2w + c); K = cin
//   kUpBack:  the data gradient: K = the four children's channels (UPB above)
//   kUpBackY: the same, on through the ReLU that made its target (kBack)
//   warps 0-7  epilogue: warps 0-3 the lower, 4-7 the upper half of the columns
//   warp 8     TMA        warp 9     MMA
// K is summed in the order of k_conv3x3_tc: the same results bit for bit.  Bound
// by memory: cold, batch 4, small image 516 x 256, 64 -> 32 channels 38.9 us (57.4
// before; 203 MB), its gradient with the ReLU 65.8 (45.0 + 32.4; half of each
// 128-byte line of the concatenation's gradient is its other half, 404 MB in all);
// 128 -> 64 at 258 x 128 24.3 (38.5) and 27.9 (26.9 + 18.7).
enum UpMode { kUp, kUpBack, kUpBackY };

struct UpArgs {
  bf16 *out;
  int out_cs, out_off;
  const float *bias;
  int B, H, W;             // the small image
  int log_bw;              // tile: 2^log_bw x 128 / 2^log_bw pixels
  int tiles_w, tiles_h, tiles;
  int in_off, kchunks, units;   // units of KB channels per tap and in all
  int n_base;              // first GEMM column of CTA row 0
  int up_cout;             // kUp: output channels
  int ncols;               // kUpBack: weight rows per child
  int stages;              // units in the ring
  int wide;
  const bf16 *y;
  int y_cs, y_off;
  float *db;
  int *err;
};
constexpr int kUpStages = 8;

template <int N, int KB, int MODE>
__global__ void __launch_bounds__(kRowThreads, 1)
    k_up_tiles(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB, UpArgs a) {
  constexpr int RING = N >= 256 ? 2 : 4;   // accumulators in TMEM
  constexpr uint32_t UNIT = kM * KB * 2, W_TILE = N * KB * 2;
  constexpr int HALF = N / 2;
  extern __shared__ uint8_t smem_raw[];
  uint8_t *smem = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  __shared__ __align__(8) uint64_t s_bar[2 * kUpStages + 1 + 2 * RING];
  __shared__ uint32_t s_slot;
  __shared__ int s_fail;
  __shared__ float4 s_bias[N / 4];
  const uint32_t S = a.stages;
  const uint32_t sW = saddr(smem), sU = sW + a.units * W_TILE;
  const uint32_t full = saddr(s_bar), empty = full + 8 * kUpStages, wbar = empty + 8 * kUpStages, tfull = wbar + 8,
                 tempty = tfull + 8 * RING;
  const int tid = threadIdx.x, warp = warp_index(), lane = tid & 31;
  const int n0 = a.n_base + int(blockIdx.y) * N;
  if (tid == 0) {
    for (int k = 0; k < kUpStages; ++k) {
      mbar_init(full + 8 * k, 1);
      mbar_init(empty + 8 * k, 1);
    }
    mbar_init(wbar, 1);
    for (int k = 0; k < RING; ++k) {
      mbar_init(tfull + 8 * k, 1);
      mbar_init(tempty + 8 * k, 8);
    }
    s_fail = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 0) tmem_alloc(saddr(&s_slot), RING * N);
  pdl_wait();
  if (tid < N)
    reinterpret_cast<float *>(s_bias)[tid] = a.bias ? a.bias[MODE == kUp ? (n0 + tid) % a.up_cout : n0 + tid] : 0.f;
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  pdl_release();
  const uint32_t tmem = s_slot;
  volatile int *fail = &s_fail;
  const int t0 = int((long long)a.tiles * blockIdx.x / gridDim.x);
  const int t1 = int((long long)a.tiles * (blockIdx.x + 1) / gridDim.x);
  const int bw = 1 << a.log_bw, bh = kM >> a.log_bw;

  if (warp == 8) {
    if (lane == 0) {
      mbar_expect_tx(wbar, a.units * W_TILE);
      for (int u = 0; u < a.units; ++u) {
        const int tap = u / a.kchunks, c0 = (u - tap * a.kchunks) * KB;
        tma_load_2d(sW + u * W_TILE, &tmB, c0, tap * a.ncols + n0, wbar);
      }
      uint32_t s = 0, ph = 1;   // next unit's slot, and the phase its release completes
      bool ok = true;
      for (int t = t0; t < t1 && ok && !*fail; ++t) {
        const int r = t / a.tiles_w, w0 = (t - r * a.tiles_w) << a.log_bw;
        const int b = r / a.tiles_h, h0 = (r - b * a.tiles_h) * bh;
        for (int u = 0; u < a.units && ok; ++u) {
          ok = mbar_wait(empty + 8 * s, ph);
          if (!ok) break;
          mbar_expect_tx(full + 8 * s, UNIT);
          if (MODE == kUp) {
            tma_load_4d(sU + s * UNIT, &tmA, a.in_off + u * KB, w0, h0, b, full + 8 * s);
          } else {
            const int tap = u / a.kchunks, c0 = (u - tap * a.kchunks) * KB;
            tma_load_5d(sU + s * UNIT, &tmA, a.in_off + c0, tap & 1, w0, tap >> 1, b * a.H + h0, full + 8 * s);
          }
          if (++s == S) {
            s = 0;
            ph ^= 1;
          }
        }
      }
      if (!ok) {
        atomicExch(&s_fail, 1);
        atomicCAS(a.err, 0, 1);
      }
    }
  } else if (warp == 9) {
    const bool leader = elect_one();
    constexpr uint32_t idesc = instr_desc<N>();
    const uint64_t dw64 = smem_desc<KB>(sW);
    const uint32_t dw = uint32_t(dw64), du = uint32_t(smem_desc<KB>(sU)), dhi = uint32_t(dw64 >> 32);
    bool ok = mbar_wait_warp(wbar, 0);
    uint32_t s = 0, ph = 0;
    for (int t = t0; t < t1 && ok; ++t) {
      const uint32_t i = t - t0, acc = i % RING;
      ok = mbar_wait_warp(tempty + 8 * acc, ((i / RING) & 1) ^ 1) && !__any_sync(0xffffffffu, *fail);
      for (int u = 0; u < a.units && ok; ++u) {
        ok = mbar_wait_warp(full + 8 * s, ph);
        if (!ok) break;
        tc_fence_after();
        if (leader) {
#pragma unroll
          for (int k = 0; k < KB / 16; ++k)
            mma_bf16_lo(tmem + acc * N, du + s * (UNIT >> 4) + 2 * k, dw + u * (W_TILE >> 4) + 2 * k, dhi, idesc,
                        (u | k) != 0 ? 1u : 0u);
          mma_commit(empty + 8 * s);
        }
        if (++s == S) {
          s = 0;
          ph ^= 1;
        }
      }
      if (ok && leader) mma_commit(tfull + 8 * acc);
    }
    if (!ok && leader) {
      atomicExch(&s_fail, 1);
      atomicCAS(a.err, 0, 2);
    }
  } else {
    // thread (warp w, lane l) owns pixel 32 (w mod 4) + l of the tile, the accumulators' TMEM lane
    const int quad = warp & 3, half = warp >> 2;
    const int p = 32 * quad + lane, ph = p >> a.log_bw, pw = p & (bw - 1);
    const int col0 = half * HALF;   // the warp's first column of the accumulator
    const bool wide = a.wide != 0;
    bool ok = true;
    float sum[MODE == kUpBackY ? HALF : 1];
    if (MODE == kUpBackY)
#pragma unroll
      for (int k = 0; k < HALF; ++k) sum[MODE == kUpBackY ? k : 0] = 0.f;
    for (int t = t0; t < t1 && ok; ++t) {
      const uint32_t i = t - t0, acc = i % RING;
      const int r = t / a.tiles_w, w = ((t - r * a.tiles_w) << a.log_bw) + pw;
      const int b = r / a.tiles_h, h = (r - b * a.tiles_h) * bh + ph;
      const bool inside = h < a.H && w < a.W;
      const size_t px = (size_t(b) * a.H + h) * a.W + w;
      uint4 yv[MODE == kUpBackY ? HALF / 8 : 1];
      if (MODE == kUpBackY) {
        const uint4 *src = reinterpret_cast<const uint4 *>(a.y + px * a.y_cs + a.y_off + n0 + col0);
#pragma unroll
        for (int k = 0; k < HALF / 8; ++k) yv[MODE == kUpBackY ? k : 0] = inside ? src[k] : make_uint4(0u, 0u, 0u, 0u);
      }
      ok = __all_sync(0xffffffffu, mbar_wait(tfull + 8 * acc, (i / RING) & 1));
      if (!ok) break;
      tc_fence_after();
      const uint32_t tl = tmem + (uint32_t(32 * quad) << 16) + acc * N + col0;
      // kUp: a child's columns come together
      int ac = MODE == kUp ? (n0 + col0) / a.up_cout : 0, co = n0 + col0 - ac * (MODE == kUp ? a.up_cout : 0);
#pragma unroll
      for (int c = 0; c < HALF; c += 16) {
        uint32_t v[16];
        tmem_ld16(tl + c, v);
        if (c + 16 == HALF) {   // read out: the MMA may use the accumulator again
          tc_fence_before();
          __syncwarp();
          if (lane == 0) mbar_arrive(tempty + 8 * acc);
        }
        uint32_t o[8];
#pragma unroll
        for (int k = 0; k < 8; k += 2) {
          const float4 bs = s_bias[(col0 + c + 2 * k) / 4];
          const float *x = reinterpret_cast<const float *>(v + 2 * k);
          o[k] = bf16_pair(x[0] + bs.x, x[1] + bs.y, false);
          o[k + 1] = bf16_pair(x[2] + bs.z, x[3] + bs.w, false);
        }
        if (MODE == kUpBackY) {
          const uint32_t *yy = reinterpret_cast<const uint32_t *>(yv + (MODE == kUpBackY ? c / 8 : 0));
#pragma unroll
          for (int k = 0; k < 8; ++k) {
            o[k] &= __hgt2_mask(*reinterpret_cast<const __nv_bfloat162 *>(yy + k), __floats2bfloat162_rn(0.f, 0.f));
            sum[MODE == kUpBackY ? c + 2 * k : 0] += __uint_as_float(o[k] << 16);
            sum[MODE == kUpBackY ? c + 2 * k + 1 : 0] += __uint_as_float(o[k] & 0xffff0000u);
          }
        }
        if (inside) {
          const size_t q = MODE == kUp ? (size_t(b) * 2 * a.H + 2 * h + (ac >> 1)) * 2 * a.W + 2 * w + (ac & 1) : px;
          store16(a.out + q * a.out_cs + a.out_off + co, o, wide);
        }
        co += 16;
        if (MODE == kUp && co == a.up_cout) {
          co = 0;
          ac += 1;
        }
        __syncwarp();
      }
    }
    if (MODE == kUpBackY) {
#pragma unroll
      for (int c = 0; c < HALF; c += 32) {
        float mine = 0.f;
#pragma unroll
        for (int k = 0; k < 32; ++k) {
          float x = sum[MODE == kUpBackY ? c + k : 0];
#pragma unroll
          for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
          if (lane == k) mine = x;
        }
        atomicAdd(&a.db[n0 + col0 + c + lane], mine);
      }
    }
    if (!ok && lane == 0) {
      atomicExch(&s_fail, 1);
      atomicCAS(a.err, 0, 3);
    }
  }
  __syncwarp();
  tc_fence_before();
  __syncthreads();
  if (warp == 0) tmem_dealloc(tmem, RING * N);
}

// ---------------------------------------------------------------- first layer
// The network's first 3x3 convolution (2 input channels -> 32) on the tensor
// cores.  The 9 taps x 2 channels of a pixel, BF16-rounded, form one K row of
// 32 (k = 2 tap + c, zeros from 18 on) of an A tile that the threads write to
// shared memory, in the non-swizzled K-major layout: core matrices of 8 rows
// x 16 bytes, 8 K values per plane of 128 rows, planes LBO = 2048 B apart,
// 8-row groups SBO = 128 B apart.  B, the 32 x 32 weight matrix, has the same
// layout (planes of 32 rows).  A CTA takes tiles of 128 consecutive pixels
// (row-major over images, rows and columns) in turn: the threads build A,
// one thread issues two MMAs of K = 16 into the TMEM accumulator and commits,
// and the four warps read their 32 lanes back (bias, activation, BF16).
constexpr int kInCh = 2, kInK = 32, kInN = 32;

__device__ __forceinline__ uint64_t plain_desc(uint32_t addr, uint32_t lbo, uint32_t sbo) {
  return uint64_t((addr & 0x3FFFF) >> 4) | (uint64_t(lbo >> 4) << 16) | (uint64_t(sbo >> 4) << 32) |
         (uint64_t(1) << 46);   // layout type 0: no swizzle
}
__device__ __forceinline__ void fence_async_smem() {
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
}
__device__ __forceinline__ uint32_t pack_bf16(float lo, float hi) {
  const uint32_t a = __bfloat16_as_ushort(__float2bfloat16_rn(lo));
  const uint32_t b = __bfloat16_as_ushort(__float2bfloat16_rn(hi));
  return a | (b << 16);
}

__global__ void __launch_bounds__(kThreads, 1)
    k_conv_in_tc(const float2 *x, const bf16 *w, int wcin, const float *bias, bf16 *out, int B, int H, int W,
                 int relu, int wide, int *err) {
  __shared__ __align__(1024) uint8_t sA[(kInK / 8) * kM * 16];     // 4 planes of 128 rows
  __shared__ __align__(1024) uint8_t sB[(kInK / 8) * kInN * 16];   // 4 planes of 32 rows
  __shared__ __align__(8) uint64_t bar;
  __shared__ uint32_t slot;
  __shared__ float sbias[kInN];
  __shared__ int s_fail;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  if (warp == 0) tmem_alloc(saddr(&slot), kInN);
  pdl_wait();
  // B[n][k] = w[n][tap][c], k = 2 tap + c < 18, else 0
  for (int i = tid; i < kInN * kInK; i += kThreads) {
    const int n = i / kInK, k = i - (i / kInK) * kInK;
    const bf16 v = k < 9 * kInCh ? w[(size_t(n) * 9 + k / kInCh) * wcin + (k % kInCh)] : __float2bfloat16(0.f);
    *reinterpret_cast<bf16 *>(sB + (k / 8) * (kInN * 16) + n * 16 + (k % 8) * 2) = v;
  }
  for (int i = tid; i < kInN; i += kThreads) sbias[i] = bias ? bias[i] : 0.f;
  if (tid == 0) {
    mbar_init(saddr(&bar), 1);
    s_fail = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  pdl_release();
  const uint32_t tmem = slot;
  constexpr uint32_t idesc = instr_desc<kInN>();
  const unsigned npix = unsigned(B) * unsigned(H) * unsigned(W);
  const unsigned ntiles = (npix + kM - 1) / kM;
  uint32_t it = 0;
  for (unsigned tile = blockIdx.x; tile < ntiles; tile += gridDim.x, ++it) {
    // this thread's pixel (the A row tid) and its 9 x 2 inputs, zeros outside
    // the image or past the end
    const unsigned p = tile * kM + unsigned(tid);
    const bool valid = p < npix;
    const unsigned r = valid ? p / unsigned(W) : 0u;
    const int wq = valid ? int(p - r * unsigned(W)) : 0;
    const int h = int(r % unsigned(H));
    float v[2 * 9];
#pragma unroll
    for (int t = 0; t < 9; ++t) {
      const int hh = h + t / 3 - 1, ww = wq + t % 3 - 1;
      float2 e = make_float2(0.f, 0.f);
      if (valid && hh >= 0 && hh < H && ww >= 0 && ww < W) e = x[int(p) + (t / 3 - 1) * W + (t % 3 - 1)];
      v[2 * t] = e.x;
      v[2 * t + 1] = e.y;
    }
    const uint4 q0 = make_uint4(pack_bf16(v[0], v[1]), pack_bf16(v[2], v[3]), pack_bf16(v[4], v[5]), pack_bf16(v[6], v[7]));
    const uint4 q1 = make_uint4(pack_bf16(v[8], v[9]), pack_bf16(v[10], v[11]), pack_bf16(v[12], v[13]),
                                pack_bf16(v[14], v[15]));
    const uint4 q2 = make_uint4(pack_bf16(v[16], v[17]), 0u, 0u, 0u);
    const uint4 q3 = make_uint4(0u, 0u, 0u, 0u);
    reinterpret_cast<uint4 *>(sA + 0 * kM * 16)[tid] = q0;
    reinterpret_cast<uint4 *>(sA + 1 * kM * 16)[tid] = q1;
    reinterpret_cast<uint4 *>(sA + 2 * kM * 16)[tid] = q2;
    reinterpret_cast<uint4 *>(sA + 3 * kM * 16)[tid] = q3;
    fence_async_smem();   // the threads' writes become visible to the tensor core's reads
    __syncthreads();
    if (tid == 0) {
      tc_fence_after();
#pragma unroll
      for (int k = 0; k < kInK / 16; ++k)   // planes 2k, 2k + 1
        mma_bf16(tmem, plain_desc(saddr(sA) + 2 * k * (kM * 16), kM * 16, 128),
                 plain_desc(saddr(sB) + 2 * k * (kInN * 16), kInN * 16, 128), idesc, k ? 1u : 0u);
      mma_commit(saddr(&bar));
    }
    __syncwarp();
    const bool ok = __all_sync(0xffffffffu, mbar_wait(saddr(&bar), it & 1));
    tc_fence_after();
    if (ok) {
      const uint32_t tl = tmem + (uint32_t(32 * warp) << 16);
#pragma unroll
      for (int n0 = 0; n0 < kInN; n0 += 16) {
        uint32_t rr[16];
        tmem_ld16(tl + n0, rr);
        if (valid) {
          uint32_t o[8];
#pragma unroll
          for (int k = 0; k < 8; ++k)
            o[k] = bf16_pair(__uint_as_float(rr[2 * k]) + sbias[n0 + 2 * k],
                             __uint_as_float(rr[2 * k + 1]) + sbias[n0 + 2 * k + 1], relu != 0);
          store16(out + size_t(p) * kInN + n0, o, wide != 0);
        }
      }
    } else if (lane == 0) {
      atomicExch(&s_fail, 1);
      atomicCAS(err, 0, 3);
    }
    tc_fence_before();
    __syncthreads();   // TMEM read and A free for the next tile
    if (s_fail) break;
  }
  if (warp == 0) tmem_dealloc(tmem, kInN);
}

// ---------------------------------------------------------------- weight gradient
// dW[co][3 dy + dx][ci] += sum_p dpre[p][co] in[p + (dy - 1, dx - 1)][ci] (zero
// padding), dpre the gradient before the ReLU [B][H][W][cout], in the layer's
// input.  A K block is KP = 64 consecutive pixels (w0 .. w0 + 63) of one input
// row hq of one image.  Both operands are MN-major: pixels (K) are the rows
// of a swizzled tile, channels (M, N) run along the row.
//  * B, the input: the row hq from pixel w0 - 8 to w0 + KP + 7 (TMA box
//    {CI, KP + 16}; the x coordinate stays a multiple of 8), CI channels.
//    The three horizontal taps are three N chunks of CI channels whose
//    starts lie one pixel row apart (LBO = one row), so N = 3 CI covers
//    dx = 0, 1, 2 at once, each chunk being the input shifted by dx - 1.
//  * A, the gradient: three consecutive slots, slot s the dpre row hq - 1 + s
//    (pixels w0 .. w0 + KP - 1, zero fill off the image), one slot per vertical
//    tap (dpre row hq + 1 - dy meets input row hq at tap dy).  M = 128 rows of D
//    are slots of CO channels at LBO = one slot: CO = 32, four slots in one MMA;
//    CO = 64, slots {0, 1} and {2, 3}.  The fourth is whatever lies there: its
//    rows of D are not read.
// D row (s, co), column (dx, ci) thus accumulates dW[co][3 (2 - s) + dx][ci] over
// the CTA's K blocks; the epilogue adds it to dW with vector atomics (FP32,
// so the sum order, not the terms, depends on the grid).
// A CTA goes down the rows of a pixel column, and each dpre row serves three K
// blocks: a segment of up to NR - 2 input rows starts at slot 0 of the NR with the
// dpre row above it.  Rows come GA (dpre) and GB (input) to a TMA box, because
// what set the pace before was neither the tensor core nor memory but the one
// thread that loaded three dpre rows and an input row anew for every K block:
// 160 cycles a box, 640 a K block of 224 (32 x 32) to 768 (64 x 64) cycles of MMA.
// Cold, batch 4: 64 -> 64 at 516 x 256 51.6 -> 43.8 us (MMA alone 21), 32 -> 32 at
// 1032 x 512 69.0 -> 51.0 (a read of both tensors 40), 256 -> 256 at 129 x 64 70.9 ->
// 49.0.
constexpr int kWKP = 64;   // pixels per K block
constexpr int kWKPB = kWKP + 16;   // the input row with 8-pixel margins

constexpr uint32_t tmem_cols(uint32_t n) {
  return n <= 32 ? 32 : n <= 64 ? 64 : n <= 128 ? 128 : n <= 256 ? 256 : 512;
}

template <int CO, int CI>
struct WRing {
  static constexpr uint32_t SLOT = kWKP * CO * 2;
  static constexpr uint32_t ROW = kWKPB * CI * 2;      // an input row; groups of 8 pixels stay whole
  static constexpr int GA = 4, GB = 2;                 // rows per TMA box
  static constexpr int NR = CO == 32 ? 16 : 12;        // dpre rows
  static constexpr int NB = CI == 64 ? 4 : 3;          // boxes of input rows
  static constexpr int NA = NR / GA;
  static constexpr uint32_t B_OFF = NR * SLOT;
  static constexpr uint32_t BAR_OFF = B_OFF + (NB * GB * ROW + 1023) / 1024 * 1024;
  // allocated, never written: keeps every address the descriptors of the last
  // input row can form inside this CTA's shared memory (the widest reading of
  // the B tile spans 3 CI rows of 8-row groups from row 55)
  static constexpr uint32_t TAIL = 6 * CI * CI + 112 * CI;
  static constexpr uint32_t BYTES = BAR_OFF + (2 * NA + 2 * NB + 1) * 8 + 16 + TAIL + 1024;
  static_assert(BYTES <= 227 * 1024 - 64, "shared memory");
  static constexpr int NM = CO == 32 ? 1 : 2;   // MMAs along M per 16 pixels
  static constexpr int N = 3 * CI;
  // A CTA's K blocks in turn go to NACC accumulators, which the epilogue adds in
  // FP32: the tensor core truncates each sum, so the error grows with the sums
  // an accumulator takes (relative error of 32 -> 32 at 4 x 1032 x 512, over 453
  // accumulators 2.2e-6, over 304 3.5e-6, over 608 1.5e-6).
  static constexpr int NACC = NM * N > 256 ? 1 : 2;
  static constexpr uint32_t NCOLS = tmem_cols(NACC * NM * N);
};

// descriptor of an MN-major tile in the swizzled layout TMA wrote with rows
// of CH channels: K rows CH x 2 bytes apart, groups of 8 rows SBO = 8 rows
// apart, chunks of CH channels along M or N at LBO
template <int CH>
__device__ __forceinline__ uint64_t mn_desc(uint32_t addr, uint32_t lbo) {
  return uint64_t((addr & 0x3FFFF) >> 4) | (uint64_t(lbo >> 4) << 16) |
         (uint64_t((8 * Swz<CH>::row_bytes) >> 4) << 32) | (uint64_t(1) << 46) | (Swz<CH>::layout << 61);
}
// kind::f16 with BF16 A and B, both MN-major (transpose bits 15 and 16)
template <int N>
__host__ __device__ constexpr uint32_t instr_desc_mn() {
  return instr_desc<N>() | (1u << 15) | (1u << 16);
}

struct WRowArgs {
  float *dw;           // [cout][9][cin]
  int cin, cout, in_off, H, nwc;
  long long rows;      // B x nwc pixel columns x H input rows
  int *err;
};

template <int CO, int CI>
__global__ void __launch_bounds__(kThreads, 1)
    k_wgrad_rows(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB, WRowArgs a) {
  using L = WRing<CO, CI>;
  constexpr int NA = L::NA, NB = L::NB, GA = L::GA, GB = L::GB;
  extern __shared__ uint8_t smem_raw[];
  uint8_t *smem = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  const uint32_t s0 = saddr(smem), sB = s0 + L::B_OFF, bar0 = s0 + L::BAR_OFF;
  // boxes of dpre rows full, empty; of input rows full, empty; all done
  const uint32_t afull = bar0, aempty = afull + 8 * NA, bfull = aempty + 8 * NA, bempty = bfull + 8 * NB,
                 done = bempty + 8 * NB;
  uint32_t *slot = reinterpret_cast<uint32_t *>(smem + L::BAR_OFF + (2 * NA + 2 * NB + 1) * 8);
  __shared__ int s_fail;
  const int tid = threadIdx.x, warp = warp_index(), lane = tid & 31;
  const int ncib = a.cin / CI;
  const int co0 = int(blockIdx.y) / ncib * CO, ci0 = int(blockIdx.y) % ncib * CI;
  const long long t0 = a.rows * blockIdx.x / gridDim.x, t1 = a.rows * (blockIdx.x + 1) / gridDim.x;
  const int nacc = int(min(t1 - t0, (long long)L::NACC));   // accumulators in use
  if (tid == 0) {
    for (int k = 0; k < 2 * (NA + NB) + 1; ++k) mbar_init(bar0 + 8 * k, 1);
    s_fail = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 0) tmem_alloc(saddr(slot), L::NCOLS);
  pdl_wait();
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  pdl_release();
  const uint32_t tmem = *slot;
  // the segments: n input rows from h0 of pixel column col
  long long t = t0, col = 0;
  int h0 = 0, n = 0;
  auto next = [&]() {
    if (t >= t1) return false;
    col = t / a.H;
    h0 = int(t - col * a.H);
    n = int(min(min(t1 - t, (long long)(a.H - h0)), (long long)(L::NR - 2)));
    t += n;
    return true;
  };

  if (warp == 0) {
    if (lane == 0) {
      uint32_t phase = ~0u;   // per dpre box: the parity its next release completes (the first round waits for none)
      uint32_t bs = 0, bph = 1;
      bool ok = true;
      while (ok && next()) {
        const int b = int(col / a.nwc), w0 = int(col - (long long)b * a.nwc) * kWKP;
        int g = 0;
        auto load_a = [&]() {
          ok = ok && mbar_wait(aempty + 8 * g, (phase >> g) & 1);
          if (!ok) return;
          phase ^= 1u << g;
          mbar_expect_tx(afull + 8 * g, GA * L::SLOT);
          tma_load_4d(s0 + g * (GA * L::SLOT), &tmA, co0, w0, h0 - 1 + GA * g, b, afull + 8 * g);
          g += 1;
        };
        load_a();
        for (int i = 0; i < n && ok; i += GB) {
          // input rows up to i + GB - 1 need dpre slots up to i + GB + 1 (the last: n + 1)
          if (min(i + GB + 1, n + 1) >= GA * g) load_a();
          ok = ok && mbar_wait(bempty + 8 * bs, bph);
          if (!ok) break;
          mbar_expect_tx(bfull + 8 * bs, GB * L::ROW);
          tma_load_4d(sB + bs * (GB * L::ROW), &tmB, a.in_off + ci0, w0 - 8, h0 + i, b, bfull + 8 * bs);
          if (++bs == NB) {
            bs = 0;
            bph ^= 1;
          }
        }
      }
      if (!ok) {
        atomicExch(&s_fail, 1);
        atomicCAS(a.err, 0, 1);
      }
    }
  } else if (warp == 1) {
    const bool leader = elect_one();
    constexpr uint32_t idesc = instr_desc_mn<L::N>();
    // descriptors: only the address field (16-byte units) varies; input rows from
    // pixel w0 - 1 on (row 7 of a box row), the tap dx = 0 chunk
    const uint64_t a64 = mn_desc<CO>(s0, L::SLOT), b64 = mn_desc<CI>(sB + 7 * (CI * 2), CI * 2);
    const uint32_t da = uint32_t(a64), ha = uint32_t(a64 >> 32), db = uint32_t(b64), hb = uint32_t(b64 >> 32);
    uint32_t phase = 0;       // per dpre box: the parity its next load completes
    uint32_t bs = 0, bph = 0;
    uint32_t acc = 0, any = 0;             // the accumulator, whether it holds anything
    long long rows = 0, until = (t1 - t0) / nacc;   // K blocks so far, those up to the next accumulator
    bool ok = true;
    while (ok && next()) {
      int g = 0, freed = 0;   // dpre boxes that have arrived, that are released
      for (int i = 0; i < n && ok; ++i) {
        if (i + 2 >= GA * g) {
          ok = mbar_wait_warp(afull + 8 * g, (phase >> g) & 1);
          phase ^= 1u << g;
          g += 1;
        }
        if (i % GB == 0) ok = ok && mbar_wait_warp(bfull + 8 * bs, bph);
        if (!ok) break;
        tc_fence_after();
        const uint32_t ra = da + i * (L::SLOT >> 4), rb = db + (bs * GB + i % GB) * (L::ROW >> 4);
        const bool box_done = i % GB == GB - 1 || i + 1 == n;
        if (leader) {
#pragma unroll
          for (int k = 0; k < kWKP / 16; ++k)
#pragma unroll
            for (int m = 0; m < L::NM; ++m)
              mma_bf16_lo(tmem + acc + m * L::N, ra + m * (2 * L::SLOT >> 4) + k * (CO * 2), ha, rb + k * (CI * 2), hb, idesc,
                          any | k);
          if (box_done) mma_commit(bempty + 8 * bs);
          // a box's last row is slot 0 of this window
          if (i % GA == GA - 1 && i + 1 < n) mma_commit(aempty + 8 * freed);
          if (i + 1 == n)
            for (int q = freed; q < g; ++q) mma_commit(aempty + 8 * q);
        }
        if (i % GA == GA - 1) freed += 1;
        any = 1;
        if (++rows == until && L::NACC > 1 && rows < t1 - t0) {
          acc += L::NM * L::N;
          any = 0;
          until = t1 - t0;
        }
        if (box_done && ++bs == NB) {
          bs = 0;
          bph ^= 1;
        }
      }
    }
    if (leader) mma_commit(done);
    if (!ok && leader) {
      atomicExch(&s_fail, 1);
      atomicCAS(a.err, 0, 2);
    }
  }

  // epilogue: warp w reads D rows 32 w .. 32 w + 31 of each accumulator
  __syncwarp();
  const bool ok = mbar_wait(done, 0);
  tc_fence_after();
  if (!ok) atomicCAS(a.err, 0, 3);
  const bool add = __all_sync(0xffffffffu, ok && !s_fail);
#pragma unroll
  for (int m = 0; m < L::NM; ++m) {
    const int row = 32 * warp + lane;                       // D row of MMA m
    const int sl = CO == 32 ? warp : 2 * m + (row >> 6);    // A slot: vertical tap 2 - sl
    const int co = co0 + (CO == 32 ? lane : (row & 63));
    if (sl == 3) continue;                                  // warp-uniform: no tap
    const uint32_t tl = tmem + (uint32_t(32 * warp) << 16) + m * L::N;
    const bool odd = lane & 1;
#pragma unroll 1
    for (int n0 = 0; n0 < L::N; n0 += 16) {
      uint32_t v[16];
      tmem_ld16(tl + n0, v);
      if (L::NACC > 1 && nacc > 1) {
        uint32_t u[16];
        tmem_ld16(tl + L::NM * L::N + n0, u);
#pragma unroll
        for (int q = 0; q < 16; ++q) v[q] = __float_as_uint(__uint_as_float(v[q]) + __uint_as_float(u[q]));
      }
      const int dx = n0 / CI, ci = ci0 + (n0 - dx * CI);
      // L2 adds 32-byte sectors: the lanes of a pair take the two halves of one row's
      // sector, then of the other's (64 -> 64: 48.0 -> 43.5 us; a row a lane took 11.7)
      float *dst = a.dw + (size_t(co & ~1) * 9 + 3 * (2 - sl) + dx) * a.cin + ci + (odd ? 4 : 0);
#pragma unroll
      for (int q = 0; q < 16; q += 8) {
        float x[4], y[4];   // of the even lane's row, of the odd lane's
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          const float lo = __uint_as_float(v[q + k]), hi = __uint_as_float(v[q + 4 + k]);
          const float got = __shfl_xor_sync(0xffffffffu, odd ? lo : hi, 1);
          x[k] = odd ? got : lo;
          y[k] = odd ? hi : got;
        }
        if (add) {
          atomicAdd(reinterpret_cast<float4 *>(dst + q), make_float4(x[0], x[1], x[2], x[3]));
          atomicAdd(reinterpret_cast<float4 *>(dst + q + 9 * size_t(a.cin)), make_float4(y[0], y[1], y[2], y[3]));
        }
      }
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 0) tmem_dealloc(tmem, L::NCOLS);
}

// The weight gradient of the 2x2 stride-2 transposed convolution,
// dW[a][c][ci][co] = sum over input pixels p of in[p][ci] g[child (a, c) of p][co],
// g its output gradient, K blocks as above.  The four slots of A are the four
// children's tiles of g (5-D boxes {CO, 1, 64, 1, 1} of g viewed as {channels, c,
// x, a, rows}), B is the input row without a shift (N = CI), and D row (t, co),
// column ci holds dW[t][ci][co]; the epilogue adds it with scalar atomics,
// consecutive lanes on consecutive co.
template <int CO, int CI, int STAGES>
struct WLayout {
  static constexpr uint32_t SLOT = kWKP * CO * 2;
  static constexpr uint32_t A_BYTES = 4 * SLOT;
  static constexpr uint32_t B_TX = kWKPB * CI * 2;
  static constexpr uint32_t B_BYTES = ((B_TX + 1023) / 1024) * 1024;
  static constexpr uint32_t STAGE = A_BYTES + B_BYTES;
  static constexpr uint32_t BAR_OFF = STAGES * STAGE;
  static constexpr uint32_t TAIL = WRing<CO, CI>::TAIL;   // as there
  static constexpr uint32_t BYTES = BAR_OFF + (2 * STAGES + 1) * 8 + 16 + TAIL + 1024;
  static constexpr int NM = CO == 32 ? 1 : 2;   // MMAs along M per 16 pixels
  static constexpr int N = CI;
  static constexpr uint32_t NCOLS = tmem_cols(NM * N);
};

struct WArgs {
  float *dw;           // [4][cin][cout]
  int cin, cout, a_off, H, nwc;
  long long nkb;       // K blocks: B H rows x nwc pixel chunks
  long long per_cta;   // K blocks per CTA along the grid's first index
  int *err;
};

template <int CO, int CI, int STAGES>
__global__ void __launch_bounds__(kThreads, 1)
    k_upwgrad_tc(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB, WArgs a) {
  using L = WLayout<CO, CI, STAGES>;
  extern __shared__ uint8_t smem_raw[];
  uint8_t *smem = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  const uint32_t s0 = saddr(smem);
  const uint32_t bar0 = s0 + L::BAR_OFF;   // full[s] = bar0 + 8 s, empty[s] = bar0 + 8 (STAGES + s)
  const uint32_t done = bar0 + 16 * STAGES;
  uint32_t *slot = reinterpret_cast<uint32_t *>(smem + L::BAR_OFF + (2 * STAGES + 1) * 8);
  __shared__ int s_fail;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int ncib = a.cin / CI;
  const int co0 = int(blockIdx.y) / ncib * CO, ci0 = int(blockIdx.y) % ncib * CI;
  const long long k0 = blockIdx.x * a.per_cta;
  const long long k1 = k0 + a.per_cta < a.nkb ? k0 + a.per_cta : a.nkb;
  const int nk = int(k1 - k0);   // at least 1 (the host sizes the grid so)

  if (tid == 0) {
    for (int s = 0; s < STAGES; ++s) {
      mbar_init(bar0 + 8 * s, 1);
      mbar_init(bar0 + 8 * (STAGES + s), 1);
    }
    mbar_init(done, 1);
    s_fail = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 0) tmem_alloc(saddr(slot), L::NCOLS);
  pdl_wait();
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  pdl_release();
  const uint32_t tmem = *slot;

  if (tid == 0) {
    for (int kb = 0; kb < nk; ++kb) {
      const int s = kb % STAGES;
      const uint32_t ph = (kb / STAGES) & 1;
      if (kb >= STAGES && !mbar_wait(bar0 + 8 * (STAGES + s), ph ^ 1)) {
        atomicExch(&s_fail, 1);
        atomicCAS(a.err, 0, 1);
        break;
      }
      if (s_fail) break;
      const long long g = k0 + kb;
      const long long r = g / a.nwc;              // b H + hq
      const int w0 = int(g - r * a.nwc) * kWKP;
      const int b = int(r / a.H), hq = int(r - (long long)b * a.H);
      const uint32_t st = s0 + s * L::STAGE;
      mbar_expect_tx(bar0 + 8 * s, 4 * L::SLOT + L::B_TX);
      for (int t = 0; t < 4; ++t)
        tma_load_5d(st + t * L::SLOT, &tmA, a.a_off + co0, t & 1, w0, t >> 1, int(r), bar0 + 8 * s);
      tma_load_4d(st + L::A_BYTES, &tmB, ci0, w0 - 8, hq, b, bar0 + 8 * s);
    }
  } else if (tid == 32) {
    constexpr uint32_t idesc = instr_desc_mn<L::N>();
    for (int kb = 0; kb < nk; ++kb) {
      const int s = kb % STAGES;
      const uint32_t ph = (kb / STAGES) & 1;
      if (!mbar_wait(bar0 + 8 * s, ph)) {
        atomicExch(&s_fail, 1);
        atomicCAS(a.err, 0, 2);
        break;
      }
      tc_fence_after();
      const uint32_t st = s0 + s * L::STAGE;
#pragma unroll
      for (int k = 0; k < kWKP / 16; ++k) {
        // input rows 8 + 16 k ..: pixel w0 + 16 k on
        const uint64_t db = mn_desc<CI>(st + L::A_BYTES + (8 + 16 * k) * (CI * 2), CI * 2);
#pragma unroll
        for (int m = 0; m < L::NM; ++m) {
          const uint64_t da = mn_desc<CO>(st + 2 * m * L::SLOT + 16 * k * (CO * 2), L::SLOT);
          mma_bf16(tmem + m * L::N, da, db, idesc, (kb | k) != 0 ? 1u : 0u);
        }
      }
      mma_commit(bar0 + 8 * (STAGES + s));
    }
    mma_commit(done);
  }

  // epilogue: warp w reads D rows 32 w .. 32 w + 31 of each accumulator
  __syncwarp();
  const bool ok = mbar_wait(done, 0);
  tc_fence_after();
  if (!ok) atomicCAS(a.err, 0, 3);
#pragma unroll
  for (int m = 0; m < L::NM; ++m) {
    const int row = 32 * warp + lane;                       // D row of MMA m
    const int sl = CO == 32 ? warp : 2 * m + (row >> 6);    // A slot: the child
    const int co = co0 + (CO == 32 ? lane : (row & 63));
    const uint32_t tl = tmem + (uint32_t(32 * warp) << 16) + m * L::N;
#pragma unroll 1
    for (int n0 = 0; n0 < L::N; n0 += 16) {
      uint32_t v[16];
      tmem_ld16(tl + n0, v);
      // consecutive lanes: consecutive co of one (t, ci) row of dW
      if (ok && !s_fail) {
        float *dst = a.dw + (size_t(sl) * a.cin + ci0 + n0) * a.cout + co;
#pragma unroll
        for (int q = 0; q < 16; ++q) atomicAdd(dst + size_t(q) * a.cout, __uint_as_float(v[q]));
      }
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 0) tmem_dealloc(tmem, L::NCOLS);
}

// ---------------------------------------------------------------- host side
PFN_cuTensorMapEncodeTiled_v12000 encode_fn() {
  static PFN_cuTensorMapEncodeTiled_v12000 fn = nullptr;
  static std::once_flag once;
  std::call_once(once, [] {
    void *p = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) ==
            cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      fn = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(p);
  });
  return fn;
}

// whether 16 channels of the output start on a 32-byte boundary wherever 16 of them divide the channel
int wide_stores(const ConvTC &c) {
  return c.out_cs % 16 == 0 && c.out_off % 16 == 0 && (reinterpret_cast<uintptr_t>(c.out) & 31) == 0;
}

CUtensorMapSwizzle swizzle_of(int kb) {
  return kb == 64 ? CU_TENSOR_MAP_SWIZZLE_128B : (kb == 32 ? CU_TENSOR_MAP_SWIZZLE_64B : CU_TENSOR_MAP_SWIZZLE_32B);
}

// Launch shape, from timings of the network's layers at 1032 x 512 (the
// results do not depend on it, bit for bit):
//  * column blocks: a layer with fewer pixel tiles than SMs splits its N
//    columns into blocks of N / 2, N / 4 (no narrower than 64), one per CTA
//    row of the grid (N 256 over 65 tiles: 22.7 us -> 18.6 us as 4 x 64);
//  * ring depth: the deepest ring (4, 3 or 2 stages) whose CTAs all fit on
//    the SMs at once; when no depth gives one wave, the depth that leaves
//    the most CTAs per SM, because more resident CTAs hide the TMA round
//    trips better than a deeper ring (N 32, KB 64: 51 us with 2 stages, 74 us
//    with 4; N 128, KB 64 over 258 tiles: 12.4 us with 3, 16.6 us with 4).
// The depth is chosen at run time for KB = 64; KB = 16 and 32 (the wide
// top level only) take one tabled depth.
constexpr uint32_t kSmemPerSm = 233472;   // shared memory of an SM for CTAs
constexpr uint32_t kSmemPerCta = 1024;    // reserved by the system per CTA

template <int N, int KB>
constexpr int stages_of() {
  return KB == 16 ? 4 : (KB == 32 ? 3 : 2);
}

// resident CTAs per SM of an instantiation: shared memory, TMEM columns, threads
template <int N, int KB, int STAGES>
constexpr int occupancy_of() {
  constexpr int by_smem = int(kSmemPerSm / (Layout<N, KB, STAGES>::BYTES + kSmemPerCta));
  constexpr int by_tmem = int(512 / Layout<N, KB, STAGES>::NCOLS);
  constexpr int by_threads = 2048 / kThreads;
  return by_smem < by_tmem ? (by_smem < by_threads ? by_smem : by_threads)
                           : (by_tmem < by_threads ? by_tmem : by_threads);
}

// the dynamic shared memory size of one instantiation (set once per process,
// before any stream capture)
template <int N, int KB, int STAGES, bool UP, bool HALO = false>
cudaError_t prepare_nks() {
  static cudaError_t e = cudaFuncSetAttribute(k_conv3x3_tc<N, KB, STAGES, UP, HALO>,
                                              cudaFuncAttributeMaxDynamicSharedMemorySize,
                                              int(Layout<N, KB, STAGES, HALO>::BYTES));
  return e;
}

template <int N, int KB, bool UP>
cudaError_t prepare_nk() {
  cudaError_t e = cudaSuccess;
  if constexpr (!UP && N <= 64) e = prepare_nks<N, KB, 2, false, true>();
  if constexpr (KB != 64) {
    const cudaError_t f = prepare_nks<N, KB, stages_of<N, KB>(), UP>();
    return e == cudaSuccess ? f : e;
  } else {
    for (cudaError_t f : {prepare_nks<N, KB, 2, UP>(), prepare_nks<N, KB, 3, UP>(), prepare_nks<N, KB, 4, UP>()})
      if (e == cudaSuccess) e = f;
    return e;
  }
}

// One launch: grid (pixel tiles, column blocks of N of the c.cout columns)
template <int N, int KB, int STAGES, bool UP, bool HALO = false>
cudaError_t launch_nks(const ConvTC &c, cudaStream_t s, int nblk) {
  auto fn = encode_fn();
  if (!fn) return cudaErrorNotSupported;
  CUtensorMap ta, tb;
  // input: {channels (the buffer's channel stride), W, H, B}; box {KB, BW, BH, 1}
  const cuuint64_t adim[4] = {cuuint64_t(c.in_cs), cuuint64_t(c.W), cuuint64_t(c.H), cuuint64_t(c.B)};
  const cuuint64_t astr[3] = {cuuint64_t(c.in_cs) * 2, cuuint64_t(c.in_cs) * 2 * c.W,
                              cuuint64_t(c.in_cs) * 2 * c.W * c.H};
  const int BW = c.W >= kM ? kM : (1 << (31 - __builtin_clz(unsigned(c.W))));
  const int BH = kM / BW;
  if (HALO && BW != kM) return cudaErrorInvalidValue;
  // the halo box is one image row of the tile and one pixel on either side
  const cuuint32_t abox[4] = {cuuint32_t(KB), cuuint32_t(HALO ? kHaloPix : BW), cuuint32_t(HALO ? 1 : BH), 1};
  const cuuint32_t one[4] = {1, 1, 1, 1};
  if (fn(&ta, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, const_cast<bf16 *>(c.in), adim, astr, abox, one,
         CU_TENSOR_MAP_INTERLEAVE_NONE, swizzle_of(KB), CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
         CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
    return cudaErrorInvalidValue;
  // weights [cout][9][cin]: {9 cin, cout}, or of the transposed convolution
  // [4 up_cout][cin]: {cin, 4 up_cout}; box {KB, N}
  const int taps = UP ? 1 : 9;
  const cuuint64_t bdim[2] = {cuuint64_t(taps) * c.cin, cuuint64_t(UP ? 4 * c.up_cout : c.cout)};
  const cuuint64_t bstr[1] = {cuuint64_t(taps) * c.cin * 2};
  const cuuint32_t bbox[2] = {cuuint32_t(KB), cuuint32_t(N)};
  if (fn(&tb, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<bf16 *>(c.w), bdim, bstr, bbox, one,
         CU_TENSOR_MAP_INTERLEAVE_NONE, swizzle_of(KB), CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
         CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
    return cudaErrorInvalidValue;
  TCArgs a;
  a.out = c.out;
  a.out_cs = c.out_cs;
  a.out_off = c.out_off;
  a.bias = c.bias;
  a.relu = c.relu;
  a.B = c.B;
  a.H = c.H;
  a.W = c.W;
  a.cin = c.cin;
  a.in_off = c.in_off;
  a.BW = BW;
  a.BH = BH;
  a.tiles_w = (c.W + BW - 1) / BW;
  a.tiles_h = (c.H + BH - 1) / BH;
  a.n_base = c.n_base;
  a.up_cout = c.up_cout;
  a.wide = wide_stores(c);
  a.err = c.err;
  auto k = k_conv3x3_tc<N, KB, STAGES, UP, HALO>;
  const cudaError_t e = prepare_nks<N, KB, STAGES, UP, HALO>();
  if (e != cudaSuccess) return e;
  const long long tiles = (long long)a.tiles_w * a.tiles_h * c.B;
  return launch(k, dim3(unsigned(tiles), unsigned(nblk)), kThreads, Layout<N, KB, STAGES, HALO>::BYTES, s, ta, tb, a);
}

// ---- the persistent row kernel (k_conv_rows)
template <int N, int KB, int KC, bool TAPS, int EPI = kPlain>
cudaError_t prepare_rows() {
  static cudaError_t e =
      cudaFuncSetAttribute(k_conv_rows<N, KB, KC, TAPS, EPI>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                           int(RowCfg<N, KB, KC>::BYTES));
  return e;
}

template <int N, int KB, int KC, bool TAPS, int EPI = kPlain>
cudaError_t launch_rows(const ConvTC &c, cudaStream_t s, int sms) {
  using R = RowCfg<N, KB, KC>;
  auto fn = encode_fn();
  if (!fn) return cudaErrorNotSupported;
  const cudaError_t attr = prepare_rows<N, KB, KC, TAPS, EPI>();
  if (attr != cudaSuccess) return attr;
  CUtensorMap ta, tb;
  const cuuint32_t one[4] = {1, 1, 1, 1};
  const cuuint64_t adim[4] = {cuuint64_t(c.in_cs), cuuint64_t(c.W), cuuint64_t(c.H), cuuint64_t(c.B)};
  const cuuint64_t astr[3] = {cuuint64_t(c.in_cs) * 2, cuuint64_t(c.in_cs) * 2 * c.W,
                              cuuint64_t(c.in_cs) * 2 * c.W * c.H};
  const cuuint32_t abox[4] = {cuuint32_t(KB), cuuint32_t(kHaloPix), 1, 1};
  if (fn(&ta, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, const_cast<bf16 *>(c.in), adim, astr, abox, one,
         CU_TENSOR_MAP_INTERLEAVE_NONE, swizzle_of(KB), CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
         CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
    return cudaErrorInvalidValue;
  const cuuint64_t bdim[2] = {cuuint64_t(9) * c.cin, cuuint64_t(c.cout)};
  const cuuint64_t bstr[1] = {cuuint64_t(9) * c.cin * 2};
  const cuuint32_t bbox[2] = {cuuint32_t(KB), cuuint32_t(N)};
  if (fn(&tb, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<bf16 *>(c.w), bdim, bstr, bbox, one,
         CU_TENSOR_MAP_INTERLEAVE_NONE, swizzle_of(KB), CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
         CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
    return cudaErrorInvalidValue;
  RowArgs a;
  a.out = c.out;
  a.out_cs = c.out_cs;
  a.out_off = c.out_off;
  a.bias = c.bias;
  a.relu = c.relu;
  a.H = c.H;
  a.W = c.W;
  a.in_off = c.in_off;
  a.cin = c.cin;
  a.col_blocks = (c.W + kM - 1) / kM;
  a.tiles = c.B * a.col_blocks * c.H;
  a.wide = wide_stores(c);
  a.err = c.err;
  a.pool = c.pool;
  a.pool_cs = c.cout;
  a.y = c.y;
  a.y_cs = c.y_cs;
  a.y_off = c.y_off;
  a.db = c.db;
  a.db_n = c.db_n;
  const int nblk = c.cout / N;
  const int ctas = std::max(1, std::min(EPI == kPool ? a.tiles / 2 : a.tiles, sms * R::CPS / nblk));
  return launch(k_conv_rows<N, KB, KC, TAPS, EPI>, dim3(unsigned(ctas), unsigned(nblk)), kRowThreads, R::BYTES, s, ta, tb,
                a);
}

template <int N, int KB, bool UP>
cudaError_t launch_nk(const ConvTC &c, cudaStream_t s, int nblk, long long ctas, int sms) {
  // the halo loads for the 3x3 convolutions of up to 64 columns on images at
  // least one tile wide (32 -> 32 at 1032 x 512: 42.5 -> 34.9 us; 128 -> 64 at
  // 516 x 256: 34.3 -> 31.1 us); with 128 columns it was slower
  if constexpr (!UP && N <= 64)
    if (c.W >= kM) return launch_nks<N, KB, 2, false, true>(c, s, nblk);
  if constexpr (KB != 64) {
    return launch_nks<N, KB, stages_of<N, KB>(), UP>(c, s, nblk);
  } else {
    if (ctas <= (long long)sms * occupancy_of<N, KB, 4>()) return launch_nks<N, KB, 4, UP>(c, s, nblk);
    if (ctas <= (long long)sms * occupancy_of<N, KB, 3>()) return launch_nks<N, KB, 3, UP>(c, s, nblk);
    return launch_nks<N, KB, 2, UP>(c, s, nblk);
  }
}

template <int N, bool UP>
cudaError_t launch_n(const ConvTC &c, cudaStream_t s, int nblk, long long ctas, int sms) {
  if (c.cin % 64 == 0) return launch_nk<N, 64, UP>(c, s, nblk, ctas, sms);
  if (c.cin % 32 == 0) return launch_nk<N, 32, UP>(c, s, nblk, ctas, sms);
  return launch_nk<N, 16, UP>(c, s, nblk, ctas, sms);
}

constexpr int kUpbStages = 3;
template <int N, int KB>
cudaError_t prepare_upb() {
  static cudaError_t e = cudaFuncSetAttribute(k_conv3x3_tc<N, KB, kUpbStages, false, false, true>,
                                              cudaFuncAttributeMaxDynamicSharedMemorySize,
                                              int(Layout<N, KB, kUpbStages>::BYTES));
  return e;
}

template <int N>
cudaError_t prepare_n() {
  cudaError_t e = cudaSuccess;
  for (cudaError_t f : {prepare_nk<N, 64, false>(), prepare_nk<N, 32, false>(), prepare_nk<N, 16, false>(),
                        prepare_nk<N, 64, true>(), prepare_nk<N, 32, true>(), prepare_nk<N, 16, true>(),
                        prepare_upb<N, 64>(), prepare_upb<N, 32>(), prepare_upb<N, 16>()})
    if (e == cudaSuccess) e = f;
  return e;
}

// Data gradient of the transposed convolution (UPB): grid (pixel tiles of
// the transposed convolution's input, column blocks of its input channels)
template <int N, int KB>
cudaError_t launch_upb(const ConvTC &c, cudaStream_t s, int nblk) {
  constexpr int STAGES = kUpbStages;
  using L = Layout<N, KB, STAGES>;
  auto fn = encode_fn();
  if (!fn) return cudaErrorNotSupported;
  const cudaError_t attr = prepare_upb<N, KB>();
  if (attr != cudaSuccess) return attr;
  CUtensorMap ta, tb;
  // the output gradient [B][2H][2W][in_cs] as {channels, c, x, a, B H}: child (a, c)
  // of input pixel (y, x) is (2y + a, 2x + c)
  const cuuint64_t e = 2;   // bytes per element
  const cuuint64_t adim[5] = {cuuint64_t(c.in_cs), 2, cuuint64_t(c.W), 2, cuuint64_t(c.B) * c.H};
  const cuuint64_t astr[4] = {cuuint64_t(c.in_cs) * e, cuuint64_t(c.in_cs) * e * 2,
                              cuuint64_t(c.in_cs) * e * 2 * c.W, cuuint64_t(c.in_cs) * e * 4 * c.W};
  const int BW = c.W >= kM ? kM : (1 << (31 - __builtin_clz(unsigned(c.W))));
  const int BH = kM / BW;
  const cuuint32_t abox[5] = {cuuint32_t(KB), 1, cuuint32_t(BW), 1, cuuint32_t(BH)};
  const cuuint32_t one[5] = {1, 1, 1, 1, 1};
  if (fn(&ta, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 5, const_cast<bf16 *>(c.in), adim, astr, abox, one,
         CU_TENSOR_MAP_INTERLEAVE_NONE, swizzle_of(KB), CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
         CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
    return cudaErrorInvalidValue;
  // weights [4 ncols][K]: {K, 4 ncols}; box {KB, N}
  const cuuint64_t bdim[2] = {cuuint64_t(c.cin), cuuint64_t(4) * c.cout};
  const cuuint64_t bstr[1] = {cuuint64_t(c.cin) * e};
  const cuuint32_t bbox[2] = {cuuint32_t(KB), cuuint32_t(N)};
  if (fn(&tb, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<bf16 *>(c.w), bdim, bstr, bbox, one,
         CU_TENSOR_MAP_INTERLEAVE_NONE, swizzle_of(KB), CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
         CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
    return cudaErrorInvalidValue;
  TCArgs a;
  a.out = c.out;
  a.out_cs = c.out_cs;
  a.out_off = c.out_off;
  a.bias = nullptr;
  a.relu = 0;
  a.B = c.B;
  a.H = c.H;
  a.W = c.W;
  a.cin = c.cin;
  a.in_off = c.in_off;
  a.BW = BW;
  a.BH = BH;
  a.tiles_w = (c.W + BW - 1) / BW;
  a.tiles_h = (c.H + BH - 1) / BH;
  a.n_base = 0;
  a.up_cout = 0;
  a.ncols = c.cout;
  a.wide = wide_stores(c);
  a.err = c.err;
  const long long tiles = (long long)a.tiles_w * a.tiles_h * c.B;
  return launch(k_conv3x3_tc<N, KB, STAGES, false, false, true>, dim3(unsigned(tiles), unsigned(nblk)), kThreads, L::BYTES,
                s, ta, tb, a);
}

template <int N>
cudaError_t launch_upb_n(const ConvTC &c, cudaStream_t s, int nblk) {
  if (c.cin % 64 == 0) return launch_upb<N, 64>(c, s, nblk);
  if (c.cin % 32 == 0) return launch_upb<N, 32>(c, s, nblk);
  return launch_upb<N, 16>(c, s, nblk);
}

constexpr int kWStages = 3;
template <int CO, int CI>
cudaError_t prepare_wgrad() {
  static cudaError_t e = cudaFuncSetAttribute(k_wgrad_rows<CO, CI>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                              int(WRing<CO, CI>::BYTES));
  return e;
}
template <int CO, int CI>
cudaError_t prepare_upwgrad() {
  static cudaError_t e = cudaFuncSetAttribute(k_upwgrad_tc<CO, CI, kWStages>,
                                              cudaFuncAttributeMaxDynamicSharedMemorySize,
                                              int(WLayout<CO, CI, kWStages>::BYTES));
  return e;
}

// CTAs of one wave over yb (co, ci) blocks, each a run of the n units (at least one)
template <class L>
long long wave_split(long long n, int sms, int yb) {
  const int res_smem = int((227u * 1024u) / L::BYTES), res_tmem = int(512u / L::NCOLS);
  const int res = res_smem < res_tmem ? (res_smem > 0 ? res_smem : 1) : res_tmem;
  return std::max(1LL, std::min(n, (long long)sms * res / yb));
}

template <int CO, int CI>
cudaError_t launch_wgrad(const WgradTC &g, cudaStream_t s, int sms) {
  using L = WRing<CO, CI>;
  auto fn = encode_fn();
  if (!fn) return cudaErrorNotSupported;
  const cudaError_t attr = prepare_wgrad<CO, CI>();
  if (attr != cudaSuccess) return attr;
  const cuuint64_t e = 2;
  const cuuint32_t one[4] = {1, 1, 1, 1};
  CUtensorMap ta, tb;
  // the gradient [B][H][W][cout] as {cout, W, H, B}, boxes {CO, 64 pixels, GA rows}
  const cuuint64_t adim[4] = {cuuint64_t(g.cout), cuuint64_t(g.W), cuuint64_t(g.H), cuuint64_t(g.B)};
  const cuuint64_t astr[3] = {cuuint64_t(g.cout) * e, cuuint64_t(g.cout) * e * g.W, cuuint64_t(g.cout) * e * g.W * g.H};
  const cuuint32_t abox[4] = {cuuint32_t(CO), cuuint32_t(kWKP), L::GA, 1};
  if (fn(&ta, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, const_cast<bf16 *>(g.dpre), adim, astr, abox, one,
         CU_TENSOR_MAP_INTERLEAVE_NONE, swizzle_of(CO), CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
         CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
    return cudaErrorInvalidValue;
  // the input [B][H][W][in_cs] as {in_cs, W, H, B}, boxes {CI, 80 pixels, GB rows}
  const cuuint64_t bdim[4] = {cuuint64_t(g.in_cs), cuuint64_t(g.W), cuuint64_t(g.H), cuuint64_t(g.B)};
  const cuuint64_t bstr[3] = {cuuint64_t(g.in_cs) * e, cuuint64_t(g.in_cs) * e * g.W,
                              cuuint64_t(g.in_cs) * e * g.W * g.H};
  const cuuint32_t bbox[4] = {cuuint32_t(CI), cuuint32_t(kWKPB), L::GB, 1};
  if (fn(&tb, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, const_cast<bf16 *>(g.in), bdim, bstr, bbox, one,
         CU_TENSOR_MAP_INTERLEAVE_NONE, swizzle_of(CI), CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
         CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
    return cudaErrorInvalidValue;
  WRowArgs a;
  a.dw = g.dw;
  a.cin = g.cin;
  a.cout = g.cout;
  a.in_off = g.in_off;
  a.H = g.H;
  a.nwc = (g.W + kWKP - 1) / kWKP;
  a.rows = (long long)g.B * g.H * a.nwc;
  a.err = g.err;
  // one wave: the CTAs that fit on the SMs at once (shared memory, TMEM
  // columns), shared out over the (co, ci) blocks; two waves where one does not
  // come out even, so that no accumulator takes more than its share (256 -> 256 at
  // 4 x 129 x 64, relative error: 1.55e-6 with 9 CTAs a block, 1.41e-6 with 10, in two
  // waves of 19 6.5e-7; 40 and 49 us)
  const int yb = (g.cout / CO) * (g.cin / CI);
  const long long wave = wave_split<L>(1LL << 40, sms, 1);   // CTAs resident at once
  const long long splits = wave_split<L>(a.rows, wave % yb && yb < wave ? 2 * sms : sms, yb);
  return launch(k_wgrad_rows<CO, CI>, dim3(unsigned(splits), unsigned(yb)), kThreads, L::BYTES, s, ta, tb, a);
}

template <int CO>
cudaError_t launch_upw(const UpWgradTC &g, cudaStream_t s, int sms) {
  constexpr int CI = 64;
  using L = WLayout<CO, CI, kWStages>;
  auto fn = encode_fn();
  if (!fn) return cudaErrorNotSupported;
  const cudaError_t attr = prepare_upwgrad<CO, CI>();
  if (attr != cudaSuccess) return attr;
  const cuuint64_t e = 2;
  const cuuint32_t one[5] = {1, 1, 1, 1, 1};
  CUtensorMap ta, tb;
  // the output gradient [B][2H][2W][g_cs] as {g_cs, c, x, a, B H}: child (a, c)
  // of input pixel (y, x) is (2y + a, 2x + c); boxes {CO, 1, 64, 1, 1}
  const cuuint64_t adim[5] = {cuuint64_t(g.g_cs), 2, cuuint64_t(g.W), 2, cuuint64_t(g.B) * g.H};
  const cuuint64_t astr[4] = {cuuint64_t(g.g_cs) * e, cuuint64_t(g.g_cs) * e * 2, cuuint64_t(g.g_cs) * e * 2 * g.W,
                              cuuint64_t(g.g_cs) * e * 4 * g.W};
  const cuuint32_t abox[5] = {cuuint32_t(CO), 1, cuuint32_t(kWKP), 1, 1};
  if (fn(&ta, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 5, const_cast<bf16 *>(g.g), adim, astr, abox, one,
         CU_TENSOR_MAP_INTERLEAVE_NONE, swizzle_of(CO), CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
         CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
    return cudaErrorInvalidValue;
  // the input [B][H][W][cin] as {cin, W, H, B}, boxes {64, 80 pixels} from 8 before
  const cuuint64_t bdim[4] = {cuuint64_t(g.cin), cuuint64_t(g.W), cuuint64_t(g.H), cuuint64_t(g.B)};
  const cuuint64_t bstr[3] = {cuuint64_t(g.cin) * e, cuuint64_t(g.cin) * e * g.W, cuuint64_t(g.cin) * e * g.W * g.H};
  const cuuint32_t bbox[4] = {cuuint32_t(CI), cuuint32_t(kWKPB), 1, 1};
  if (fn(&tb, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, const_cast<bf16 *>(g.in), bdim, bstr, bbox, one,
         CU_TENSOR_MAP_INTERLEAVE_NONE, swizzle_of(CI), CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
         CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
    return cudaErrorInvalidValue;
  WArgs a;
  a.dw = g.dw;
  a.cin = g.cin;
  a.cout = g.cout;
  a.a_off = g.g_off;
  a.H = g.H;
  a.nwc = (g.W + kWKP - 1) / kWKP;
  a.nkb = (long long)g.B * g.H * a.nwc;
  a.err = g.err;
  const int yb = (g.cout / CO) * (g.cin / CI);
  const long long splits = wave_split<L>(a.nkb, sms, yb);
  a.per_cta = (a.nkb + splits - 1) / splits;
  return launch(k_upwgrad_tc<CO, CI, kWStages>, dim3(unsigned((a.nkb + a.per_cta - 1) / a.per_cta), unsigned(yb)), kThreads,
                L::BYTES, s, ta, tb, a);
}

// The persistent transposed convolution (up_cout > 0: all 4 up_cout columns from
// n_base 0 on, c.cout of them) and its data gradient; cudaErrorNotSupported for
// channel counts that are no multiples of 32, or columns that 64 does not divide.
constexpr int kUpSmem = 227 * 1024 - 2048;   // beside the static shared memory
template <int N, int KB, int MODE>
cudaError_t prepare_up() {
  static cudaError_t e = cudaFuncSetAttribute(k_up_tiles<N, KB, MODE>, cudaFuncAttributeMaxDynamicSharedMemorySize, kUpSmem);
  return e;
}

template <int N, int KB, int MODE>
cudaError_t launch_up(const ConvTC &c, cudaStream_t s, int sms, const CUtensorMap &ta, UpArgs a) {
  auto fn = encode_fn();
  const cudaError_t attr = prepare_up<N, KB, MODE>();
  if (attr != cudaSuccess) return attr;
  // weights [rows][cin]: {cin, 4 up_cout} or {cin, 4 cout}; box {KB, N}
  CUtensorMap tb;
  const cuuint32_t one[2] = {1, 1};
  const cuuint64_t bdim[2] = {cuuint64_t(c.cin), cuuint64_t(4) * (MODE == kUp ? c.up_cout : c.cout)};
  const cuuint64_t bstr[1] = {cuuint64_t(c.cin) * 2};
  const cuuint32_t bbox[2] = {cuuint32_t(KB), cuuint32_t(N)};
  if (fn(&tb, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<bf16 *>(c.w), bdim, bstr, bbox, one,
         CU_TENSOR_MAP_INTERLEAVE_NONE, swizzle_of(KB), CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
         CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
    return cudaErrorInvalidValue;
  const int wbytes = a.units * N * KB * 2, unit = kM * KB * 2;
  a.stages = std::min(kUpStages, (kUpSmem - 1024 - wbytes) / unit);
  const int nblk = c.cout / N, ctas = std::max(1, std::min(a.tiles, sms / nblk));
  return launch(k_up_tiles<N, KB, MODE>, dim3(unsigned(ctas), unsigned(nblk)), kRowThreads,
                1024 + wbytes + a.stages * unit, s, ta, tb, a);
}

template <int KB, int MODE>
cudaError_t launch_up_kb(const ConvTC &c, cudaStream_t s, int sms) {
  auto fn = encode_fn();
  if (!fn) return cudaErrorNotSupported;
  UpArgs a;
  a.out = c.out;
  a.out_cs = c.out_cs;
  a.out_off = c.out_off;
  a.bias = c.bias;
  a.B = c.B;
  a.H = c.H;
  a.W = c.W;
  a.log_bw = c.W >= kM ? 7 : 31 - __builtin_clz(unsigned(c.W));
  const int bw = 1 << a.log_bw, bh = kM >> a.log_bw;
  a.tiles_w = (c.W + bw - 1) / bw;
  a.tiles_h = (c.H + bh - 1) / bh;
  const long long tiles = (long long)a.tiles_w * a.tiles_h * c.B;
  if (tiles >= (1LL << 31)) return cudaErrorNotSupported;
  a.tiles = int(tiles);
  a.in_off = c.in_off;
  a.kchunks = c.cin / KB;
  a.units = (MODE == kUp ? 1 : 4) * a.kchunks;
  a.n_base = c.n_base;
  a.up_cout = c.up_cout;
  a.ncols = MODE == kUp ? 0 : c.cout;
  a.wide = wide_stores(c);
  a.y = c.y;
  a.y_cs = c.y_cs;
  a.y_off = c.y_off;
  a.db = c.db;
  a.err = c.err;
  // Columns a CTA: the fewest column-tiles in the longest CTA's sequence (a tile
  // also costs about 32 columns' time for its pixels), wider on a tie; at least 3
  // units beside the weights.
  int best = 0;
  long long best_cost = 0;
  for (int n : {256, 128, 64}) {
    if (c.cout % n || (MODE != kUp && n == 256) || c.cout / n > sms) continue;
    if ((long long)a.units * n * KB * 2 + 3 * kM * KB * 2 + 1024 > kUpSmem) continue;
    const long long per = sms / (c.cout / n), cost = (tiles + per - 1) / per * (n + 32);
    if (!best || cost < best_cost) {
      best = n;
      best_cost = cost;
    }
  }
  if (!best) return cudaErrorNotSupported;
  // Four column blocks of 64 each load all of the pixels; with few units beside the
  // weights, on many tiles, that costs more than one pass of the tile kernel (a call
  // with 256 channels from 256 at 1032 tiles 231 us against 223, at 774 203 against 210;
  // from 320 at 400 tiles 178 against 174, at 1032 279 against 243; from 192 never).
  if (MODE == kUpBack && c.cout / best >= 4 && tiles * (a.units * KB / 64 - 12) > 20LL * sms)
    return cudaErrorNotSupported;
  CUtensorMap ta;
  const cuuint32_t one[5] = {1, 1, 1, 1, 1};
  const cuuint64_t e = 2, cs = c.in_cs;   // bytes per element
  CUresult r;
  if (MODE == kUp) {
    // input {channels, W, H, B}; box {KB, bw, bh, 1}
    const cuuint64_t dim[4] = {cs, cuuint64_t(c.W), cuuint64_t(c.H), cuuint64_t(c.B)};
    const cuuint64_t str[3] = {cs * e, cs * e * c.W, cs * e * c.W * c.H};
    const cuuint32_t box[4] = {cuuint32_t(KB), cuuint32_t(bw), cuuint32_t(bh), 1};
    r = fn(&ta, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, const_cast<bf16 *>(c.in), dim, str, box, one,
           CU_TENSOR_MAP_INTERLEAVE_NONE, swizzle_of(KB), CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
           CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  } else {
    // the output gradient [B][2H][2W][in_cs] as {channels, c, x, a, B H}
    const cuuint64_t dim[5] = {cs, 2, cuuint64_t(c.W), 2, cuuint64_t(c.B) * c.H};
    const cuuint64_t str[4] = {cs * e, cs * e * 2, cs * e * 2 * c.W, cs * e * 4 * c.W};
    const cuuint32_t box[5] = {cuuint32_t(KB), 1, cuuint32_t(bw), 1, cuuint32_t(bh)};
    r = fn(&ta, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 5, const_cast<bf16 *>(c.in), dim, str, box, one,
           CU_TENSOR_MAP_INTERLEAVE_NONE, swizzle_of(KB), CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
           CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  }
  if (r != CUDA_SUCCESS) return cudaErrorInvalidValue;
  if (best == 64) return launch_up<64, KB, MODE>(c, s, sms, ta, a);
  if (MODE != kUp || best == 128) return launch_up<128, KB, MODE>(c, s, sms, ta, a);
  if constexpr (MODE == kUp) return launch_up<256, KB, MODE>(c, s, sms, ta, a);
  return cudaErrorNotSupported;
}

template <int KB>
cudaError_t prepare_up_kb() {
  for (cudaError_t e : {prepare_up<64, KB, kUp>(), prepare_up<128, KB, kUp>(), prepare_up<256, KB, kUp>(),
                        prepare_up<64, KB, kUpBack>(), prepare_up<128, KB, kUpBack>(), prepare_up<64, KB, kUpBackY>(),
                        prepare_up<128, KB, kUpBackY>()})
    if (e != cudaSuccess) return e;
  return cudaSuccess;
}

int sm_count() {
  int dev = 0, sms = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
    return 0;
  return sms;
}

}  // namespace tc

cudaError_t conv3x3_tc_prepare() {
  cudaError_t e = tc::prepare_n<32>();
  if (e == cudaSuccess) e = tc::prepare_up_kb<32>();
  if (e == cudaSuccess) e = tc::prepare_up_kb<64>();
  if (e == cudaSuccess) e = tc::prepare_n<64>();
  if (e == cudaSuccess) e = tc::prepare_n<128>();
  if (e == cudaSuccess) e = tc::prepare_n<256>();
  for (cudaError_t f : {tc::prepare_wgrad<32, 16>(), tc::prepare_wgrad<32, 32>(), tc::prepare_wgrad<32, 64>(),
                        tc::prepare_wgrad<64, 16>(), tc::prepare_wgrad<64, 32>(), tc::prepare_wgrad<64, 64>(),
                        tc::prepare_upwgrad<32, 64>(), tc::prepare_upwgrad<64, 64>(),
                        tc::prepare_rows<32, 32, 1, false>(), tc::prepare_rows<32, 64, 1, false>(),
                        tc::prepare_rows<64, 32, 1, false>(), tc::prepare_rows<64, 64, 1, false>(),
                        tc::prepare_rows<64, 64, 2, false>(), tc::prepare_rows<64, 64, 1, true>(),
                        tc::prepare_rows<64, 64, 2, true>(), tc::prepare_rows<32, 64, 4, false>(),
                        tc::prepare_rows<32, 64, 4, true>(),
                        tc::prepare_rows<32, 32, 1, false, tc::kPool>(), tc::prepare_rows<64, 64, 1, false, tc::kPool>(),
                        tc::prepare_rows<64, 64, 2, false, tc::kPool>(), tc::prepare_rows<64, 64, 2, true, tc::kPool>(),
                        tc::prepare_rows<64, 32, 1, false, tc::kSum>(), tc::prepare_rows<64, 64, 1, false, tc::kSum>(),
                        tc::prepare_rows<64, 64, 2, false, tc::kSum>(), tc::prepare_rows<64, 64, 1, true, tc::kSum>(),
                        tc::prepare_rows<64, 64, 2, true, tc::kSum>(),
                        tc::prepare_rows<32, 32, 1, false, tc::kBack>(), tc::prepare_rows<64, 64, 1, false, tc::kBack>(),
                        tc::prepare_rows<64, 64, 2, false, tc::kBack>(), tc::prepare_rows<64, 64, 2, true, tc::kBack>()})
    if (e == cudaSuccess) e = f;
  return e;
}

bool conv3x3_tc_supported(int cin, int cout, int in_cs, int in_off, int out_cs, int out_off, int W) {
  return cin >= 16 && cin % 16 == 0 && (cout == 32 || cout == 64 || cout == 128 || cout == 256) &&
         in_cs % 8 == 0 && in_off % 8 == 0 && out_cs % 8 == 0 && out_off % 8 == 0 && W >= 8 &&
         tc::encode_fn() != nullptr;
}

cudaError_t conv3x3_tc(const ConvTC &c, cudaStream_t s) {
  if (!conv3x3_tc_supported(c.cin, c.cout, c.in_cs, c.in_off, c.out_cs, c.out_off, c.W))
    return cudaErrorNotSupported;
  // the transposed convolution's GEMM columns come in launches of at most 256
  if (c.up_cout && (c.up_cout % 16 || c.n_base % c.up_cout || c.n_base + c.cout > 4 * c.up_cout))
    return cudaErrorNotSupported;
  const int sms = tc::sm_count();
  if (sms < 1) return cudaErrorInvalidValue;
  const int BW = c.W >= tc::kM ? tc::kM : (1 << (31 - __builtin_clz(unsigned(c.W))));
  const long long tiles = (long long)((c.W + BW - 1) / BW) * ((c.H + tc::kM / BW - 1) / (tc::kM / BW)) * c.B;
  // column blocks while the pixel tiles alone leave SMs idle
  int n = c.cout, nblk = 1;
  while (n > 64 && tiles * nblk < sms) {
    n >>= 1;
    nblk <<= 1;
  }
  const long long ctas = tiles * nblk;
  const bool up = c.up_cout != 0;
  // the persistent row kernel (whole 128-pixel rows; input channels whose
  // weights fit beside a row), with the K order of the kernel it replaces: that
  // one takes (dy, chunk, dx) up to 64 columns a CTA and (dy, dx, chunk) above
  const bool rows = !up && c.W >= tc::kM && (long long)c.B * ((c.W + tc::kM - 1) / tc::kM) * c.H < (1LL << 31);
  // its other epilogues: as many channels out as in, up to 128 (the blocks' second layers)
  if (c.pool || c.y) {
    if (!rows || c.cin != c.cout || (c.pool && (c.y || c.H % 2 || c.W % 2)) ||
        (c.y && (c.y_cs % 8 || c.y_off % 8 || !c.db)))
      return cudaErrorNotSupported;
    if (n == 32 && c.cin == 32)
      return c.pool ? tc::launch_rows<32, 32, 1, false, tc::kPool>(c, s, sms)
                    : tc::launch_rows<32, 32, 1, false, tc::kBack>(c, s, sms);
    if (n == 64 && c.cin == 64)
      return c.pool ? tc::launch_rows<64, 64, 1, false, tc::kPool>(c, s, sms)
                    : tc::launch_rows<64, 64, 1, false, tc::kBack>(c, s, sms);
    if (n == 64 && c.cin == 128)
      return c.pool ? tc::launch_rows<64, 64, 2, false, tc::kPool>(c, s, sms)
                    : tc::launch_rows<64, 64, 2, false, tc::kBack>(c, s, sms);
    if (n == 128 && c.cin == 128)
      return c.pool ? tc::launch_rows<64, 64, 2, true, tc::kPool>(c, s, sms)
                    : tc::launch_rows<64, 64, 2, true, tc::kBack>(c, s, sms);
    return cudaErrorNotSupported;
  }
  if (c.db) {   // the concatenations' gradients: twice as many channels out as in
    if (!rows || c.cout != 2 * c.cin || c.db_n != c.cin) return cudaErrorNotSupported;
    if (n == 64 && c.cin == 32) return tc::launch_rows<64, 32, 1, false, tc::kSum>(c, s, sms);
    if (n == 64 && c.cin == 64) return tc::launch_rows<64, 64, 1, false, tc::kSum>(c, s, sms);
    if (n == 64 && c.cin == 128) return tc::launch_rows<64, 64, 2, false, tc::kSum>(c, s, sms);
    if (n >= 128 && c.cin == 64) return tc::launch_rows<64, 64, 1, true, tc::kSum>(c, s, sms);
    if (n >= 128 && c.cin == 128) return tc::launch_rows<64, 64, 2, true, tc::kSum>(c, s, sms);
    return cudaErrorNotSupported;
  }
  if (rows) {
    if (n == 32 && c.cin == 32) return tc::launch_rows<32, 32, 1, false>(c, s, sms);
    if (n == 32 && c.cin == 64) return tc::launch_rows<32, 64, 1, false>(c, s, sms);
    if (n == 64 && c.cin == 32) return tc::launch_rows<64, 32, 1, false>(c, s, sms);
    if (n == 64 && c.cin == 64) return tc::launch_rows<64, 64, 1, false>(c, s, sms);
    if (n == 64 && c.cin == 128) return tc::launch_rows<64, 64, 2, false>(c, s, sms);
    if (n == 64 && c.cin == 256) return tc::launch_rows<32, 64, 4, false>(c, s, sms);
    if (n >= 128 && c.cin == 64) return tc::launch_rows<64, 64, 1, true>(c, s, sms);
    if (n >= 128 && c.cin == 128) return tc::launch_rows<64, 64, 2, true>(c, s, sms);
    if (n >= 128 && c.cin == 256) return tc::launch_rows<32, 64, 4, true>(c, s, sms);
  }
  switch (n) {
    case 32: return up ? tc::launch_n<32, true>(c, s, nblk, ctas, sms) : tc::launch_n<32, false>(c, s, nblk, ctas, sms);
    case 64: return up ? tc::launch_n<64, true>(c, s, nblk, ctas, sms) : tc::launch_n<64, false>(c, s, nblk, ctas, sms);
    case 128: return up ? tc::launch_n<128, true>(c, s, nblk, ctas, sms) : tc::launch_n<128, false>(c, s, nblk, ctas, sms);
    default: return up ? tc::launch_n<256, true>(c, s, nblk, ctas, sms) : tc::launch_n<256, false>(c, s, nblk, ctas, sms);
  }
}

cudaError_t conv_in_tc(const float2 *x, const __nv_bfloat16 *w, int wcin, const float *bias,
                       __nv_bfloat16 *out, int B, int H, int W, int relu, int *err, cudaStream_t s) {
  const int sms = tc::sm_count();
  if (sms < 1 || wcin < tc::kInCh) return cudaErrorInvalidValue;
  const long long npix = (long long)B * H * W;
  if (npix < 1 || npix >= (1LL << 31)) return cudaErrorInvalidValue;
  const long long ntiles = (npix + tc::kM - 1) / tc::kM;
  const long long grid = ntiles < 8LL * sms ? ntiles : 8LL * sms;   // 8 CTAs per SM, tiles in turn
  return launch(tc::k_conv_in_tc, dim3(unsigned(grid)), tc::kThreads, 0, s, x, w, wcin, bias, out, B, H, W, relu,
                (reinterpret_cast<uintptr_t>(out) & 31) == 0 ? 1 : 0, err);
}

cudaError_t conv_up_tc(const ConvTC &c, cudaStream_t s) {
  const int total = 4 * c.up_cout, step = std::min(total, 256);
  if (c.up_cout < 1 || c.up_cout % 16 || total % step || !conv3x3_tc_supported(c.cin, step, c.in_cs, c.in_off, c.out_cs, c.out_off, c.W))
    return cudaErrorNotSupported;
  ConvTC q = c;
  q.cout = total;
  q.n_base = 0;
  if (total % 64 == 0 && c.cin % 32 == 0) {
    const int sms = tc::sm_count();
    if (sms < 1) return cudaErrorInvalidValue;
    const cudaError_t e = c.cin % 64 == 0 ? tc::launch_up_kb<64, tc::kUp>(q, s, sms) : tc::launch_up_kb<32, tc::kUp>(q, s, sms);
    if (e != cudaErrorNotSupported) return e;
  }
  for (q.n_base = 0; q.n_base < total; q.n_base += step) {
    q.cout = step;
    const cudaError_t e = conv3x3_tc(q, s);
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

cudaError_t conv_upback_tc(const ConvTC &c, cudaStream_t s) {
  if (!conv3x3_tc_supported(c.cin, c.cout, c.in_cs, c.in_off, c.out_cs, c.out_off, c.W) ||
      (long long)c.B * c.H >= (1LL << 31))
    return cudaErrorNotSupported;
  const int sms = tc::sm_count();
  if (sms < 1) return cudaErrorInvalidValue;
  if (c.cin % 32 == 0 && c.cout % 64 == 0 && !(c.y && (c.y_cs % 8 || c.y_off % 8 || !c.db))) {
    const cudaError_t e = c.cin % 64 == 0 ? (c.y ? tc::launch_up_kb<64, tc::kUpBackY>(c, s, sms)
                                                 : tc::launch_up_kb<64, tc::kUpBack>(c, s, sms))
                                          : (c.y ? tc::launch_up_kb<32, tc::kUpBackY>(c, s, sms)
                                                 : tc::launch_up_kb<32, tc::kUpBack>(c, s, sms));
    if (e != cudaErrorNotSupported) return e;
  }
  if (c.y) return cudaErrorNotSupported;
  const int BW = c.W >= tc::kM ? tc::kM : (1 << (31 - __builtin_clz(unsigned(c.W))));
  const long long tiles = (long long)((c.W + BW - 1) / BW) * ((c.H + tc::kM / BW - 1) / (tc::kM / BW)) * c.B;
  int n = c.cout, nblk = 1;
  while (n > 64 && tiles * nblk < sms) {
    n >>= 1;
    nblk <<= 1;
  }
  switch (n) {
    case 32: return tc::launch_upb_n<32>(c, s, nblk);
    case 64: return tc::launch_upb_n<64>(c, s, nblk);
    case 128: return tc::launch_upb_n<128>(c, s, nblk);
    default: return tc::launch_upb_n<256>(c, s, nblk);
  }
}

bool conv_wgrad_tc_supported(int cin, int cout, int in_cs, int in_off, const float *dw) {
  return (cout == 32 || (cout >= 64 && cout % 64 == 0)) && (cin == 16 || cin == 32 || (cin >= 64 && cin % 64 == 0)) &&
         in_cs % 8 == 0 && in_off % 8 == 0 && in_off + cin <= in_cs && (reinterpret_cast<uintptr_t>(dw) & 15) == 0 &&
         tc::encode_fn() != nullptr;
}

cudaError_t conv_wgrad_tc(const WgradTC &g, cudaStream_t s) {
  if (!conv_wgrad_tc_supported(g.cin, g.cout, g.in_cs, g.in_off, g.dw) || g.B < 1 || g.H < 1 || g.W < 1)
    return cudaErrorNotSupported;
  const int sms = tc::sm_count();
  if (sms < 1) return cudaErrorInvalidValue;
  const int ci = g.cin >= 64 ? 64 : g.cin;
  if (g.cout == 32) {
    if (ci == 16) return tc::launch_wgrad<32, 16>(g, s, sms);
    if (ci == 32) return tc::launch_wgrad<32, 32>(g, s, sms);
    return tc::launch_wgrad<32, 64>(g, s, sms);
  }
  if (ci == 16) return tc::launch_wgrad<64, 16>(g, s, sms);
  if (ci == 32) return tc::launch_wgrad<64, 32>(g, s, sms);
  return tc::launch_wgrad<64, 64>(g, s, sms);
}

bool conv_upwgrad_tc_supported(int cin, int cout, int g_cs, int g_off) {
  return (cout == 32 || (cout >= 64 && cout % 64 == 0)) && cin >= 64 && cin % 64 == 0 && g_cs % 8 == 0 &&
         g_off % 8 == 0 && g_off + cout <= g_cs && tc::encode_fn() != nullptr;
}

cudaError_t conv_upwgrad_tc(const UpWgradTC &g, cudaStream_t s) {
  if (!conv_upwgrad_tc_supported(g.cin, g.cout, g.g_cs, g.g_off) || g.B < 1 || g.H < 1 || g.W < 1 ||
      (long long)g.B * g.H >= (1LL << 31))
    return cudaErrorNotSupported;
  const int sms = tc::sm_count();
  if (sms < 1) return cudaErrorInvalidValue;
  return g.cout == 32 ? tc::launch_upw<32>(g, s, sms) : tc::launch_upw<64>(g, s, sms);
}

}  // namespace picgb
