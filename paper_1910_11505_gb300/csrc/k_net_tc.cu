// Output layer of the learned warm start, and one training pass through it, on the 5th-generation
// tensor cores (tcgen05).
//
// Forward (tc_out_kernel): Y = H2 W3^T + b3 for a batch: H2 is B x h2 (h2 <= 64, FP32, rounded to
// BF16 here), W3 is out x h2 (the network's BF16 copy), Y is B x out.  One CTA of 128 threads
// computes a 128 x 128 tile of Y (128 batch rows x 128 output units) as one
// tcgen05.mma.kind::f16 chain over K = 64 (four K = 16 steps), BF16 operands from shared memory,
// FP32 accumulator in tensor memory (TMEM, 128 lanes x 128 columns).  The epilogue reads the
// accumulator back with tcgen05.ld (warp w owns TMEM lanes 32w .. 32w + 31, i.e. batch rows), turns
// each 32 x 32 piece over in shared memory so global rows are accessed 128 bytes at a time, and
// writes Y + b3.
//
// Training with a fixed output layer (tc_train_kernel): residual against the targets, loss and
// back-propagation into the hidden layer in one pass over the targets (see there).
//
// Operand layout in shared memory: the canonical K-major layout without swizzle.  A tile of R
// rows x 64 K (BF16) is cut into core matrices of 8 rows x 16 bytes (8 K values), each 128
// contiguous bytes; core matrix (row group g, K chunk c) sits at byte (8 g + c) * 128.  So the
// matrix descriptor's leading byte offset (next core matrix along K) is 128 and its stride byte
// offset (next 8-row group) is 1024; the K = 16 step kk starts 256 kk bytes in.
//
// Every wait is bounded: if the MMA completion does not arrive within kWaitLimit polls the CTA
// raises the error word, waits (bounded again) and still frees its TMEM columns.
#include <cuda_bf16.h>

#include <algorithm>

#include "sg_internal.h"

namespace sg {
namespace {

constexpr int kTcRows = 128;           // batch rows per CTA (MMA M)
constexpr int kTcUnits = 128;          // output units per CTA (MMA N)
constexpr int kTcK = 64;               // K (h2 padded with zeros)
constexpr int kTcTileBytes = kTcRows * kTcK * 2;  // 16 KB per operand tile
// Dynamic shared memory requested per CTA: the two tiles plus room that keeps at most four CTAs
// on an SM, so their TMEM columns (128 each) never exceed the SM's 512.
constexpr int kTcSmem = 56 * 1024;
constexpr unsigned kTcCols = 128;

__device__ __forceinline__ unsigned long long tc_smem_desc(unsigned saddr, unsigned lbo_bytes = 128,
                                                           unsigned sbo_bytes = 1024) {
  const unsigned long long start = (saddr & 0x3FFFFu) >> 4;  // bits 0-13
  const unsigned long long lbo = lbo_bytes >> 4;              // bits 16-29
  const unsigned long long sbo = sbo_bytes >> 4;              // bits 32-45
  return start | (lbo << 16) | (sbo << 32) | (1ull << 46);    // version 1; no swizzle
}

__device__ __forceinline__ void tc_mma(unsigned d, unsigned long long a, unsigned long long b,
                                       unsigned idesc, int accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}\n" ::"r"(d),
      "l"(a), "l"(b), "r"(idesc), "r"(accumulate)
      : "memory");
}

__device__ __forceinline__ void tc_commit(unsigned long long* bar) {
  asm volatile(
      "tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n" ::"r"(
          smem_u32(bar))
      : "memory");
}

// 32 TMEM columns from taddr on: thread = TMEM lane of the warp's quarter.
__device__ __forceinline__ void tc_ld32(unsigned taddr, unsigned (&v)[32]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,"
      "%14,%15,%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];\n"
      : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]),
        "=r"(v[7]), "=r"(v[8]), "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]),
        "=r"(v[14]), "=r"(v[15]), "=r"(v[16]), "=r"(v[17]), "=r"(v[18]), "=r"(v[19]),
        "=r"(v[20]), "=r"(v[21]), "=r"(v[22]), "=r"(v[23]), "=r"(v[24]), "=r"(v[25]),
        "=r"(v[26]), "=r"(v[27]), "=r"(v[28]), "=r"(v[29]), "=r"(v[30]), "=r"(v[31])
      : "r"(taddr)
      : "memory");
  asm volatile("tcgen05.wait::ld.sync.aligned;\n" ::: "memory");
}

// Instruction descriptor of kind::f16: FP32 accumulator, BF16 A and B, both K-major, M = 128,
// N = 128.
constexpr unsigned kTcIdesc = (1u << 4)            // D format: F32
                              | (1u << 7)          // A format: BF16
                              | (1u << 10)         // B format: BF16
                              | ((kTcUnits >> 3) << 17)   // N >> 3
                              | ((kTcRows >> 4) << 24);   // M >> 4

// Byte offset of element (row, k) in the canonical layout above.
__device__ __forceinline__ int tc_off(int row, int k) {
  return (((row >> 3) * 8 + (k >> 3)) << 7) + ((row & 7) << 4) + ((k & 7) << 1);
}

__device__ __forceinline__ void tc_ld16(unsigned taddr, unsigned (&v)[16]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,"
      "%15}, [%16];\n"
      : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]),
        "=r"(v[7]), "=r"(v[8]), "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]),
        "=r"(v[14]), "=r"(v[15])
      : "r"(taddr)
      : "memory");
  asm volatile("tcgen05.wait::ld.sync.aligned;\n" ::: "memory");
}

template <typename TY>
__global__ void __launch_bounds__(128) tc_out_kernel(int B, int h2, int out,
                                                     const float* __restrict__ H2,
                                                     const __nv_bfloat16* __restrict__ W3h,
                                                     const float* __restrict__ b3,
                                                     TY* __restrict__ Y, int* __restrict__ err) {
  extern __shared__ __align__(1024) unsigned char smem_raw[];
  unsigned char* At = smem_raw;                     // H2 rows
  unsigned char* Bt = smem_raw + kTcTileBytes;      // W3 rows
  unsigned long long* bar = reinterpret_cast<unsigned long long*>(smem_raw + 2 * kTcTileBytes);
  unsigned* tslot = reinterpret_cast<unsigned*>(smem_raw + 2 * kTcTileBytes + 16);
  float* stage = reinterpret_cast<float*>(smem_raw + 2 * kTcTileBytes + 64);  // 4 x 32 x 33
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int j0 = blockIdx.x * kTcUnits, b0 = blockIdx.y * kTcRows;

  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;\n" ::"r"(
                     smem_u32(tslot)),
                 "r"(kTcCols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;\n" ::: "memory");
  }
  if (tid == 0) {
    mbar_init(bar, 1);
    asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
  }
  // operand tiles: 8 K values (16 bytes) per item; rows and K beyond the data are zero.  With
  // h2 = 64 a row is 16-byte aligned in both arrays and is read by vector loads.
  const bool full = h2 == kTcK;
  for (int it = tid; it < kTcRows * (kTcK / 8); it += blockDim.x) {
    const int row = it >> 3, kc = (it & 7) * 8;
    __align__(16) __nv_bfloat16 a[8], w[8];
    const int b = b0 + row, j = j0 + row;
    if (full) {
      float4 h0 = make_float4(0.f, 0.f, 0.f, 0.f), h1 = h0;
      if (b < B) {
        h0 = *reinterpret_cast<const float4*>(H2 + (size_t)b * kTcK + kc);
        h1 = *reinterpret_cast<const float4*>(H2 + (size_t)b * kTcK + kc + 4);
      }
      a[0] = __float2bfloat16_rn(h0.x); a[1] = __float2bfloat16_rn(h0.y);
      a[2] = __float2bfloat16_rn(h0.z); a[3] = __float2bfloat16_rn(h0.w);
      a[4] = __float2bfloat16_rn(h1.x); a[5] = __float2bfloat16_rn(h1.y);
      a[6] = __float2bfloat16_rn(h1.z); a[7] = __float2bfloat16_rn(h1.w);
      const uint4 wv = j < out ? *reinterpret_cast<const uint4*>(W3h + (size_t)j * kTcK + kc)
                               : make_uint4(0u, 0u, 0u, 0u);
      *reinterpret_cast<uint4*>(w) = wv;
    } else {
#pragma unroll
      for (int t = 0; t < 8; ++t) {
        const int k = kc + t;
        a[t] = __float2bfloat16_rn(b < B && k < h2 ? H2[(size_t)b * h2 + k] : 0.0f);
        w[t] = j < out && k < h2 ? W3h[(size_t)j * h2 + k] : __float2bfloat16_rn(0.0f);
      }
    }
    *reinterpret_cast<uint4*>(At + tc_off(row, kc)) = *reinterpret_cast<const uint4*>(a);
    *reinterpret_cast<uint4*>(Bt + tc_off(row, kc)) = *reinterpret_cast<const uint4*>(w);
  }
  // the tiles were written by ordinary stores: make them visible to the tensor core's proxy
  asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
  asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
  const unsigned tmem = *tslot;

  if (tid == 0) {
    const unsigned a0 = smem_u32(At), bb0 = smem_u32(Bt);
#pragma unroll
    for (int kk = 0; kk < kTcK / 16; ++kk)
      tc_mma(tmem, tc_smem_desc(a0 + 256u * kk), tc_smem_desc(bb0 + 256u * kk), kTcIdesc, kk);
    tc_commit(bar);
  }
  // warp-uniform: tcgen05.ld below is a .sync.aligned warp instruction
  const bool ok = __all_sync(0xffffffffu, mbar_wait_bounded(bar, 0));
  asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");

  if (ok) {
    // each warp reads its 32 rows x 32 columns at a time (thread = row), turns them over in its
    // own shared-memory stage (padded rows), and writes / reads the global arrays a row at a time
    // with the lanes along the units (128-byte accesses)
    float* S = stage + warp * 32 * 33;
#pragma unroll 1
    for (int c0 = 0; c0 < kTcUnits; c0 += 32) {
      unsigned v[32];
      const unsigned taddr = tmem + ((unsigned)(warp * 32) << 16) + (unsigned)c0;
      tc_ld32(taddr, v);
#pragma unroll
      for (int t = 0; t < 32; ++t) S[lane * 33 + t] = __uint_as_float(v[t]);
      __syncwarp();
      const int j = j0 + c0 + lane;
      const float bias = j < out ? b3[j] : 0.0f;
#pragma unroll 4
      for (int r = 0; r < 32; ++r) {
        const int b = b0 + warp * 32 + r;
        if (b < B && j < out) Y[(size_t)b * out + j] = (TY)(S[r * 33 + lane] + bias);
      }
      __syncwarp();
    }
  } else if (lane == 0) {
    atomicExch(err, 1);
    mbar_wait_bounded(bar, 0);  // let the MMAs finish (bounded) before the columns are freed
  }
  asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
  __syncthreads();
  if (warp == 0) {
    asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;\n" ::"r"(tmem),
                 "r"(kTcCols)
                 : "memory");
  }
}

// One training pass with a fixed output layer: residual dY = 2 (H2 W3^T + b3 - T) / (B out) (rounded
// to BF16), the sum of squares, and dH2 = dY W3, in one pass over the targets; dY never leaves the
// SM.  CTA (s, y) takes batch rows 128 y .. 128 y + 127 and the tiles of 128 output
// units s, s + S, ...; per tile
//   1. MMA 1: D1[unit][row] = W3 tile (M = 128 units, K = 64) x H2 (N = 128 rows): TMEM lanes are
//      units, so a warp's T values of one row are 128 contiguous bytes;
//   2. the epilogue forms dY for the thread's unit and 32 rows, eight rows at a time as one 16-byte
//      store into the dY tile;
//   3. MMA 2: D2[row][k] += dY tile (M = 128 rows, K = 128 units) x W3 tile (N = 64, K = 128 units),
//      both MN-major: the W3 tile of MMA 1 read the other way round (the core matrices are the
//      same bytes).
// T goes through shared memory in two buffers by 16-byte cp.async (arriving on an mbarrier per
// buffer): a row of T starts on any multiple of 4 bytes, so the copies take the 528 bytes from the
// 16-byte boundary at or below it and the threads read from the remainder (four cases, by the row
// mod 4).  A tile whose copies would leave T (the last units of a row, the first of a T off its
// alignment) is read by plain loads.  The W3 tile comes by one bulk copy from a copy of W3 kept in
// core-matrix order (W3c).
//
// Sixteen warps do the epilogue; a seventeenth fetches W3 and issues the MMAs: MMA 1 a tile ahead
// into the other half of D1, MMA 2 when the dY tile is full (mbarrier).  The epilogue warps have
// their results in registers before they wait for MMA 2 of the tile before, which reads the dY
// tile they write next, so that MMA 2 runs beside their loads and arithmetic.
//
// Measured on one GB300 at B = 256, out = 147 875 (151 MB of targets, 19 MB of W3): 61 us against
// 266 us for the residual kernel that wrote dY plus 83 us for the product that read it back; 2.8
// TB/s.  Without the copies of T the kernel runs in 37 us, without MMA 2 in 57 us: the copies'
// passage through the SM's load path bounds it (4-byte copies 62 us; one bulk copy per row 101 us,
// a warp issuing them one after the other; loads into registers, two CTAs per SM, 84 us).
// Memory order of the dY tile: core matrix (8 units) x (8 rows) of unit group g and row group r at
// byte 2048 g + 128 r, unit u of the group at 16 u.
constexpr int kTcDyBytes = 128 * 128 * 2;
constexpr int kTcTRow = 132;  // floats of a row's copy
constexpr int kTcTBytes = 128 * kTcTRow * 4;
constexpr int kTcTrainTiles = kTcTileBytes * 3 + kTcDyBytes + 2 * kTcTBytes;  // H2, two W3, dY, T
constexpr int kTcTrainSmem = kTcTrainTiles + 256;  // one CTA on an SM
constexpr unsigned kTcTrainCols = 512;             // D1 twice (128 columns each), D2 (64)
constexpr unsigned kTcMnIdesc = (1u << 4) | (1u << 7) | (1u << 10) | (1u << 15) | (1u << 16) |
                                ((64u >> 3) << 17) | ((128u >> 4) << 24);

__global__ void __launch_bounds__(544, 1) tc_train_kernel(
    int B, int h2, int out, const float* __restrict__ H2, const __nv_bfloat16* __restrict__ W3c,
    const float* __restrict__ b3, const float* __restrict__ T, float* __restrict__ part,
    float* __restrict__ lpart, int* __restrict__ err) {
  extern __shared__ __align__(1024) unsigned char smem_raw[];
  unsigned char* Ht = smem_raw;
  unsigned char* Wt = smem_raw + kTcTileBytes;
  unsigned char* Dy = smem_raw + 3 * kTcTileBytes;
  float* Tb = reinterpret_cast<float*>(smem_raw + 3 * kTcTileBytes + kTcDyBytes);
  unsigned long long* bar = reinterpret_cast<unsigned long long*>(smem_raw + kTcTrainTiles);
  unsigned long long *bar1 = bar, *bar2 = bar + 2, *wfull = bar + 3, *dyfull = bar + 5,
                     *tfull = bar + 6;  // of 2, 1, 2, 1 and 2
  unsigned* tslot = reinterpret_cast<unsigned*>(bar + 8);
  volatile int* vfail = reinterpret_cast<volatile int*>(bar + 9);
  float* red = reinterpret_cast<float*>(bar + 10);  // 16
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int b0 = blockIdx.y * kTcRows, S = gridDim.x;
  const int ntiles = (out + kTcUnits - 1) / kTcUnits;
  const int unit = (warp & 3) * 32 + lane;  // TMEM lane of this thread
  const int c0 = (warp >> 2) * 32;          // its first batch row in the block
  const int nrow = min(32, B - b0 - c0);    // rows of the batch among its 32 (may be <= 0)
  // tiles of this CTA (the launch gives every CTA at least one)
  const int n_tiles = (ntiles - (int)blockIdx.x + S - 1) / S;
  if (warp == 16) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;\n" ::"r"(
                     smem_u32(tslot)),
                 "r"(kTcTrainCols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;\n" ::: "memory");
  }
  if (tid == 0) {
    *vfail = 0;
    for (int i = 0; i < 5; ++i) mbar_init(&bar[i], 1);
    mbar_init(dyfull, 16);  // the epilogue warps
    mbar_init(&tfull[0], 512);  // their threads' copies
    mbar_init(&tfull[1], 512);
    asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
  }
  // the CTA's n-th tile by bulk copies (else by plain loads)?  Row r starts shift(r) values after a
  // 16-byte boundary
  const unsigned tw = (unsigned)(reinterpret_cast<unsigned long long>(T) >> 2);
  auto bulk_t = [&](int n) {
    const int j0 = (blockIdx.x + n * S) * kTcUnits;
    return j0 + kTcTRow <= out && (j0 >= 4 || (tw & 3u) == 0);
  };
  // 16-byte chunks tid, tid + 512, ... of the block's rows x 33: place in T (of tile 0), or null.
  // (Pointers: a row of the block starts up to 127 x 4 out bytes in, past 4 GB from out = 8.5 M on.)
  constexpr int kChunks = kTcTRow / 4, kMine = (kTcRows * kChunks + 511) / 512;
  const unsigned char* tsrc[kMine];
#pragma unroll
  for (int k = 0; k < kMine; ++k) {
    const int c = (tid & 511) + 512 * k, r = c / kChunks;
    const unsigned long long row = reinterpret_cast<unsigned long long>(T + (size_t)(b0 + r) * out) & ~15ull;
    tsrc[k] = r < kTcRows && b0 + r < B
                  ? reinterpret_cast<const unsigned char*>(row) + 16 * (c - r * kChunks)
                  : nullptr;
  }
  auto load_t = [&](int n) {
    if (n < n_tiles && bulk_t(n)) {
      const size_t at = (size_t)(blockIdx.x + n * S) * (kTcUnits * 4);
      const unsigned dst = smem_u32(Tb) + (n & 1) * kTcTBytes + 16u * tid;
#pragma unroll
      for (int k = 0; k < kMine; ++k)
        if (tsrc[k] != nullptr)
          asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(dst + 8192u * k), "l"(tsrc[k] + at)
                       : "memory");
    }
    // (arrives when this thread's copies so far have landed)
    asm volatile("cp.async.mbarrier.arrive.noinc.shared::cta.b64 [%0];\n" ::"r"(smem_u32(&tfull[n & 1])) : "memory");
  };
  for (int it = tid; it < kTcRows * (kTcK / 8); it += blockDim.x) {  // H2 rows as BF16
    const int row = it >> 3, kc = (it & 7) * 8, b = b0 + row;
    __align__(16) __nv_bfloat16 a[8];
#pragma unroll
    for (int t = 0; t < 8; ++t)
      a[t] = __float2bfloat16_rn(b < B && kc + t < h2 ? H2[(size_t)b * h2 + kc + t] : 0.0f);
    *reinterpret_cast<uint4*>(Ht + tc_off(row, kc)) = *reinterpret_cast<const uint4*>(a);
  }
  asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
  asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
  const unsigned tmem = *tslot, d2 = tmem + 256;
  // a wait that has failed once is not made again: the loops run out on garbage that ends as NaN
  auto wait = [&](unsigned long long* b, int phase) {
    if (!*vfail && !mbar_wait_bounded(b, (unsigned)(phase & 1))) *vfail = 1;
  };
  // the tiles' sums, compensated (a thread has 32 squares a tile, thousands in all; in FP64, whose
  // pipe takes 65 cycles an instruction, a step at out = 42 250, B = 83 took 45.6 us instead of 44.1)
  float lsum = 0.0f, lcomp = 0.0f;
  if (warp == 16) {
    if (lane == 0) {
      const unsigned ha = smem_u32(Ht), wa = smem_u32(Wt), da = smem_u32(Dy);
      auto load_w = [&](int n) {
        if (n >= n_tiles) return;
        if (n + 2 < n_tiles)
          asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(
                           W3c + (size_t)(blockIdx.x + (n + 2) * S) * (kTcTileBytes / 2)),
                       "r"(kTcTileBytes)
                       : "memory");
        mbar_expect_tx(&wfull[n & 1], kTcTileBytes);
        bulk_g2s(Wt + (n & 1) * kTcTileBytes, W3c + (size_t)(blockIdx.x + n * S) * (kTcTileBytes / 2),
                 kTcTileBytes, &wfull[n & 1]);
      };
      auto mma1 = [&](int n) {  // D1[n & 1] of the CTA's n-th tile
        if (n >= n_tiles) return;
        wait(&wfull[n & 1], n >> 1);
        if (*vfail) return;
        const unsigned w = wa + (n & 1) * kTcTileBytes;
#pragma unroll
        for (int kk = 0; kk < kTcK / 16; ++kk)
          tc_mma(tmem + (n & 1) * 128, tc_smem_desc(w + 256u * kk), tc_smem_desc(ha + 256u * kk),
                 kTcIdesc, kk);
        tc_commit(&bar1[n & 1]);
      };
      load_w(0);
      load_w(1);
      mma1(0);
      int n = 0;
      for (; n < n_tiles && !*vfail; ++n) {
        mma1(n + 1);  // the epilogue of tile n - 1, which read this half of D1, has filled its dY tile
        wait(dyfull, n);
        if (*vfail) break;
        asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
        const unsigned w = wa + (n & 1) * kTcTileBytes;
#pragma unroll
        for (int kk = 0; kk < kTcUnits / 16; ++kk)  // K step of 16 units: two unit groups
          tc_mma(d2, tc_smem_desc(da + 4096u * kk, 2048, 128), tc_smem_desc(w + 2048u * kk, 1024, 128),
                 kTcMnIdesc, n > 0 || kk > 0);
        tc_commit(bar2);
        wait(bar2, n);
        if (!*vfail) load_w(n + 2);
      }
      if (*vfail) {  // let what is in flight land (bounded) before the columns and the tiles go
        atomicExch(err, 1);
        for (int k = n; k <= n + 1 && k < n_tiles; ++k) {
          mbar_wait_bounded(&bar1[k & 1], (unsigned)((k >> 1) & 1));
          mbar_wait_bounded(&wfull[k & 1], (unsigned)((k >> 1) & 1));
        }
        if (n < n_tiles) mbar_wait_bounded(bar2, (unsigned)(n & 1));
      }
    }
    __syncwarp();
  } else {
    int shift[4];  // of rows c0 + q, by q mod 4 (c0 is a multiple of 4)
#pragma unroll
    for (int q = 0; q < 4; ++q) shift[q] = (int)((tw + (unsigned)(b0 + q) * (unsigned)out) & 3u);
    const float scale = 2.0f / ((float)B * (float)out);
    auto bias_of = [&](int n) {
      const int j = (blockIdx.x + n * S) * kTcUnits + unit;
      return n < n_tiles && j < out ? b3[j] : 0.0f;
    };
    load_t(0);
    load_t(1);
    float bias = bias_of(0);
    for (int n = 0; n < n_tiles; ++n) {
      const int j = (blockIdx.x + n * S) * kTcUnits + unit;
      const bool bulk = bulk_t(n);
      const float bias_next = bias_of(n + 1);
      wait(&bar1[n & 1], n >> 1);
      wait(&tfull[n & 1], n >> 1);
      __syncwarp();
      asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
      const unsigned ta = tmem + ((unsigned)((warp & 3) * 32) << 16) + (unsigned)((n & 1) * 128 + c0);
      float* tp = Tb + (n & 1) * (kTcTBytes / 4) + c0 * kTcTRow + unit;
      __align__(16) __nv_bfloat162 dy[16];
      if (!bulk) {  // plain loads of this thread's own values (zero beyond the units and the batch)
        const float* tg = T + (size_t)(b0 + c0) * out + j;
#pragma unroll 1
        for (int q = 0; q < 32; ++q)
          tp[q * kTcTRow + shift[0]] = q < nrow && j < out ? tg[(size_t)q * out] : 0.0f;
      }
      const int sh1 = bulk ? shift[1] : shift[0], sh2 = bulk ? shift[2] : shift[0],
                sh3 = bulk ? shift[3] : shift[0];
      float tsum = 0.0f;
      // (units beyond the layer have W3 = b3 = T = 0, rows beyond the batch are masked)
#pragma unroll
      for (int hf = 0; hf < 32; hf += 16) {
        unsigned v[16];
        tc_ld16(ta + hf, v);
#pragma unroll
        for (int q = 0; q < 16; q += 2) {
          const float* t2 = tp + (hf + q) * kTcTRow;
          float r0 = (__uint_as_float(v[q]) + bias) - t2[q & 2 ? sh2 : shift[0]];
          float r1 = (__uint_as_float(v[q + 1]) + bias) - t2[kTcTRow + (q & 2 ? sh3 : sh1)];
          if (hf + q >= nrow) r0 = 0.0f;
          if (hf + q + 1 >= nrow) r1 = 0.0f;
          tsum = fmaf(r0, r0, tsum);
          tsum = fmaf(r1, r1, tsum);
          dy[(hf + q) / 2] = __floats2bfloat162_rn(scale * r0, scale * r1);
        }
      }
      const float add = tsum - lcomp, sum = lsum + add;
      lcomp = fabsf(sum) < INFINITY ? (sum - lsum) - add : 0.0f;
      lsum = sum;
      bias = bias_next;
      asm volatile("bar.sync 1, 512;\n" ::: "memory");  // every warp has read this T buffer
      load_t(n + 2);
      if (n > 0) wait(bar2, n - 1);  // MMA 2 of the tile before has read the dY tile
#pragma unroll
      for (int q = 0; q < 32; q += 8)
        *reinterpret_cast<uint4*>(Dy + (unit >> 3) * 2048 + ((c0 + q) >> 3) * 128 + (unit & 7) * 16) =
            *reinterpret_cast<const uint4*>(&dy[q / 2]);
      asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
      asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
      __syncwarp();
      if (lane == 0) asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];\n" ::"r"(smem_u32(dyfull)) : "memory");
    }
    asm volatile("cp.async.wait_all;\n" ::: "memory");
    wait(bar2, n_tiles - 1);
  }
  __syncthreads();
  const bool failed = *vfail != 0;
  asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
  if (warp < 8) {  // D2: lanes are batch rows; warps 0-3 take columns 0-31, warps 4-7 columns 32-63
    const int b = b0 + unit;
    float* o = part + ((size_t)blockIdx.x * B + b) * 64 + (warp >> 2) * 32;
    if (!failed) {
      unsigned v[32];
      tc_ld32(d2 + ((unsigned)((warp & 3) * 32) << 16) + (unsigned)((warp >> 2) * 32), v);
      if (b < B) {
#pragma unroll
        for (int t = 0; t < 32; t += 4)
          *reinterpret_cast<uint4*>(o + t) = make_uint4(v[t], v[t + 1], v[t + 2], v[t + 3]);
      }
    } else if (b < B) {
      for (int t = 0; t < 32; ++t) o[t] = __int_as_float(0x7fc00000);
    }
  }
  asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) lsum += __shfl_xor_sync(0xffffffffu, lsum, o);
  if (lane == 0 && warp < 16) red[warp] = lsum;
  __syncthreads();
  if (warp == 16) {
    asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;\n" ::"r"(tmem),
                 "r"(kTcTrainCols)
                 : "memory");
  }
  if (warp == 0) {
    float l = lane < 16 ? red[lane] : 0.0f;
#pragma unroll
    for (int o = 8; o > 0; o >>= 1) l += __shfl_xor_sync(0xffffffffu, l, o);
    if (lane == 0) lpart[(size_t)blockIdx.y * gridDim.x + blockIdx.x] = l;
  }
}

// W3c: W3 rounded to BF16 in tiles of 128 units x 64, each in core-matrix order (see tc_off),
// zero beyond out and h2.
__global__ void w3_tiles_kernel(int out, int h2, size_t total, const float* __restrict__ W3,
                                __nv_bfloat16* __restrict__ W3c) {
  for (size_t t = (size_t)blockIdx.x * blockDim.x + threadIdx.x; t < total;
       t += (size_t)gridDim.x * blockDim.x) {
    const int w = (int)(t % (kTcUnits * kTcK));
    const int core = w >> 6, k = (core & 7) * 8 + (w & 7);
    const size_t j = t / (kTcUnits * kTcK) * kTcUnits + (core >> 3) * 8 + ((w >> 3) & 7);
    W3c[t] = __float2bfloat16_rn(k < h2 && j < (size_t)out ? W3[j * h2 + k] : 0.0f);
  }
}

}  // namespace

// Launch of the forward output layer on the tensor cores: Y (float Yf or double Yd) = H2 W3^T + b3.
int launch_out_tc(int B, int h2, int out, const float* H2, const __nv_bfloat16* W3h,
                  const float* b3, float* Yf, double* Yd, int* err, cudaStream_t st) {
  if (h2 < 1 || h2 > kTcK || B < 1 || out < 1) return fail(SG_ERR_ARG, "tensor-core output layer: sizes");
  const dim3 grid((out + kTcUnits - 1) / kTcUnits, (B + kTcRows - 1) / kTcRows);
  if (Yd != nullptr) {
    auto k = tc_out_kernel<double>;
    SG_TRY(ensure_smem((const void*)k, kTcSmem));
    k<<<grid, 128, kTcSmem, st>>>(B, h2, out, H2, W3h, b3, Yd, err);
  } else {
    auto k = tc_out_kernel<float>;
    SG_TRY(ensure_smem((const void*)k, kTcSmem));
    k<<<grid, 128, kTcSmem, st>>>(B, h2, out, H2, W3h, b3, Yf, err);
  }
  return check_launch("tc_out");
}

// One training pass (see tc_train_kernel): part[s][row][64] holds *nsplit partial sums of dH2,
// lpart one loss partial per CTA (*nparts).  One CTA per SM, the batch blocks sharing the SMs.
int launch_train_tc(int B, int h2, int out, const float* H2, const __nv_bfloat16* W3c,
                    const float* b3, const float* T, float* part, float* lpart, int* err,
                    cudaStream_t st, int* nsplit, int* nparts) {
  if (h2 < 1 || h2 > kTcK || B < 1 || out < 1) return fail(SG_ERR_ARG, "tensor-core training pass: sizes");
  const int nb = (B + kTcRows - 1) / kTcRows, ntiles = (out + kTcUnits - 1) / kTcUnits;
  const int s = std::max(1, std::min(ntiles, kTcTrainCtas / nb));
  *nsplit = s;
  *nparts = s * nb;
  SG_TRY(ensure_smem((const void*)tc_train_kernel, kTcTrainSmem));
  tc_train_kernel<<<dim3(s, nb), 544, kTcTrainSmem, st>>>(B, h2, out, H2, W3c, b3, T, part, lpart, err);
  return check_launch("tc_train");
}

size_t w3_tiles_elems(int out) { return (size_t)(out + kTcUnits - 1) / kTcUnits * kTcUnits * kTcK; }

int launch_w3_tiles(int out, int h2, const float* W3, __nv_bfloat16* W3c, cudaStream_t st) {
  w3_tiles_kernel<<<608, 256, 0, st>>>(out, h2, w3_tiles_elems(out), W3, W3c);
  return check_launch("w3_tiles");
}

}  // namespace sg
