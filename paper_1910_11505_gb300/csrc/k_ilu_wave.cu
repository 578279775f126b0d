// ILU(0) block solves of many columns in the natural node order (FP32): a wavefront of warps without
// CTA barriers, one CTA per column.
//
// Row (x, y) of the lower factor needs (x-1, y), (x+1, y-1), (x, y-1), (x-1, y-1), so the rows
// x + 2y = const are independent (k_precond.cu).  Here a lane owns a grid line and a warp 32 of
// them: at step s lane r holds x = s - 2r, its left neighbour is its own last result, and the
// three values of the line below arrive by one shuffle per step from lane r - 1, which computed
// z(x+1, y-1) in the step before (the two older ones are kept in registers).  Warp w takes the lines
// after warp w - 1's; its last lane's results go through shared memory, with an mbarrier for every
// eight steps.  The upper factor is the same sweep with steps, lanes and warps in reverse.
//
// Layout: everything that a step needs lies in the order of the steps.  The columns are stored as
// [column][warp][step][lane] (zero where a lane has no node), filled from and written back to the
// N x P field by two kernels that read and write whole nodes; the factors as one stream per set
// and warp.  A producer warp beside each compute warp fetches both, kWaveBlock steps at a time, by
// bulk copies into a ring, so that a step of the compute warp is some twenty instructions: a lone
// warp runs a few dependent instructions per hundred cycles, and the column's strided reads and
// writes inside the sweep had taken half of the time.
//
// Bound: the dependent chain of a step (a shuffle and two multiply-adds) and its instructions.
// (FP64 spreads a row's four multiply-adds of 65 cycles over two lanes, k_ilu_lines.cu.)  One application by 84 columns on one GB300, barrier kernels
// -> here: 32 x 32 41.5 -> 21 us, 128 x 128 150 -> 60 us, 256 x 256 571 -> 121 us.
#include <algorithm>

#include "sg_internal.h"

namespace sg {

namespace {

constexpr int kWaveMaxWarps = 8;   // compute warps: lines up to 256
// Fewer lines go to the barrier kernels: 7 lines take 16 us there and 20 us here (62 steps of
// idle lanes and a third launch), 15 lines 25.0 and 20.8, 31 lines 41.4 and 21.1.
constexpr int kWaveMinLines = 12;
constexpr int kWaveBlock = 8;      // steps of a ring slot
constexpr int kWaveSlots = 4;
constexpr int kWaveCols = 64;      // columns per CTA of the kernels that fill and empty the buffer
constexpr int kSub = 4;            // steps whose factors are in registers ahead

// Values per step of a warp's factor stream: per lane the couplings to its own last result and to
// the three values of the line before, newest first; in the upper sweep then 1/u_ii per lane.
template <bool UPPER>
__host__ __device__ constexpr int wave_vals() { return UPPER ? 32 * 5 : 32 * 4; }
constexpr int kSlotFloats = kWaveBlock * (32 * 5 + 32);
__host__ __device__ constexpr int wave_steps(int nx) { return (nx + 62 + kWaveBlock - 1) / kWaveBlock * kWaveBlock; }
// The last lane's results of every step, and what the reads past the last step meet.
__host__ __device__ constexpr int wave_bnd(int nx) { return wave_steps(nx) + 72; }

size_t wave_smem(int nx) {
  const int warps = (nx + 31) / 32, blocks = wave_steps(nx) / kWaveBlock;
  return (size_t)warps * (4 * kWaveSlots * kSlotFloats + 8 * blocks + 4 * wave_bnd(nx));
}

struct WaveBars {
  unsigned long long full[kWaveMaxWarps][kWaveSlots], empty[kWaveMaxWarps][kWaveSlots];
};

// Producer of one warp's sweep (one thread): per block of steps the factors and the column values.
template <bool UPPER>
__device__ __forceinline__ void wave_produce(const float* fac, const float* val, float* ring,
                                             unsigned long long* full, unsigned long long* empty,
                                             unsigned use0, int nblk, volatile int* vfail) {
  constexpr int kVals = wave_vals<UPPER>();
  int b = 0;
  for (; b < nblk; ++b) {
    const unsigned u = use0 + b, slot = u % kWaveSlots;
    if (u >= kWaveSlots && (*vfail || !mbar_wait_bounded(&empty[slot], ((u / kWaveSlots) - 1u) & 1u))) {
      *vfail = 1;
      break;
    }
    float* dst = ring + slot * kSlotFloats;
    mbar_expect_tx(&full[slot], 4u * kWaveBlock * (kVals + 32));
    bulk_g2s(dst, fac + (size_t)b * kWaveBlock * kVals, 4u * kWaveBlock * kVals, &full[slot]);
    bulk_g2s(dst + kWaveBlock * 160, val + (size_t)(UPPER ? nblk - 1 - b : b) * kWaveBlock * 32,
             4u * kWaveBlock * 32, &full[slot]);
  }
  // what is under way lands before the CTA ends, also when a compute warp gave up
  for (int c = max(0, b - kWaveSlots); c < b; ++c)
    mbar_wait_bounded(&full[(use0 + c) % kWaveSlots], ((use0 + c) / kWaveSlots) & 1u);
}

// One sweep of a compute warp: results to val (in place of the column's values), the last lane's
// of step t to bnd_own[t]; done_own[i] is arrived at after steps 8 i .. 8 i + 7.
template <bool UPPER>
__device__ __forceinline__ void wave_sweep(float* val, const float* ring, unsigned long long* full,
                                           unsigned long long* empty, unsigned use0, float* bnd_own,
                                           const float* bnd_prev, unsigned long long* done_own,
                                           unsigned long long* done_prev, int steps, bool first,
                                           volatile int* vfail) {
  constexpr int kVals = wave_vals<UPPER>();
  const int lane = threadIdx.x & 31, nblk = steps / kWaveBlock;
  const int in_lane = UPPER ? 31 : 0, out_lane = 31 - in_lane;
  float z = 0.0f, up2 = 0.0f, up3 = 0.0f, bn = 0.0f;
  float4 f[2][kSub];
  float dinv[2][kSub], wv[2][kSub];
  auto take = [&](int b, int h, float4(&fo)[kSub], float(&di)[kSub], float(&wo)[kSub]) {
    const unsigned slot = (use0 + b) % kWaveSlots;
    const float* fb = ring + slot * kSlotFloats + h * kSub * kVals;
    const float* vb = ring + slot * kSlotFloats + kWaveBlock * 160;
#pragma unroll
    for (int j = 0; j < kSub; ++j) {
      fo[j] = *reinterpret_cast<const float4*>(fb + j * kVals + 4 * lane);
      if (UPPER) di[j] = fb[j * kVals + 128 + lane];
      const int t = h * kSub + j;
      wo[j] = vb[(UPPER ? kWaveBlock - 1 - t : t) * 32 + lane];
    }
  };
  auto wait_block = [&](int b) {
    const unsigned u = use0 + b;
    mbar_wait_or_fail(&full[u % kWaveSlots], (u / kWaveSlots) & 1u, vfail);
  };
  wait_block(0);
  take(0, 0, f[0], dinv[0], wv[0]);
  float* out = val + (UPPER ? (size_t)(steps - 1) * 32 : 0) + lane;
  for (int b = 0; b < nblk; ++b) {
    // this block's steps read ahead to step 8 b + 71 of the line before
    if (!first) {
      mbar_wait_or_fail(&done_prev[min(b + 8, nblk - 1)], UPPER ? 1u : 0u, vfail);
      if (b == 0) {  // the line before at the next and at this node of the first step
        bn = bnd_prev[63];
        if (lane == in_lane) up2 = bnd_prev[62];
      }
    }
    const float* bp = bnd_prev + 8 * b + 64;
    float* bo = bnd_own + 8 * b;
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      if (h == 0) {
        take(b, 1, f[1], dinv[1], wv[1]);
      } else if (b + 1 < nblk) {
        wait_block(b + 1);
        take(b + 1, 0, f[0], dinv[0], wv[0]);
      }
#pragma unroll
      for (int j = 0; j < kSub; ++j) {
        const int t = h * kSub + j;
        const float sh = UPPER ? __shfl_down_sync(0xffffffffu, z, 1) : __shfl_up_sync(0xffffffffu, z, 1);
        const float up1 = lane == in_lane ? bn : sh;
        float v = wv[h][j];
        if (UPPER) v *= dinv[h][j];
        if (!first) bn = bp[t];
        v = fmaf(-f[h][j].w, up3, v);
        v = fmaf(-f[h][j].z, up2, v);
        v = fmaf(-f[h][j].x, z, v);
        z = fmaf(-f[h][j].y, up1, v);
        up3 = up2;
        up2 = up1;
        *out = z;
        out += UPPER ? -32 : 32;
        if (lane == out_lane) bo[t] = z;
      }
      if (h == 0) {
        __syncwarp();  // both halves of this block are in registers
        if (lane == 0) asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];\n" ::"r"(smem_u32(&empty[(use0 + b) % kWaveSlots])) : "memory");
      }
    }
    if (lane == out_lane)
      asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];\n" ::"r"(smem_u32(&done_own[b])) : "memory");
  }
}

// CTA c solves column c with factor set (fac_per_col ? c : 0), in place in V.  Warps 0 .. warps - 1
// compute, the others produce.
__global__ void __launch_bounds__(kWaveMaxWarps * 64, 1) ilu_wave_kernel(
    int nx, int fac_per_col, const float* __restrict__ low, const float* __restrict__ upp,
    float* V, const int* __restrict__ done) {
  if (done != nullptr && *done) return;
  extern __shared__ __align__(128) unsigned char smem_raw[];
  __shared__ WaveBars bars;
  __shared__ int s_fail;
  volatile int* vfail = &s_fail;
  const int warps = (nx + 31) / 32, steps = wave_steps(nx), nblk = steps / kWaveBlock;
  const int wp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const bool producer = wp >= warps;
  const int w = producer ? wp - warps : wp;
  float* ring = reinterpret_cast<float*>(smem_raw) + (size_t)w * kWaveSlots * kSlotFloats;
  unsigned long long* done8 = reinterpret_cast<unsigned long long*>(
      smem_raw + (size_t)warps * 4 * kWaveSlots * kSlotFloats);
  float* bnd = reinterpret_cast<float*>(done8 + (size_t)warps * nblk);
  if (threadIdx.x == 0) s_fail = 0;
  for (int i = threadIdx.x; i < warps * nblk; i += blockDim.x) mbar_init(&done8[i], 1);
  for (int i = threadIdx.x; i < warps * kWaveSlots; i += blockDim.x) {
    mbar_init(&bars.full[i / kWaveSlots][i % kWaveSlots], 1);
    mbar_init(&bars.empty[i / kWaveSlots][i % kWaveSlots], 1);
  }
  for (int i = threadIdx.x; i < warps * 72; i += blockDim.x) bnd[(size_t)(i / 72) * wave_bnd(nx) + steps + i % 72] = 0.0f;
  asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
  asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
  __syncthreads();
  const size_t at = ((size_t)(fac_per_col ? blockIdx.x : 0) * warps + w) * steps;
  float* val = V + ((size_t)blockIdx.x * warps + w) * steps * 32;
  const int nb = wave_bnd(nx);
  for (int up = 0; up < 2; ++up) {
    const unsigned use0 = up ? nblk : 0;
    if (producer) {
      if (lane == 0) {
        if (up)
          wave_produce<true>(upp + at * wave_vals<true>(), val, ring, bars.full[w], bars.empty[w], use0, nblk, vfail);
        else
          wave_produce<false>(low + at * wave_vals<false>(), val, ring, bars.full[w], bars.empty[w], use0, nblk, vfail);
      }
    } else if (up) {
      const int pr = w + 1 < warps ? w + 1 : w;
      wave_sweep<true>(val, ring, bars.full[w], bars.empty[w], use0, bnd + (size_t)w * nb, bnd + (size_t)pr * nb,
                       done8 + w * nblk, done8 + pr * nblk, steps, w == warps - 1, vfail);
    } else {
      const int pr = w > 0 ? w - 1 : 0;
      wave_sweep<false>(val, ring, bars.full[w], bars.empty[w], use0, bnd + (size_t)w * nb, bnd + (size_t)pr * nb,
                        done8 + w * nblk, done8 + pr * nblk, steps, w == 0, vfail);
    }
    // the upper sweep's copies read what this sweep has stored
    asm volatile("fence.proxy.async;\n" ::: "memory");
    __syncthreads();
  }
  if (*vfail)  // a wait gave up: no caller may take the column as a result
    for (int i = threadIdx.x; i < warps * steps * 32; i += blockDim.x)
      V[(size_t)blockIdx.x * warps * steps * 32 + i] = __int_as_float(0x7fc00000);
}

// Node of (warp, step, lane), or -1.
__device__ __forceinline__ int wave_node(int m, int w, int s, int lane) {
  const int nx = m - 2, xi = s - 2 * lane, r = 32 * w + lane;
  return xi >= 0 && xi < nx && r < nx ? 1 + xi + m * (1 + r) : -1;
}

// V[c][w][s][lane] = R[node, c] (zero without a node).  CTA (s, w, z): 32 nodes, kWaveCols columns.
__global__ void __launch_bounds__(256) wave_in_kernel(int m, int P, const float* __restrict__ R,
                                                      float* __restrict__ V,
                                                      const int* __restrict__ done) {
  if (done != nullptr && *done) return;
  __shared__ float tile[32][kWaveCols + 1];
  const int s = blockIdx.x, w = blockIdx.y, steps = gridDim.x, warps = gridDim.y;
  const int lane = threadIdx.x & 31, wp = threadIdx.x >> 5;
  const int c0 = blockIdx.z * kWaveCols, nc = min(kWaveCols, P - c0);
  for (int l = wp; l < 32; l += 8) {
    const int node = wave_node(m, w, s, l);
    for (int c = lane; c < nc; c += 32) tile[l][c] = node >= 0 ? R[(size_t)node * P + c0 + c] : 0.0f;
  }
  __syncthreads();
  for (int c = wp; c < nc; c += 8)
    V[(((size_t)(c0 + c) * warps + w) * steps + s) * 32 + lane] = tile[lane][c];
}

// Z[node, c] = V[c][w][s][lane]; CTAs beyond the steps: the boundary rows, scaled by 1/u_ii (slot 4
// of the level-major factors).
__global__ void __launch_bounds__(256) wave_out_kernel(int m, int N, int P, int steps, int fac_per_col,
                                                       const int* __restrict__ lev_off,
                                                       const float* __restrict__ lu9,
                                                       const float* __restrict__ V,
                                                       const float* __restrict__ R,
                                                       float* __restrict__ Z,
                                                       const int* __restrict__ done) {
  if (done != nullptr && *done) return;
  __shared__ float tile[32][kWaveCols + 1];
  const int s = blockIdx.x, w = blockIdx.y, warps = gridDim.y;
  const int lane = threadIdx.x & 31, wp = threadIdx.x >> 5;
  const int c0 = blockIdx.z * kWaveCols, nc = min(kWaveCols, P - c0);
  if (s >= steps) {
    const int nb = 4 * (m - 1), parts = (gridDim.x - steps) * warps;
    for (int k = ((s - steps) * warps + w) * 8 + wp; k < nb; k += parts * 8) {
      const int side = k / (m - 1), q = k - side * (m - 1);
      const int x = side == 0 ? q : side == 1 ? m - 1 : side == 2 ? m - 1 - q : 0;
      const int y = side == 0 ? 0 : side == 1 ? q : side == 2 ? m - 1 : m - 1 - q;
      const int l = x + 2 * y, ylo = max(0, (l - (m - 1) + 1) >> 1), pos = lev_off[l] + (y - ylo);
      for (int c = c0 + lane; c < c0 + nc; c += 32) {
        const size_t o = (size_t)(x + m * y) * P + c;
        Z[o] = R[o] * lu9[((size_t)(fac_per_col ? c : 0) * 9 + 4) * N + pos];
      }
    }
    return;
  }
  for (int c = wp; c < nc; c += 8)
    tile[lane][c] = V[(((size_t)(c0 + c) * warps + w) * steps + s) * 32 + lane];
  __syncthreads();
  for (int l = wp; l < 32; l += 8) {
    const int node = wave_node(m, w, s, l);
    if (node >= 0)
      for (int c = lane; c < nc; c += 32) Z[(size_t)node * P + c0 + c] = tile[l][c];
  }
}

// Factor streams from the level-major slots: thread (set, warp, step, lane); the upper stream in
// the order of its sweep, last step first.
__global__ void wave_factors_kernel(int m, int N, int nfac, const int* __restrict__ lev_off,
                                    const double* __restrict__ lu9, float* __restrict__ low,
                                    float* __restrict__ upp) {
  const int nx = m - 2, warps = (nx + 31) / 32, steps = wave_steps(nx);
  const long long total = (long long)nfac * warps * steps * 32;
  for (long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x; t < total;
       t += (long long)gridDim.x * blockDim.x) {
    const int lane = (int)(t & 31);
    const long long ws = t >> 5;
    const int s = (int)(ws % steps);
    const long long fw = ws / steps;
    const int w = (int)(fw % warps), f = (int)(fw / warps);
    const int node = wave_node(m, w, s, lane);
    const int x = node >= 0 ? node % m : 0, y = node >= 0 ? node / m : 0;
    const int l = x + 2 * y, ylo = max(0, (l - (m - 1) + 1) >> 1), pos = lev_off[l] + (y - ylo);
    auto slot = [&](int sl) { return node >= 0 ? (float)lu9[((size_t)f * 9 + sl) * N + pos] : 0.0f; };
    float* o = low + ws * wave_vals<false>() + 4 * lane;
    for (int q = 0; q < 4; ++q) o[q] = slot(3 - q);
    const long long wu = fw * steps + (steps - 1 - s);
    o = upp + wu * wave_vals<true>() + 4 * lane;
    for (int q = 0; q < 4; ++q) o[q] = slot(5 + q);
    upp[wu * wave_vals<true>() + 128 + lane] = slot(4);
  }
}

}  // namespace

// Factor streams and column buffer of the mean-based and Jacobi forms of a mixed system, where the
// mesh's lines fit and a sixteenth of the device's memory holds them.
int wave_setup(System& s, cudaStream_t st) {
  const int nx = s.pat.m - 2, warps = (nx + 31) / 32;
  if (s.lean || nx < kWaveMinLines || warps > kWaveMaxWarps || wave_smem(nx) + 1024 > smem_optin_max()) return SG_OK;
  const size_t lanes = (size_t)warps * wave_steps(nx) * 32, n = lanes * s.nfac;
  const size_t bytes = sizeof(float) * (9 * n + lanes * s.P);
  size_t free_b = 0, total_b = 0;
  if (cudaMemGetInfo(&free_b, &total_b) != cudaSuccess) {
    cudaGetLastError();
    return SG_OK;
  }
  if (bytes > total_b / 16 || free_b < bytes + total_b / 2) return SG_OK;
  SG_TRY(s.wave_low.alloc(n * 4));
  SG_TRY(s.wave_up.alloc(n * 5));
  SG_TRY(s.wave_v.alloc(lanes * s.P));
  const int grid = (int)std::min<size_t>((n + 255) / 256, 152 * 32);
  wave_factors_kernel<<<grid, 256, 0, st>>>(s.pat.m, s.N, s.nfac, s.lev9_off.p, s.lu9.p, s.wave_low.p,
                                            s.wave_up.p);
  return check_launch("wave_factors");
}

// Z = (block diagonal ILU)^-1 R for all P columns.
int launch_wave_solve(System& s, int fac_per_col, const float* R, float* Z, cudaStream_t st,
                      const int* done) {
  const int m = s.pat.m, nx = m - 2, warps = (nx + 31) / 32, steps = wave_steps(nx);
  const int parts = (s.P + kWaveCols - 1) / kWaveCols;
  const size_t smem = wave_smem(nx);
  SG_TRY(ensure_smem((const void*)ilu_wave_kernel, smem));
  {
    TimeScope ts(s.timer, K_OTHER, st);
    wave_in_kernel<<<dim3(steps, warps, parts), 256, 0, st>>>(m, s.P, R, s.wave_v.p, done);
  }
  SG_TRY(check_launch("wave_in"));
  {
    TimeScope ts(s.timer, K_ILU_SOLVE, st);
    ilu_wave_kernel<<<s.P, warps * 64, smem, st>>>(nx, fac_per_col, s.wave_low.p, s.wave_up.p,
                                                   s.wave_v.p, done);
  }
  SG_TRY(check_launch("ilu_wave"));
  TimeScope ts(s.timer, K_OTHER, st);
  wave_out_kernel<<<dim3(steps + 8, warps, parts), 256, 0, st>>>(m, s.N, s.P, steps, fac_per_col, s.lev9_off.p,
                                                             s.lu9_f32.p, s.wave_v.p, R, Z, done);
  return check_launch("wave_out");
}

}  // namespace sg
