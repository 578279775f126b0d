// ILU(0) block solves in the natural node order (FP64): a wavefront of warps whose lanes split each
// row's couplings; one CTA per column, the column in shared memory.
//
// As in k_ilu_wave.cu a lane owns a grid line (16 lines a warp here) and holds x = s - 2l at step s,
// and lane l - 1 has computed z(x+1, y-1) one step before.  An FP64 multiply-add holds its SM
// sub-partition for 65 cycles whatever the number of active lanes, and its result takes as long, so
// the four of a row are spread over two lanes: while lane l applies the two newest values (its own
// last result and the one that lane l - 1 has just found) to step s, lane l + 16 applies the two
// older ones to step s + 1, whose values are known by then.  Both halves run the same two
// instructions, and a step's chain is two shuffles and two multiply-adds.
//
//   iteration t:  A = q of lane l + 16,  B = q of lane l - 1 (or of the last lane of the warp before)
//     lanes 0-15 (step t - 1):   q = (A - f0 q) - f1 B                     f0: (x-1, y), f1: (x+1, y-1)
//     lanes 16-31 (step t):      q = (w - f0 B of t - 1) - f1 B            f0: (x-1, y-1), f1: (x, y-1)
//
// The upper factor runs with warps, lanes and x reversed.  A warp that has ended its lower sweep
// scales its lines by 1/u_ii and goes on with the upper one when the warp before has; no CTA
// barrier stands between.  The factors lie in the order of the iterations and come through a ring per
// warp, filled by a producer warp's bulk copies.
//
// Bound: that chain, 3 m iterations a sweep, and 36 of each warp's start behind the one before.
// Measured on one GB300, barrier kernel -> here (the solves of all columns, 6 of them unless
// stated): 32 x 32 52 -> 41 us, 64 x 64 93 -> 74 us (35 columns), 128 x 128 182 -> 150 us; an iteration
// takes 227 cycles without the waits for the ring and the warp before, 260 with them.
#include <algorithm>

#include "sg_internal.h"

namespace sg {

namespace {

constexpr int kLineWarps = 9;   // compute warps of 16 lines at most
// Fewer lines go to the barrier kernels: 7 lines take 19.9 us there and 22.4 us here, 15 lines 30.5
// and 24.6, 31 lines 52.3 and 40.7.
constexpr int kLineMin = 12;
constexpr int kLineBlock = 4;   // iterations of a ring slot and of one hand-over between warps
constexpr int kLineSlots = 4;
constexpr int kLineRing = kLineSlots * kLineBlock * 32;  // pairs of values per warp

__host__ __device__ constexpr int line_warps(int nx) { return (nx + 15) / 16; }
__host__ __device__ constexpr int line_iters(int nx) { return (nx + 31 + 7) / 8 * 8; }
// The last lane's results of every iteration, and what the reads past the last one meet.
__host__ __device__ constexpr int line_bnd(int nx) { return line_iters(nx) + 40; }
// An odd stride: the lanes of a warp read the column at steps of stride - 2 values.
__host__ __device__ constexpr int line_stride(int nx) { return nx | 1; }

size_t line_smem(int nx) {
  const size_t warps = line_warps(nx);
  return warps * (16 * kLineRing + 8 * (size_t)line_bnd(nx) + 16 * (size_t)line_iters(nx) / kLineBlock) +
         8 * (size_t)nx * line_stride(nx);
}

struct LineBars {
  unsigned long long full[kLineWarps][kLineSlots], empty[kLineWarps][kLineSlots];
};

__device__ __forceinline__ void bar_arrive(unsigned long long* bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];\n" ::"r"(smem_u32(bar)) : "memory");
}

// One sweep of a compute warp over its 16 lines, in place in col.
template <bool UPPER>
__device__ __forceinline__ void line_sweep(const double2* ring, unsigned long long* full,
                                           unsigned long long* empty, unsigned use0, double* col,
                                           int nx, double* bnd_own, const double* bnd_prev,
                                           unsigned long long* done_own,
                                           unsigned long long* done_prev, int w, bool first,
                                           volatile int* vfail) {
  const int lane = threadIdx.x & 31, l = lane & 15;
  const bool older = lane >= 16;
  const int iters = line_iters(nx), line = 16 * w + (UPPER ? 15 - l : l);
  const bool live = line < nx;
  // at iteration t the older half reads, and the newer one writes, element xi + t of the line
  const int xi = -2 * l - (older ? 0 : 1);
  const unsigned nr = older && live ? nx : 0, nw = !older && live ? nx : 0;
  double* lcol = col + (live ? line : 0) * line_stride(nx) + (UPPER ? nx - 1 - xi : xi);
  const int src_a = lane | 16, src_b = (l - 1) & 15;
  const double2* src = ring + lane;
  double q = 0.0, bprev = 0.0, bn = 0.0;
  mbar_wait_or_fail(&full[use0 % kLineSlots], (use0 / kLineSlots) & 1u, vfail);
  double2 f = src[(use0 % kLineSlots) * kLineBlock * 32];
  double wv = (unsigned)xi < nr ? *lcol : 0.0;
  for (int t0 = 0; t0 < iters; t0 += kLineBlock) {
    // the iterations of this block read ahead to iteration t0 + 35 of the line before
    if (!first) {
      mbar_wait_or_fail(&done_prev[min(t0 + 32, iters - 1) / kLineBlock], 0u, vfail);
      if (t0 == 0) bn = bnd_prev[31];
    }
    const unsigned u = use0 + (unsigned)t0 / kLineBlock;
#pragma unroll
    for (int j = 0; j < kLineBlock; ++j) {
      const int t = t0 + j;
      const bool last = j + 1 == kLineBlock;
      const double A = __shfl_sync(0xffffffffu, q, src_a);
      const double Bs = __shfl_sync(0xffffffffu, q, src_b);
      const double B = l == 0 ? bn : Bs;
      const double d = fma(-f.x, older ? bprev : q, older ? wv : A);
      const double fy = f.y;
      // the next iteration's values
      if (!first) bn = bnd_prev[t + 32];
      if (last) {
        __syncwarp();  // this slot's factors are in registers
        if (lane == 0) bar_arrive(&empty[u % kLineSlots]);
        if (t + 1 < iters) mbar_wait_or_fail(&full[(u + 1) % kLineSlots], ((u + 1) / kLineSlots) & 1u, vfail);
      }
      f = src[((last ? u + 1 : u) % kLineSlots * kLineBlock + (j + 1) % kLineBlock) * 32];
      wv = 0.0;
      if ((unsigned)(xi + t + 1) < nr) wv = lcol[UPPER ? -(t + 1) : t + 1];
      q = fma(-fy, B, d);
      bprev = B;
      if ((unsigned)(xi + t) < nw) lcol[UPPER ? -t : t] = q;
      if (lane == 15) bnd_own[t] = q;
    }
    if (lane == 15) bar_arrive(&done_own[t0 / kLineBlock]);
  }
}

// CTA c solves column a = a0 + c with factor set (fac_per_col ? a : 0): Rt[a * ldN + node] to
// Z[node * P + a].  Warps 0 .. warps - 1 compute, the others fill their rings.
__global__ void __launch_bounds__(kLineWarps * 64, 1) ilu_lines_kernel(
    int m, int N, int ldN, int P, int a0, int fac_per_col, const int* __restrict__ lev_off,
    const double* __restrict__ lu9, const double2* __restrict__ fac, const double* __restrict__ dinv,
    const double* __restrict__ Rt, double* Z, const int* __restrict__ done) {
  extern __shared__ __align__(128) unsigned char smem_raw[];
  __shared__ LineBars bars;
  __shared__ int s_fail;
  volatile int* vfail = &s_fail;
  const int nx = m - 2, warps = line_warps(nx), iters = line_iters(nx), nblk = iters / kLineBlock;
  const int nb = line_bnd(nx), S = line_stride(nx);
  const int wp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const bool producer = wp >= warps;
  const int w = producer ? wp - warps : wp;
  const int a = a0 + blockIdx.x, set = fac_per_col ? a : 0;
  double2* rings = reinterpret_cast<double2*>(smem_raw);
  double* bnd = reinterpret_cast<double*>(rings + (size_t)warps * kLineRing);
  unsigned long long* done4 = reinterpret_cast<unsigned long long*>(bnd + (size_t)warps * nb);
  double* col = reinterpret_cast<double*>(done4 + (size_t)2 * warps * nblk);
  const double* rhs = Rt + (size_t)a * ldN;
  if (threadIdx.x == 0) s_fail = 0;
  for (int i = threadIdx.x; i < 2 * warps * nblk; i += blockDim.x) mbar_init(&done4[i], 1);
  for (int i = threadIdx.x; i < warps * kLineSlots; i += blockDim.x) {
    mbar_init(&bars.full[i / kLineSlots][i % kLineSlots], 1);
    mbar_init(&bars.empty[i / kLineSlots][i % kLineSlots], 1);
  }
  for (int i = threadIdx.x; i < warps * 40; i += blockDim.x) bnd[(size_t)(i / 40) * nb + iters + i % 40] = 0.0;
  asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
  asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
  __syncthreads();
  double2* ring = rings + (size_t)w * kLineRing;
  if (producer) {
    if (lane == 0) {
      // both sweeps' factors of this warp follow one another
      const double2* src = fac + ((size_t)set * warps + w) * 2 * iters * 32;
      const unsigned total = 2u * nblk;
      constexpr unsigned kBytes = 16u * kLineBlock * 32;
      unsigned u = 0;
      for (; u < total; ++u) {
        const unsigned slot = u % kLineSlots;
        if (u == kLineSlots) {  // the first slots are filled while the kernel before still runs
          pdl_wait();
          if (done != nullptr && *done) break;
        }
        if (u >= kLineSlots &&
            (*vfail || !mbar_wait_bounded(&bars.empty[w][slot], ((u / kLineSlots) - 1u) & 1u))) {
          *vfail = 1;
          break;
        }
        mbar_expect_tx(&bars.full[w][slot], kBytes);
        bulk_g2s(ring + slot * kLineBlock * 32, src + (size_t)u * kLineBlock * 32, kBytes, &bars.full[w][slot]);
      }
      // what is under way lands before the CTA ends, also when a compute warp gave up
      for (unsigned c = u > kLineSlots ? u - kLineSlots : 0; c < u; ++c)
        mbar_wait_bounded(&bars.full[w][c % kLineSlots], (c / kLineSlots) & 1u);
    }
    __syncwarp();
    pdl_wait();
    if (done != nullptr && *done) return;
    // the boundary rows: their scaling by 1/u_ii
    for (int k = w * 32 + lane; k < 4 * (m - 1); k += warps * 32) {
      const int side = k / (m - 1), s = k - side * (m - 1);
      const int x = side == 0 ? s : side == 1 ? m - 1 : side == 2 ? m - 1 - s : 0;
      const int y = side == 0 ? 0 : side == 1 ? s : side == 2 ? m - 1 : m - 1 - s;
      const int lv = x + 2 * y, ylo = max(0, (lv - (m - 1) + 1) >> 1);
      Z[(size_t)(x + m * y) * P + a] =
          rhs[x + m * y] * lu9[((size_t)set * 9 + 4) * N + lev_off[lv] + (y - ylo)];
    }
  } else {
    pdl_wait();
    if (done != nullptr && *done) return;
    const int r0 = 16 * w, nr = min(16, nx - r0);
    // the warp's lines, 16 loads a lane in flight
    for (int x = lane; x < nx; x += 32) {
      double v[16];
#pragma unroll
      for (int r = 0; r < 16; ++r) v[r] = r < nr ? rhs[(x + 1) + m * (r0 + r + 1)] : 0.0;
#pragma unroll
      for (int r = 0; r < 16; ++r)
        if (r < nr) col[(size_t)(r0 + r) * S + x] = v[r];
    }
    __syncwarp();
    double* bo = bnd + (size_t)w * nb;
    const int lo = w > 0 ? w - 1 : 0, hi = w + 1 < warps ? w + 1 : w;
    line_sweep<false>(ring, bars.full[w], bars.empty[w], 0u, col, nx, bo, bnd + (size_t)lo * nb,
                      done4 + (size_t)w * nblk, done4 + (size_t)lo * nblk, w, w == 0, vfail);
    __syncwarp();
    const double* dl = dinv + (size_t)set * nx * nx;
    for (int x = lane; x < nx; x += 32) {
      double v[16];
#pragma unroll
      for (int r = 0; r < 16; ++r) v[r] = r < nr ? dl[(size_t)(r0 + r) * nx + x] : 0.0;
#pragma unroll
      for (int r = 0; r < 16; ++r)
        if (r < nr) col[(size_t)(r0 + r) * S + x] *= v[r];
    }
    __syncwarp();
    line_sweep<true>(ring, bars.full[w], bars.empty[w], (unsigned)nblk, col, nx, bo,
                     bnd + (size_t)hi * nb, done4 + (size_t)(warps + w) * nblk,
                     done4 + (size_t)(warps + hi) * nblk, w, w == warps - 1, vfail);
    __syncwarp();
    for (int x = lane; x < nx; x += 32)
#pragma unroll
      for (int r = 0; r < 16; ++r)
        if (r < nr) Z[((size_t)(x + 1) + (size_t)m * (r0 + r + 1)) * P + a] = col[(size_t)(r0 + r) * S + x];
  }
  __syncthreads();
  if (*vfail)  // a wait gave up: no caller may take the column as a result
    for (int i = threadIdx.x; i < N; i += blockDim.x) Z[(size_t)i * P + a] = __longlong_as_double(0x7ff8000000000000ll);
}

// Factor streams and 1/u_ii by lines from the level-major slots: thread (set, warp, sweep, iteration,
// lane).
__global__ void line_factors_kernel(int m, int N, int nfac, const int* __restrict__ lev_off,
                                    const double* __restrict__ lu9, double2* __restrict__ fac,
                                    double* __restrict__ dinv) {
  const int nx = m - 2, warps = line_warps(nx), iters = line_iters(nx);
  const long long total = (long long)nfac * warps * 2 * iters * 32;
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < total;
       i += (long long)gridDim.x * blockDim.x) {
    const int lane = (int)(i & 31), l = lane & 15;
    const long long q = i >> 5;
    const int t = (int)(q % iters), up = (int)(q / iters % 2);
    const long long fw = q / iters / 2;
    const int w = (int)(fw % warps), f = (int)(fw / warps);
    const bool older = lane >= 16;
    const int line = 16 * w + (up ? 15 - l : l), xi = (older ? t : t - 1) - 2 * l;
    double2 v = make_double2(0.0, 0.0);
    if (line < nx && xi >= 0 && xi < nx) {
      const int x = up ? nx - xi : xi + 1, y = line + 1;
      const int lv = x + 2 * y, ylo = max(0, (lv - (m - 1) + 1) >> 1), pos = lev_off[lv] + (y - ylo);
      const double* lu = lu9 + (size_t)f * 9 * N + pos;
      const int s0 = older ? 0 : 3, s1 = older ? 1 : 2;
      v.x = lu[(size_t)(up ? 8 - s0 : s0) * N];
      v.y = lu[(size_t)(up ? 8 - s1 : s1) * N];
      if (!older && !up) dinv[((size_t)f * nx + line) * nx + xi] = lu[(size_t)4 * N];
    }
    fac[i] = v;
  }
}

}  // namespace

// Factor streams of an FP64 system, where a column fits in shared memory and a sixteenth of the
// device's memory holds them.
int lines_setup(System& s, cudaStream_t st) {
  const int nx = s.pat.m - 2;
  if (s.lean || nx < kLineMin || line_warps(nx) > kLineWarps || line_smem(nx) + 1024 > smem_optin_max()) return SG_OK;
  const size_t n = (size_t)s.nfac * line_warps(nx) * 2 * line_iters(nx) * 32;
  const size_t nd = (size_t)s.nfac * nx * nx, bytes = sizeof(double) * (2 * n + nd);
  size_t free_b = 0, total_b = 0;
  if (cudaMemGetInfo(&free_b, &total_b) != cudaSuccess) {
    cudaGetLastError();
    return SG_OK;
  }
  if (bytes > total_b / 16 || free_b < bytes + total_b / 2) return SG_OK;
  SG_TRY(s.line_fac.alloc(2 * n));
  SG_TRY(s.line_dinv.alloc(nd));
  const int grid = (int)std::min<size_t>((n + 255) / 256, 152 * 32);
  line_factors_kernel<<<grid, 256, 0, st>>>(s.pat.m, s.N, s.nfac, s.lev9_off.p, s.lu9.p,
                                            reinterpret_cast<double2*>(s.line_fac.p), s.line_dinv.p);
  return check_launch("line_factors");
}

// Z[:, a] = ILU_a^-1 Rt[a] for columns a0 .. a0 + ncols - 1.
int launch_lines_solve(System& s, int a0, int ncols, int fac_per_col, const double* Rt, double* Z,
                       cudaStream_t st, const int* done) {
  const int nx = s.pat.m - 2;
  size_t smem = line_smem(nx);
  // a single-column (Gauss-Seidel) solve takes a whole SM, as in the barrier kernels
  if (ncols == 1) smem = std::max(smem, smem_optin_max() - 1024);
  SG_TRY(ensure_smem((const void*)ilu_lines_kernel, smem));
  TimeScope ts(s.timer, K_ILU_SOLVE, st);
  return launch_pdl(ilu_lines_kernel, dim3(ncols), dim3(line_warps(nx) * 64), smem, st, s.pat.m, s.N, s.ldN,
                    s.P, a0, fac_per_col, s.lev9_off.p, s.lu9.p,
                    reinterpret_cast<const double2*>(s.line_fac.p), s.line_dinv.p, Rt, Z, done);
}

}  // namespace sg
