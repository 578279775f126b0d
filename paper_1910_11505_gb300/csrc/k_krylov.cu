// Krylov kernels of restarted GMRES (Sec. 3) on the device: classical Gram-Schmidt applied twice
// (CGS2) with deterministic two-level reductions, the Givens least-squares update, the
// back-substitution and the solution update.  Every kernel of one Arnoldi step reads the
// system's ``done`` flag first and returns at once when the cycle has already converged, so a
// whole cycle can be queued without a host round trip.
//
// Reductions: each CTA writes its partial sums, the last CTA to arrive (atomic ticket) adds the
// partials in a fixed order, one warp per sum, and resets the ticket, so results are bitwise
// reproducible.
//
// Vectors of at most kStepMax entries take the whole step (dots, update, dots, update, norm,
// Givens, scaling) in one kernel on one thread-block cluster (arnoldi_cluster_kernel): the four
// kernels' launches and grid-wide reductions took 115 us a step at n = 1734, of which the data's
// share is below 1 us.  Longer ones need more than a cluster's bandwidth.
#include <algorithm>
#include <map>
#include <mutex>

#include "sg_internal.h"

namespace sg {

constexpr int kRedBlocks = 304;   // 2 CTAs per SM on 152 SMs
constexpr int kRedThreads = 256;
constexpr int kMaxBasis = 1025;   // restart <= 1024 -> at most 1025 basis vectors
constexpr int kLT = 8;            // basis vectors per register tile

namespace {

__device__ __forceinline__ double block_sum(double v, double* sh) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  int w = threadIdx.x >> 5, l = threadIdx.x & 31;
  __syncthreads();
  if (l == 0) sh[w] = v;
  __syncthreads();
  double s = 0.0;
  if (threadIdx.x == 0)
    for (int i = 0; i < (int)(blockDim.x >> 5); ++i) s += sh[i];
  return s;  // valid in thread 0
}

__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// Sums over the warp of kLT values per lane by a transposing butterfly: lane t receives the sum of
// value warp_slot(t).  Nine additions instead of forty: an FP64 instruction of a warp holds its
// sub-partition for some sixty cycles on this GPU, so the reductions' count is what costs.
__device__ __forceinline__ int warp_slot(int lane) { return (lane >> 2 & 4) | (lane >> 2 & 2) | (lane >> 2 & 1); }
__device__ __forceinline__ double warp_sums(double (&a)[8]) {
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int h = 4, o = 16; h >= 1; h >>= 1, o >>= 1) {
    const bool up = lane & o;
#pragma unroll
    for (int q = 0; q < h; ++q) {
      const double keep = up ? a[q + h] : a[q], send = up ? a[q] : a[q + h];
      a[q] = keep + __shfl_xor_sync(0xffffffffu, send, o);
    }
  }
  a[0] += __shfl_xor_sync(0xffffffffu, a[0], 2);
  a[0] += __shfl_xor_sync(0xffffffffu, a[0], 1);
  return a[0];
}

// Partial dot products of w with basis vectors [0, nv) for this CTA's grid-stride slice;
// partial[l * kRedBlocks + CTA].
__device__ void partial_dots(size_t n, const double* __restrict__ V, int nv,
                             const double* __restrict__ w, double* __restrict__ partial,
                             double (*sh)[kLT]) {
  const int wp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  for (int l0 = 0; l0 < nv; l0 += kLT) {
    double acc[kLT];
#pragma unroll
    for (int q = 0; q < kLT; ++q) acc[q] = 0.0;
    int lc = min(kLT, nv - l0);
    for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
         i += (size_t)gridDim.x * blockDim.x) {
      double wi = w[i];
#pragma unroll
      for (int q = 0; q < kLT; ++q)
        if (q < lc) acc[q] = fma(V[(size_t)(l0 + q) * n + i], wi, acc[q]);
    }
    const double t = warp_sums(acc);
    if ((lane & 3) == 0) sh[wp][warp_slot(lane)] = t;
    __syncthreads();
    if ((int)threadIdx.x < lc) {
      double s = 0.0;
      for (int i = 0; i < kRedThreads / 32; ++i) s += sh[i][threadIdx.x];
      partial[(size_t)(l0 + threadIdx.x) * kRedBlocks + blockIdx.x] = s;
    }
    __syncthreads();
  }
}

// Returns true in every thread of the CTA that arrives last.
__device__ bool arrive_last(unsigned int* ticket) {
  __shared__ bool last;
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) last = (atomicAdd(ticket, 1u) == gridDim.x - 1);
  __syncthreads();
  return last;
}

// Sum of the CTAs' partials of one value by one warp, in a fixed order.
__device__ __forceinline__ double sum_partials(const double* p) {
  double s = 0.0;
#pragma unroll 4
  for (int b = threadIdx.x & 31; b < (int)gridDim.x; b += 32) s += __ldcg(p + b);
  return warp_sum(s);
}

__device__ void finish_sums(const double* partial, int nv, double* out, unsigned int* ticket) {
  __threadfence();
  for (int l = threadIdx.x >> 5; l < nv; l += kRedThreads / 32) {
    const double s = sum_partials(partial + (size_t)l * kRedBlocks);
    if ((threadIdx.x & 31) == 0) out[l] = s;
  }
  if (threadIdx.x == 0) *ticket = 0u;
}

// Givens step of column j = nv - 1 by one warp, in two parts.  First the previous rotations: col
// (j + 1 entries, h1 + h2) and the rotations staged in shared memory, cn scratch of j + 1 entries;
// the rotated column goes to Hcol, its last entry is returned (in every lane).  Only the chain over
// the rotations is serial, one multiply-add each.
__device__ double givens_chain(int j, const double* col, double* cn, const double* c_s,
                               const double* s_s, double* __restrict__ Hcol) {
  const int lane = threadIdx.x & 31;
  for (int i = lane; i < j; i += 32) cn[i] = c_s[i] * col[i + 1];
  __syncwarp();
  double cur = col[0];  // every lane runs the chain (one instruction for the warp)
  for (int i = 0; i < j; ++i) {
    const double v = cur;
    cur = fma(-s_s[i], cur, cn[i]);
    __syncwarp();
    if (lane == 0) cn[i] = v;
  }
  __syncwarp();
  for (int i = lane; i < j; i += 32) Hcol[i] = c_s[i] * cn[i] + s_s[i] * col[i + 1];
  return cur;
}

// Then the new rotation from the column's last entry and hn = ||w||: to cs, sn, g and Hcol;
// state[3] = 1 / h_{j+1,j}; flags: [0] done, [1] columns in this cycle, [2] status.  The three
// quotients are one division, on three lanes.
__device__ void givens_finish(int j, double cur, double hn, double* __restrict__ Hcol,
                              double* __restrict__ cs, double* __restrict__ sn,
                              double* __restrict__ g, double* __restrict__ state,
                              int* __restrict__ flags, int last_col) {
  const int lane = threadIdx.x & 31;
  const double den = hypot(cur, hn);
  const bool bad = !isfinite(den) || !isfinite(hn);
  const double q = (lane == 0 ? cur : lane == 1 ? hn : 1.0) / (lane < 2 ? den : hn);
  const double q1 = __shfl_sync(0xffffffffu, q, 1), q2 = __shfl_sync(0xffffffffu, q, 2);
  if (lane != 0) return;
  if (bad) {
    flags[2] = SG_ERR_NAN;
    flags[0] = 1;
    return;
  }
  const double c = den > 0.0 ? q : 1.0;
  const double sgn = den > 0.0 ? q1 : 0.0;
  cs[j] = c;
  sn[j] = sgn;
  Hcol[j] = den;
  const double gj = g[j], gn = -sgn * gj;
  g[j + 1] = gn;
  g[j] = c * gj;
  flags[1] = j + 1;
  state[3] = hn > 0.0 ? q2 : 0.0;
  if (fabs(gn) <= state[0] || hn == 0.0 || den == 0.0 || j == last_col) flags[0] = 1;
}

// h = V[0:nv]^T w; with ``w32`` w is first set to its FP64 values
__global__ void __launch_bounds__(kRedThreads) cgs_dots_kernel(
    size_t n, const double* __restrict__ V, int nv, double* __restrict__ w,
    const float* __restrict__ w32, double* __restrict__ partial, unsigned int* ticket,
    double* __restrict__ h, const int* __restrict__ done) {
  pdl_trigger();
  pdl_wait();
  if (*done) return;
  __shared__ double sh[kRedThreads / 32][kLT];
  if (w32 != nullptr)
    for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
         i += (size_t)gridDim.x * blockDim.x)
      w[i] = (double)w32[i];
  // each thread re-reads only the entries it wrote itself
  partial_dots(n, V, nv, w, partial, sh);
  if (arrive_last(ticket)) finish_sums(partial, nv, h, ticket);
}

// w -= V[0:nv] h1, then h2 = V[0:nv]^T w
__global__ void __launch_bounds__(kRedThreads) cgs_update_dots_kernel(
    size_t n, const double* __restrict__ V, int nv, double* __restrict__ w,
    const double* __restrict__ h1, double* __restrict__ partial, unsigned int* ticket,
    double* __restrict__ h2, const int* __restrict__ done) {
  pdl_trigger();
  pdl_wait();
  if (*done) return;
  __shared__ double sh[kRedThreads / 32][kLT];
  __shared__ double hs[kMaxBasis];
  for (int l = threadIdx.x; l < nv; l += blockDim.x) hs[l] = h1[l];
  __syncthreads();
  for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
       i += (size_t)gridDim.x * blockDim.x) {
    double v = w[i];
    for (int l = 0; l < nv; ++l) v = fma(-V[(size_t)l * n + i], hs[l], v);
    w[i] = v;
  }
  // each thread re-reads only the entries it wrote itself
  partial_dots(n, V, nv, w, partial, sh);
  if (arrive_last(ticket)) finish_sums(partial, nv, h2, ticket);
}

// w -= V[0:nv] h2; column j = nv-1 of the Hessenberg matrix is h1 + h2 and ||w||; the last CTA
// applies the previous Givens rotations to it, makes the new one, updates g and the flags.
// state: [0] target (absolute), [1] beta, [2] ||F||, [3] 1/h_{j+1,j}
// flags: [0] done, [1] columns in this cycle, [2] status
__global__ void __launch_bounds__(kRedThreads) cgs_update_norm_kernel(
    size_t n, const double* __restrict__ V, int nv, double* __restrict__ w,
    const double* __restrict__ h1, const double* __restrict__ h2, double* __restrict__ partial,
    unsigned int* ticket, double* __restrict__ Hs, int ldh, double* __restrict__ cs,
    double* __restrict__ sn, double* __restrict__ g, double* __restrict__ state,
    int* __restrict__ flags, int last_col) {
  pdl_trigger();
  pdl_wait();
  if (flags[0]) return;
  __shared__ double sh[32];
  __shared__ double hs[kMaxBasis], c_s[kMaxBasis], s_s[kMaxBasis], cn[kMaxBasis];
  for (int l = threadIdx.x; l < nv; l += blockDim.x) hs[l] = h2[l];
  __syncthreads();
  double acc = 0.0;
  for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
       i += (size_t)gridDim.x * blockDim.x) {
    double v = w[i];
    for (int l = 0; l < nv; ++l) v = fma(-V[(size_t)l * n + i], hs[l], v);
    w[i] = v;
    acc = fma(v, v, acc);
  }
  double s = block_sum(acc, sh);
  if (threadIdx.x == 0) partial[blockIdx.x] = s;
  if (!arrive_last(ticket)) return;
  __threadfence();
  const int j = nv - 1;
  for (int l = threadIdx.x; l <= j; l += blockDim.x) {
    hs[l] += __ldcg(h1 + l);
    if (l < j) {
      c_s[l] = cs[l];
      s_s[l] = sn[l];
    }
  }
  __syncthreads();
  if (threadIdx.x >= 32) return;
  const double ss = sum_partials(partial);
  if (threadIdx.x == 0) *ticket = 0u;
  double* Hcol = Hs + (size_t)j * ldh;
  const double cur = givens_chain(j, hs, cn, c_s, s_s, Hcol);
  givens_finish(j, cur, sqrt(ss), Hcol, cs, sn, g, state, flags, last_col);
}

// A whole Arnoldi step of a short vector on one cluster: CTA r holds a contiguous slice of w in
// shared memory; a warp forms eight dots over a share of the slice, the shares' sums are added in
// order, then over the CTAs through distributed shared memory in rank order (every CTA forms the
// same sums), with a cluster barrier per reduction.  CTA 0's first warp makes the Givens step.
//
// Bound: latency and the FP64 pipe.  The basis slices are copied into shared memory once where they
// fit (four passes read them), the previous rotations are applied while the other warps form the
// norm.  An FP64 instruction takes 65 cycles of its sub-partition whatever its
// lanes, so a slice is cut into shares only while sub-partitions are idle (a share costs its
// reduction), scalars (the norm, its root and reciprocal) are formed by one warp, and the cluster
// has 16 CTAs where the device schedules that (non-portable) size, else 8.
constexpr int kStepThreads = 256;
constexpr size_t kStepMax = 32768;  // entries: at most 32 KB of w per CTA
constexpr size_t kStepStage = 160 * 1024;  // shared memory a CTA may take

__device__ __forceinline__ void cluster_sync() {
  asm volatile("barrier.cluster.arrive.release.aligned;\n"
               "barrier.cluster.wait.acquire.aligned;\n" ::: "memory");
}
__device__ __forceinline__ double ld_cluster(const double* p, unsigned rank) {
  unsigned a;
  double v;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : "r"(smem_u32(p)), "r"(rank));
  asm volatile("ld.shared::cluster.f64 %0, [%1];" : "=d"(v) : "r"(a) : "memory");
  return v;
}

__host__ __device__ constexpr int step_sums(int nv) { return nv + kLT > 4 * kLT ? nv + kLT : 4 * kLT; }

__global__ void __launch_bounds__(kStepThreads)
    arnoldi_cluster_kernel(int n, const double* __restrict__ V, int nv, double* __restrict__ w,
                           const float* __restrict__ w32, double* __restrict__ Hs, int ldh,
                           double* __restrict__ cs, double* __restrict__ sn, double* __restrict__ g,
                           double* __restrict__ state, int* __restrict__ flags, int last_col,
                           float* __restrict__ v32, int stage) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  double* ws = reinterpret_cast<double*>(smem_raw);   // the slice
  const int ctas = gridDim.x;  // one cluster
  const int chunk = (n + ctas - 1) / ctas;
  double* hp0 = ws + chunk;      // this CTA's partial sums (two buffers, and the norm's)
  double* hp1 = hp0 + nv;
  double* h1 = hp1 + nv + 1;     // h1, then h1 + h2
  double* h2 = h1 + nv;
  double* c_s = h2 + nv;
  double* s_s = c_s + nv;
  double* sums = s_s + nv;       // shares' sums (step_sums entries), then the Givens scratch
  __shared__ double red[32], scal[2];
  __shared__ int skip;
  pdl_trigger();
  pdl_wait();
  if (threadIdx.x == 0) skip = flags[0];
  // (the flag changes only in this kernel's last phase, after a cluster barrier)
  __syncthreads();
  if (skip) return;
  const int rank = blockIdx.x;
  const int i0 = rank * chunk, len = max(0, min(chunk, n - i0));
  const int wp = threadIdx.x >> 5, lane = threadIdx.x & 31, nw = kStepThreads / 32;
  const int j = nv - 1;
  // basis slices: vector l at Vp + l ldv
  const double* Vp = V + i0;
  size_t ldv = n;
  if (stage) {
    double* vs = sums + step_sums(nv);
    for (int l = wp; l < nv; l += nw)
      for (int i = lane; i < len; i += 32)
        asm volatile("cp.async.ca.shared.global [%0], [%1], 8;\n" ::"r"(smem_u32(vs + (size_t)l * chunk + i)),
                     "l"(V + (size_t)l * n + i0 + i)
                     : "memory");
    Vp = vs;
    ldv = chunk;
  }
  for (int i = threadIdx.x; i < len; i += kStepThreads) ws[i] = w32 ? (double)w32[i0 + i] : w[i0 + i];
  for (int l = threadIdx.x; l < j; l += kStepThreads) {
    c_s[l] = cs[l];
    s_s[l] = sn[l];
  }
  asm volatile("cp.async.wait_all;\n" ::: "memory");
  __syncthreads();
  auto dots = [&](double* hp, double* h) {
    const int groups = (nv + kLT - 1) / kLT, shares = max(1, 4 / groups);
    for (int it = wp; it < groups * shares; it += nw) {
      const int l0 = it / shares * kLT, p = it % shares;
      const double* v = Vp + (size_t)l0 * ldv;
      const int lc = min(kLT, nv - l0);
      double acc[kLT];
#pragma unroll
      for (int q = 0; q < kLT; ++q) acc[q] = 0.0;
#pragma unroll 2
      for (int i = 32 * p + lane; i < len; i += 32 * shares) {
        const double wi = ws[i];
#pragma unroll
        for (int q = 0; q < kLT; ++q)
          if (q < lc) acc[q] = fma(v[(size_t)q * ldv + i], wi, acc[q]);
      }
      const double t = warp_sums(acc);
      if ((lane & 3) == 0) sums[p * groups * kLT + l0 + warp_slot(lane)] = t;
    }
    __syncthreads();
    for (int l = threadIdx.x; l < nv; l += kStepThreads) {
      double s = 0.0;
      for (int p = 0; p < shares; ++p) s += sums[p * groups * kLT + l];
      hp[l] = s;
    }
    cluster_sync();
    for (int l = threadIdx.x; l < nv; l += kStepThreads) {
      double v[16], s = 0.0;
#pragma unroll
      for (int r = 0; r < 16; ++r) v[r] = r < ctas ? ld_cluster(hp + l, r) : 0.0;
      for (int r = 0; r < ctas; r += 8)
        s += ((v[r] + v[r + 1]) + (v[r + 2] + v[r + 3])) + ((v[r + 4] + v[r + 5]) + (v[r + 6] + v[r + 7]));
      h[l] = s;
    }
    __syncthreads();
  };
  auto update = [&](const double* h, int threads) {
    double acc = 0.0;
    for (int i = threadIdx.x; i < len; i += threads) {
      double v = ws[i];
#pragma unroll 8
      for (int l = 0; l < nv; ++l) v = fma(-Vp[(size_t)l * ldv + i], h[l], v);
      ws[i] = v;
      acc = fma(v, v, acc);
    }
    return acc;
  };
  dots(hp0, h1);
  update(h1, kStepThreads);
  __syncthreads();
  dots(hp1, h2);
  // the last warp takes no part in this update: in CTA 0 it applies the previous rotations
  double acc = 0.0, cur = 0.0;
  double* Hcol = Hs + (size_t)j * ldh;
  if (wp < nw - 1) {
    acc = update(h2, kStepThreads - 32);
  } else if (rank == 0) {
    for (int l = lane; l < nv; l += 32) h1[l] += h2[l];
    __syncwarp();
    cur = givens_chain(j, h1, sums, c_s, s_s, Hcol);
  }
  const double part = block_sum(acc, red);
  if (threadIdx.x == 0) hp1[nv] = part;  // (hp1[0 .. nv) may still be read by other CTAs)
  cluster_sync();
  if (wp == 0) {
    double ss = lane < ctas ? ld_cluster(hp1 + nv, lane) : 0.0;
    for (int o = 8; o > 0; o >>= 1) ss += __shfl_xor_sync(0xffffffffu, ss, o);
    const double hn = sqrt(ss);
    if (lane == 0) {
      scal[0] = hn;
      scal[1] = hn > 0.0 ? 1.0 / hn : 0.0;
    }
  }
  __syncthreads();
  const double sc = scal[1];
  for (int i = threadIdx.x; i < len; i += kStepThreads) {
    const double v = ws[i] * sc;
    w[i0 + i] = v;
    if (v32 != nullptr) v32[i0 + i] = (float)v;
  }
  if (rank == 0 && wp == nw - 1)
    givens_finish(j, cur, scal[0], Hcol, cs, sn, g, state, flags, last_col);
  cluster_sync();  // no CTA's shared memory goes while another may read it
}

size_t step_smem(size_t n, int nv, int ctas) {
  return sizeof(double) * ((n + ctas - 1) / ctas + 6 * (size_t)nv + 1 + step_sums(nv));
}

// CTAs of the cluster: 16 (a non-portable size) where the device can schedule it, else 8; asked
// once per device.
int step_ctas() {
  static std::mutex mu;
  static std::map<int, int> known;
  int dev = 0;
  cudaGetDevice(&dev);
  std::lock_guard<std::mutex> lock(mu);
  auto it = known.find(dev);
  if (it != known.end()) return it->second;
  int ctas = 8;
  auto kern = arnoldi_cluster_kernel;
  static_assert(kStepStage >= sizeof(double) * (kStepMax / 8 + 7 * kMaxBasis + kLT + 1), "shared memory of a step");
  if (cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) == cudaSuccess &&
      ensure_smem((const void*)kern, kStepStage) == SG_OK) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(16, 1, 1);
    cfg.blockDim = dim3(kStepThreads, 1, 1);
    cfg.dynamicSmemBytes = kStepStage;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = 16;
    attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    int n = 0;
    if (cudaOccupancyMaxActiveClusters(&n, kern, &cfg) == cudaSuccess && n >= 2) ctas = 16;
  }
  cudaGetLastError();
  known[dev] = ctas;
  return ctas;
}

// v *= state[3]  (normalise the new basis vector)
// with ``v32`` also its FP32 copy, the next step's preconditioner operand
__global__ void scale_kernel(size_t n, double* __restrict__ v, float* __restrict__ v32,
                             const double* __restrict__ state, const int* __restrict__ flags) {
  pdl_trigger();
  pdl_wait();
  if (flags[0]) return;
  double sc = state[3];
  for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
       i += (size_t)gridDim.x * blockDim.x) {
    const double x = v[i] * sc;
    v[i] = x;
    if (v32 != nullptr) v32[i] = (float)x;
  }
}

// ||r||_2 -> out
__global__ void __launch_bounds__(kRedThreads) norm_kernel(size_t n, const double* __restrict__ r,
                                                           double* __restrict__ partial,
                                                           unsigned int* ticket,
                                                           double* __restrict__ out) {
  __shared__ double sh[32];
  double acc = 0.0;
  for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
       i += (size_t)gridDim.x * blockDim.x)
    acc = fma(r[i], r[i], acc);
  double s = block_sum(acc, sh);
  if (threadIdx.x == 0) partial[blockIdx.x] = s;
  if (!arrive_last(ticket)) return;
  __threadfence();
  if (threadIdx.x >= 32) return;
  const double ss = sum_partials(partial);
  if (threadIdx.x != 0) return;
  *ticket = 0u;
  *out = sqrt(ss);
}

// Start of a cycle: V0 = r / beta (and its FP32 copy), g = (beta, 0, ...), flags cleared.
__global__ void init_cycle_kernel(size_t n, const double* __restrict__ r, double* __restrict__ V0,
                                  float* __restrict__ v32, const double* __restrict__ state, double* __restrict__ g,
                                  int glen, int* __restrict__ flags) {
  double beta = state[1];
  double inv = beta > 0.0 ? 1.0 / beta : 0.0;
  for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
       i += (size_t)gridDim.x * blockDim.x) {
    const double v = r[i] * inv;
    V0[i] = v;
    if (v32 != nullptr) v32[i] = (float)v;
  }
  if (blockIdx.x == 0)
    for (int i = threadIdx.x; i < glen; i += blockDim.x) g[i] = i == 0 ? beta : 0.0;
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    flags[0] = 0;
    flags[1] = 0;
  }
}

// y = H(0:k,0:k)^{-1} g(0:k), k = flags[1]: column-oriented back substitution by one CTA; after y_i
// is known H(l,i) y_i is removed from the right-hand-side entries l < i.  Up to kBackWarp columns
// one warp does it with four entries per lane, the matrix staged in shared memory by the CTA (the
// CTA-wide form below takes two barriers and a trip to L2 per column: 40 us at k = 43).
constexpr int kBackWarp = 128;

__global__ void __launch_bounds__(1024) backsolve_kernel(const double* __restrict__ Hs, int ldh,
                                                         const double* __restrict__ g,
                                                         double* __restrict__ y,
                                                         const int* __restrict__ flags) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int k = flags[1];
  if (k <= kBackWarp) {
    double* H = reinterpret_cast<double*>(smem_raw);  // column i at i * kBackWarp
    for (int t = threadIdx.x; t < k * kBackWarp; t += blockDim.x) {
      const int i = t / kBackWarp, l = t & (kBackWarp - 1);
      if (l <= i) H[t] = Hs[(size_t)i * ldh + l];
    }
    __syncthreads();
    if (threadIdx.x >= 32) return;
    const int lane = threadIdx.x;
    double r[kBackWarp / 32];
#pragma unroll
    for (int q = 0; q < kBackWarp / 32; ++q) r[q] = lane + 32 * q < k ? g[lane + 32 * q] : 0.0;
#pragma unroll
    for (int q = kBackWarp / 32 - 1; q >= 0; --q)
      for (int i = min(k - 1, 32 * q + 31); i >= 32 * q; --i) {
        const double* col = H + (size_t)i * kBackWarp;
        const double yi = __shfl_sync(0xffffffffu, r[q], i & 31) / col[i];
        if (lane == (i & 31)) y[i] = yi;
#pragma unroll
        for (int p = 0; p <= q; ++p)
          if (lane + 32 * p < i) r[p] -= col[lane + 32 * p] * yi;
      }
    return;
  }
  __shared__ double rhs[kMaxBasis];
  __shared__ double yi;
  for (int l = threadIdx.x; l < k; l += blockDim.x) rhs[l] = g[l];
  __syncthreads();
  for (int i = k - 1; i >= 0; --i) {
    const double* col = Hs + (size_t)i * ldh;
    if (threadIdx.x == 0) {
      yi = rhs[i] / col[i];
      y[i] = yi;
    }
    __syncthreads();
    const double v = yi;
    for (int l = threadIdx.x; l < i; l += blockDim.x) rhs[l] -= col[l] * v;
    __syncthreads();
  }
}

// x += sum_{l < k} Z_l y_l  (Z rows FP64 or FP32)
template <typename TZ>
__global__ void update_x_kernel(size_t n, const TZ* __restrict__ Z, const double* __restrict__ y,
                                const int* __restrict__ flags, double* __restrict__ x) {
  __shared__ double ys[kMaxBasis];
  int k = flags[1];
  for (int l = threadIdx.x; l < k; l += blockDim.x) ys[l] = y[l];
  __syncthreads();
  for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
       i += (size_t)gridDim.x * blockDim.x) {
    double v = x[i];
    for (int l = 0; l < k; ++l) v = fma((double)Z[(size_t)l * n + i], ys[l], v);
    x[i] = v;
  }
}

// *flag = 0 if any of x[0..n) is nonzero (the caller sets it nonzero beforehand).
__global__ void any_nonzero_kernel(size_t n, const double* __restrict__ x, int* __restrict__ flag) {
  bool nz = false;
  for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < n && !nz;
       i += (size_t)gridDim.x * blockDim.x)
    nz = x[i] != 0.0;
  if (__syncthreads_or(nz) && threadIdx.x == 0) *flag = 0;
}

}  // namespace

// ------------------------------------------------------------------ launchers used by the driver

int k_zero_flag(System& s, size_t n, const double* x, int* flag, cudaStream_t st) {
  TimeScope ts(s.timer, K_OTHER, st);
  SG_CUDA(cudaMemsetAsync(flag, 1, sizeof(int), st));
  any_nonzero_kernel<<<kRedBlocks, kRedThreads, 0, st>>>(n, x, flag);
  return check_launch("any_nonzero");
}

// CTAs of a reduction over n entries: two entries per thread at least.
static int red_grid(size_t n) {
  return (int)std::max<size_t>(1, std::min<size_t>(kRedBlocks, (n + 2 * kRedThreads - 1) / (2 * kRedThreads)));
}

int k_norm(System& s, size_t n, const double* r, double* out, cudaStream_t st) {
  TimeScope ts(s.timer, K_OTHER, st);
  norm_kernel<<<red_grid(n), kRedThreads, 0, st>>>(n, r, s.red.p, s.ticket.p, out);
  return check_launch("norm");
}

int k_init_cycle(System& s, size_t n, const double* r, cudaStream_t st) {
  TimeScope ts(s.timer, K_OTHER, st);
  init_cycle_kernel<<<kRedBlocks, kRedThreads, 0, st>>>(n, r, s.V.p, s.mv32a.p, s.scal.p, s.g.p,
                                                        s.m + 1, s.flags.p);
  return check_launch("init_cycle");
}

// CGS2 on the new vector V[j+1] against V[0..j], Givens update, normalisation.  ``w32``: the new
// vector in FP32 (mixed precision), else it is in V[j+1].  In mixed precision the normalised
// vector's FP32 copy is left in mv32a.
int k_arnoldi(System& s, size_t n, int j, int last_col, const float* w32, cudaStream_t st) {
  int nv = j + 1;
  double* w = s.V.p + (size_t)(j + 1) * n;
  double* h1 = s.y.p + kMaxBasis;       // scratch: two h vectors after y
  double* h2 = s.y.p + 2 * kMaxBasis;
  if (n <= kStepMax) {
    const int ctas = step_ctas();
    const size_t head = step_smem(n, nv, ctas), slices = sizeof(double) * nv * ((n + ctas - 1) / ctas);
    const int stage = head + slices <= kStepStage;
    SG_TRY(ensure_smem((const void*)arnoldi_cluster_kernel, kStepStage));
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)ctas, 1, 1);
    cfg.blockDim = dim3(kStepThreads, 1, 1);
    cfg.dynamicSmemBytes = stage ? head + slices : head;
    cfg.stream = st;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = (unsigned)ctas;
    attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
    attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 2;
    TimeScope ts(s.timer, K_ARNOLDI, st);
    SG_CUDA(cudaLaunchKernelEx(&cfg, arnoldi_cluster_kernel, (int)n, (const double*)s.V.p, nv, w, w32,
                               s.Hs.p, s.m + 1, s.cs.p, s.sn.p, s.g.p, s.scal.p, s.flags.p, last_col,
                               s.mv32a.p, stage));
    return check_launch("arnoldi_cluster");
  }
  const int grid = red_grid(n);
  {
    TimeScope ts(s.timer, K_ARNOLDI, st);
    SG_TRY(launch_pdl(cgs_dots_kernel, dim3(grid), dim3(kRedThreads), 0, st, n, (const double*)s.V.p, nv,
                      w, w32, s.red.p, s.ticket.p, h1, (const int*)s.flags.p));
  }
  {
    TimeScope ts(s.timer, K_ARNOLDI, st);
    SG_TRY(launch_pdl(cgs_update_dots_kernel, dim3(grid), dim3(kRedThreads), 0, st, n,
                      (const double*)s.V.p, nv, w, (const double*)h1, s.red.p, s.ticket.p, h2,
                      (const int*)s.flags.p));
  }
  {
    TimeScope ts(s.timer, K_ARNOLDI, st);
    SG_TRY(launch_pdl(cgs_update_norm_kernel, dim3(grid), dim3(kRedThreads), 0, st, n,
                      (const double*)s.V.p, nv, w, (const double*)h1, (const double*)h2, s.red.p,
                      s.ticket.p, s.Hs.p, s.m + 1, s.cs.p, s.sn.p, s.g.p, s.scal.p, s.flags.p, last_col));
  }
  {
    TimeScope ts(s.timer, K_ARNOLDI, st);
    return launch_pdl(scale_kernel, dim3(kRedBlocks), dim3(kRedThreads), 0, st, n, w, s.mv32a.p,
                      (const double*)s.scal.p, (const int*)s.flags.p);
  }
}

int k_finish_cycle(System& s, size_t n, double* x, bool z32, cudaStream_t st) {
  TimeScope ts(s.timer, K_OTHER, st);
  const size_t smem = sizeof(double) * kBackWarp * kBackWarp;
  SG_TRY(ensure_smem((const void*)backsolve_kernel, smem));
  backsolve_kernel<<<1, 1024, smem, st>>>(s.Hs.p, s.m + 1, s.g.p, s.y.p, s.flags.p);
  SG_TRY(check_launch("backsolve"));
  if (z32)
    update_x_kernel<float><<<kRedBlocks * 2, kRedThreads, 0, st>>>(n, s.Z32.p, s.y.p, s.flags.p, x);
  else
    update_x_kernel<double><<<kRedBlocks * 2, kRedThreads, 0, st>>>(n, s.Z.p, s.y.p, s.flags.p, x);
  return check_launch("update_x");
}

int krylov_red_blocks() { return kRedBlocks; }
int krylov_max_basis() { return kMaxBasis; }

}  // namespace sg
