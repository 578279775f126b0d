// The SG operator Y = sum_k A_k X G_k^T (Eqs. stochastic_matrix and K_matrix), block-stencil form:
// the P x P blocks K_ij = sum_k G_k A_k[i,j] of K are assembled once at setup and streamed.
//
// Why.  The sparse form (k_apply_tile.cuh) does 9 U + nnz_G multiply-adds per node through shared
// memory and is bound by instruction issue (FP32) or by the FP64 pipe.  K is symmetric in the
// fields and, the stiffness matrices being symmetric, K_ji = K_ij between the nodes.  With
//   S_i = sum_j K_ij,   Y_i = S_i x_i + sum_{j != i} K_ij (x_j - x_i),
// the product K_ij (x_j - x_i) of an edge {i, j} serves both of its nodes with opposite signs, so
// a node needs five blocks: S_i and the edges to its E, NW, N and NE neighbours.  That is
// 5 P^2 multiply-adds and 5 P (P + 1) / 2 values per node (P = 84: 35 k against 115 k, in FP32
// 71 KB; P = 35: 6.1 k against 20.5 k).  The differences of a smooth x carry no cancellation, as in
// the difference form of the row-tiled kernel.
//
// Work item: 32 consecutive nodes (one per lane) x one of the five blocks.  Nodes are taken in the
// natural numbering without regard to line ends (the two boundary nodes of a line have zero
// blocks), so a neighbour is a fixed offset and the X rows of an item are two contiguous ranges.
// The fields are cut into nb ranges of TS; block (A, B), A < B, is a tile of TS x TS values x 32
// nodes that two warps read from shared memory, warp A for f_A += K_AB d_B and warp B for
// f_B += K_AB^T d_A; a diagonal tile holds its upper triangle.  Warp w keeps f of range w in
// registers over the whole item.  The tiles come in rounds of a round-robin schedule in which
// every warp takes part in one tile (circle method), fetched by a producer warp through a ring of
// bulk copies (cp.async.bulk) with a full and an empty mbarrier per slot, so warps wait only for
// the tiles that they need.  A second kernel adds the five products of every node in a fixed
// order (the results do not depend on scheduling).
//
// Bound: HBM in FP32 (tiles read once), the FP64 pipe in FP64.  Measured on one GB300 against the
// row-tiled kernel: n = 256, P = 84 FP32 0.75 ms (5.0 GB of tiles, 6.7 TB/s) against 2.04 ms, FP64
// 4.25 ms (2.3 G multiply-adds, 1.09 TFLOP/s) against 19.3 ms; n = 128, P = 35 FP64 0.206 ms
// against 0.917 ms.  The tiles take 2.2 times the row-tiled stack's memory at P = 84, L = 924.
//
// Every wait is bounded: after kWaitLimit polls the CTA raises the error word, stops waiting,
// lets its copies in flight land (bounded) and writes NaN.  A warp whose wait was given up does not
// arrive on the empty barriers: it runs ahead of the others, and two arrivals of a diagonal tile on a
// barrier that waits for one are undefined.
#include <algorithm>

#include "sg_internal.h"

namespace sg {

namespace {

constexpr int kBR = 32;        // nodes per item
constexpr int kBLd = kBR + 1;  // row stride of the staged differences (no bank conflicts)
constexpr int kBlockEdges = 5;
constexpr int kBlockMaxWarps = 31;  // one range of fields each, plus the producer warp

struct BlockArgs {
  int N, m, P, nb, rounds, ntile, ntiles_row, slots;
  long long item_elems;
  int evict_first;
  int fail;  // tests: start as if a wait had given up
};

template <typename T>
__device__ __forceinline__ T block_nan();
template <>
__device__ __forceinline__ double block_nan<double>() { return __longlong_as_double(0x7ff8000000000000LL); }
template <>
__device__ __forceinline__ float block_nan<float>() { return __int_as_float(0x7fc00000); }

__device__ __forceinline__ void mbar_arrive_n(unsigned long long* bar, unsigned n) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0], %1;\n" ::"r"(smem_u32(bar)), "r"(n) : "memory");
}

// Bulk copy whose lines are the first to leave L2 (values read once per application).
__device__ __forceinline__ void bulk_g2s_stream(void* dst, const void* src, unsigned bytes,
                                                unsigned long long* bar) {
  asm volatile(
      "{\n\t.reg .b64 pol;\n\t"
      "createpolicy.fractional.L2::evict_first.b64 pol, 1.0;\n\t"
      "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint [%0], [%1], "
      "%2, [%3], pol;\n\t}\n" ::"r"(smem_u32(dst)),
      "l"(src), "r"(bytes), "r"(smem_u32(bar))
      : "memory");
}

// Node offset of the neighbour of edge block e: S, E, NW, N, NE.
__host__ __device__ __forceinline__ int block_off(int e, int m) {
  return e == 0 ? 0 : e == 1 ? 1 : m + e - 3;
}

// F[e][i][a]: f of edge block e at node i (S_i x_i for e = 0).  Table entry of (round, warp):
// tile | partner << 16 | kind << 24 (0: rows of the tile, 1: columns, 2: diagonal); tkind: 1 for
// diagonal tiles, in the order of the item's tiles.
template <typename T, int TS>
__global__ void __launch_bounds__((kBlockMaxWarps + 1) * 32) block_edge_kernel(
    BlockArgs g, const int* __restrict__ table, const int* __restrict__ tkind,
    const T* __restrict__ K, const T* __restrict__ X, T* __restrict__ F,
    const int* __restrict__ done, int* __restrict__ err) {
  constexpr int kPair = TS * TS, kDiag = TS * (TS + 1) / 2;
  constexpr unsigned kSlot = kPair * kBR * sizeof(T);
  extern __shared__ __align__(128) unsigned char smem_raw[];
  T* ring = reinterpret_cast<T*>(smem_raw);
  unsigned char* rest = smem_raw + (size_t)g.slots * kSlot;
  unsigned long long* full = reinterpret_cast<unsigned long long*>(rest);
  unsigned long long* empty = full + g.slots;
  int* s_fail = reinterpret_cast<int*>(empty + g.slots);
  int* tab = s_fail + 4;                    // rounds x nb
  int* kinds = tab + g.rounds * g.nb;       // ntile
  T* D = reinterpret_cast<T*>(smem_raw + (size_t)g.slots * kSlot +
                              ((16 * (size_t)g.slots + 16 +
                                4 * (size_t)(g.rounds * g.nb + g.ntile) + 15) & ~(size_t)15));
  const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
  const int nb = g.nb, nthr = nb * 32, P = g.P, m = g.m;
  const int slot_mask = g.slots - 1, slot_log = __ffs(g.slots) - 1;
  const int row0 = m + 1, nrows = g.N - 2 * (m + 1);
  const int nitems = g.ntiles_row * kBlockEdges;
  // The next kernel's CTAs come in with a CTA's last item: earlier they would only take room from
  // the items' (256 x 256 FP32: 773 us with the trigger here for all, 752 us without).
  if (nitems <= (int)gridDim.x) pdl_trigger();
  for (int i = tid; i < g.rounds * nb; i += blockDim.x) tab[i] = table[i];
  for (int i = tid; i < g.ntile; i += blockDim.x) kinds[i] = tkind[i];
  if (tid == 0) {
    s_fail[0] = g.fail;
    s_fail[1] = 0;
    for (int s = 0; s < g.slots; ++s) {
      mbar_init(&full[s], 1);
      mbar_init(&empty[s], 2);
    }
    asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
  }
  __syncthreads();
  volatile int* vfail = s_fail;
  // tiles issued so far.  A warp's next tile may lie more than a ring ahead of the one it had, so
  // that the parity of its slot's barrier alone would not tell this use of the slot from the one
  // two before; once the tile is issued (every earlier use of the slot is over) it does.
  volatile unsigned* vissued = reinterpret_cast<volatile unsigned*>(s_fail + 1);

  if (w == nb) {  // producer: the first ring of tiles before the kernel before this one has ended
    if (lane == 0) {
      unsigned cnt = 0;
      bool ok = true;
      auto wait_room = [&](unsigned long long* bar, unsigned parity) {
        if (mbar_try_wait(bar, parity)) return true;
        for (long long n = 0; n < kWaitLimit && !*vfail; ++n)
          if (mbar_try_wait(bar, parity)) return true;
        return false;
      };
      for (int it = blockIdx.x; it < nitems && ok; it += gridDim.x) {
        const T* src = K + (size_t)it * g.item_elems;
        for (int s = 0; s < g.ntile; ++s, ++cnt) {
          if (cnt == (unsigned)g.slots) {
            pdl_wait();
            if (done != nullptr && *done) {
              ok = false;
              break;
            }
          }
          const int slot = (int)(cnt & slot_mask);
          if (cnt >= (unsigned)g.slots &&
              !wait_room(&empty[slot], ((cnt >> slot_log) - 1u) & 1u)) {
            *vfail = 1;
            ok = false;
            break;
          }
          const int elems = (kinds[s] ? kDiag : kPair) * kBR;
          mbar_expect_tx(&full[slot], (unsigned)(elems * sizeof(T)));
          if (g.evict_first)
            bulk_g2s_stream(ring + (size_t)slot * kPair * kBR, src, (unsigned)(elems * sizeof(T)), &full[slot]);
          else
            bulk_g2s(ring + (size_t)slot * kPair * kBR, src, (unsigned)(elems * sizeof(T)), &full[slot]);
          src += elems;
          __threadfence_block();
          *vissued = cnt + 1;
        }
      }
      // no copy may be in flight when the CTA ends: the last copy of every slot has landed
      const unsigned used = cnt < (unsigned)g.slots ? cnt : (unsigned)g.slots;
      for (unsigned c = cnt - used; c != cnt; ++c)
        if (!mbar_wait_bounded(&full[c & slot_mask], (c >> slot_log) & 1u)) *vfail = 1;
      if (*vfail) atomicExch(err, 1);
    }
    return;
  }

  pdl_wait();
  if (done != nullptr && *done) return;
  // consumers: thread tid stages elements tid, tid + nthr, ... of an item's 32 x P differences
  auto bar = [&]() { asm volatile("bar.sync 1, %0;\n" ::"r"(nthr) : "memory"); };
  T xi[TS], xj[TS];
  auto fetch = [&](int it) {
    const int t = it / kBlockEdges, e = it - t * kBlockEdges;
    const int valid = min(kBR, nrows - t * kBR) * P;
    const T* p = X + ((size_t)row0 + (size_t)t * kBR) * P + tid;
    const T* q = p + (long long)block_off(e, m) * P;
#pragma unroll
    for (int j = 0; j < TS; ++j) {
      const bool ok = tid + j * nthr < valid;
      xi[j] = ok ? p[j * nthr] : T(0);
      xj[j] = ok && e > 0 ? q[j * nthr] : T(0);
    }
  };
  unsigned base = 0, issued = 0;
  auto wait_tile = [&](unsigned c, int slot) {
    for (long long n = 0; (int)(issued - c) <= 0; ++n) {
      issued = *vissued;
      if (n >= kWaitLimit || *vfail) return false;
    }
    __threadfence_block();
    return mbar_wait_bounded(&full[slot], (c >> slot_log) & 1u);
  };
  if (sizeof(T) == 4 && (int)blockIdx.x < nitems) fetch(blockIdx.x);
  for (int it = blockIdx.x; it < nitems; it += gridDim.x, base += (unsigned)g.ntile) {
    if (nitems > (int)gridDim.x && it + (int)gridDim.x >= nitems) pdl_trigger();
    const int t = it / kBlockEdges, e = it - t * kBlockEdges;
    if (sizeof(T) == 8) fetch(it);
#pragma unroll
    for (int j = 0; j < TS; ++j) {
      const int q = tid + j * nthr;
      if (q < kBR * P) {
        const int r = q / P, b = q - r * P;
        D[b * kBLd + r] = e > 0 ? xj[j] - xi[j] : xi[j];
      }
    }
    // fields beyond P (the last range's padding) are zero
    for (int q = P * kBR + tid; q < nb * TS * kBR; q += nthr) D[(q >> 5) * kBLd + (q & 31)] = T(0);
    bar();
    // FP32: the X rows of the next item are in flight while this one's tiles are used (in FP64 the
    // item's multiply-adds hide them anyway)
    if (sizeof(T) == 4 && it + (int)gridDim.x < nitems) fetch(it + gridDim.x);
    T f[TS];
#pragma unroll
    for (int i = 0; i < TS; ++i) f[i] = T(0);
    for (int r = 0; r < g.rounds; ++r) {
      const int en = tab[r * nb + w];
      const unsigned c = base + (unsigned)(en & 0xffff);
      const int slot = (int)(c & slot_mask), kind = en >> 24;
      const bool got = !*vfail && wait_tile(c, slot);
      if (!got) *vfail = 1;
      const T* k = ring + (size_t)slot * kPair * kBR + lane;
      const T* db = D + (size_t)((en >> 16) & 0xff) * TS * kBLd + lane;
      T d[TS];
#pragma unroll
      for (int j = 0; j < TS; ++j) d[j] = db[j * kBLd];
      if (kind == 0) {
#pragma unroll
        for (int j = 0; j < TS; ++j)
#pragma unroll
          for (int i = 0; i < TS; ++i) f[i] = fma(k[(i * TS + j) * kBR], d[j], f[i]);
      } else if (kind == 1) {
#pragma unroll
        for (int i = 0; i < TS; ++i)
#pragma unroll
          for (int j = 0; j < TS; ++j) f[j] = fma(k[(i * TS + j) * kBR], d[i], f[j]);
      } else {
#pragma unroll
        for (int i = 0; i < TS; ++i)
#pragma unroll
          for (int j = i; j < TS; ++j) {
            const T v = k[(i * TS - i * (i - 1) / 2 + j - i) * kBR];
            f[i] = fma(v, d[j], f[i]);
            if (j > i) f[j] = fma(v, d[i], f[j]);
          }
      }
      __syncwarp();
      if (lane == 0 && got) mbar_arrive_n(&empty[slot], kind == 2 ? 2u : 1u);
    }
    bar();  // every warp has read the differences: f takes their place
    if (*vfail) {
#pragma unroll
      for (int i = 0; i < TS; ++i) f[i] = block_nan<T>();
    }
#pragma unroll
    for (int i = 0; i < TS; ++i) D[(size_t)(w * TS + i) * kBLd + lane] = f[i];
    bar();
    // the thread that reads element q here is the one that stages element q of the next item
    const int valid = min(kBR, nrows - t * kBR) * P;
    T* o = F + ((size_t)e * g.N + row0 + (size_t)t * kBR) * P;
#pragma unroll
    for (int j = 0; j < TS; ++j) {
      const int q = tid + j * nthr;
      if (q < valid) {
        const int r = q / P, b = q - r * P;
        o[q] = D[b * kBLd + r];
      }
    }
  }
}

// Y_i = alpha (S_i x_i + sum_e (f_e(i) - f_e(i - off_e))) + beta B_i at interior nodes (edges of
// boundary nodes are zero: f is not stored before the first interior row), alpha X + beta B at
// boundary nodes.  V values per thread.
template <typename T, int V>
struct __align__(V * sizeof(T)) BlockVec { T v[V]; };

template <typename T, int V>
__global__ void __launch_bounds__(256) block_sum_kernel(int N, int m, int P,
                                                        const T* __restrict__ F,
                                                        const T* __restrict__ X, T* __restrict__ Y,
                                                        T alpha, const T* __restrict__ B, T beta,
                                                        const int* __restrict__ done) {
  pdl_trigger();
  pdl_wait();
  if (done != nullptr && *done) return;
  using W = BlockVec<T, V>;
  const unsigned NP = (unsigned)N * (unsigned)P;
  for (unsigned q = (blockIdx.x * blockDim.x + threadIdx.x) * V; q < NP; q += gridDim.x * blockDim.x * V) {
    const int i = (int)(q / (unsigned)P), y = i / m, x = i - y * m;
    W s;
    if (x > 0 && y > 0 && x < m - 1 && y < m - 1) {
      s = *reinterpret_cast<const W*>(F + q);
      W own[4], nb[4];
#pragma unroll
      for (int e = 1; e < kBlockEdges; ++e) {
        const T* f = F + (size_t)e * NP + q;
        own[e - 1] = *reinterpret_cast<const W*>(f);
        const int off = block_off(e, m);
        if (i - off > m)
          nb[e - 1] = *reinterpret_cast<const W*>(f - (long long)off * P);
        else
#pragma unroll
          for (int v = 0; v < V; ++v) nb[e - 1].v[v] = T(0);
      }
#pragma unroll
      for (int e = 0; e < 4; ++e)
#pragma unroll
        for (int v = 0; v < V; ++v) s.v[v] += own[e].v[v] - nb[e].v[v];
    } else {
      s = *reinterpret_cast<const W*>(X + q);
    }
#pragma unroll
    for (int v = 0; v < V; ++v) s.v[v] *= alpha;
    if (B != nullptr) {
      const W bv = *reinterpret_cast<const W*>(B + q);
#pragma unroll
      for (int v = 0; v < V; ++v) s.v[v] = fma(beta, bv.v[v], s.v[v]);
    }
    *reinterpret_cast<W*>(Y + q) = s;
  }
}

// Tiles of every item from the FP64 stack: CTA (rows RT b .. RT b + RT - 1 of the padded row list,
// edge block e) stages the RT stiffness vectors A_k[i, j] (for S_i the sum over the row's nine
// entries) in shared memory and forms value v, the field pair (a, b) of the tile order, as
// sum over its triples (k, G_k[a,b]) in k order, in FP64.
template <typename T, int RT>
__global__ void __launch_bounds__(512) block_assemble_kernel(
    int N, int m, int L, int nval, const int* __restrict__ rowptr,
    const double* __restrict__ stack, const int* __restrict__ vptr, const int* __restrict__ vk,
    const double* __restrict__ vg, T* __restrict__ K) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  double* A = reinterpret_cast<double*>(smem_raw);  // L x (RT + 1)
  const int e = blockIdx.y, r0 = blockIdx.x * RT;
  const int nrows = N - 2 * (m + 1);
  const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5, nw = blockDim.x >> 5;
  for (int r = w; r < RT; r += nw) {
    const int i = m + 1 + r0 + r, x = i % m;
    const bool inner = r0 + r < nrows && x > 0 && x < m - 1;
    const double* src = inner ? stack + (size_t)rowptr[i] * L : nullptr;
    for (int k = lane; k < L; k += 32) {
      double v = 0.0;
      if (inner) {
        if (e == 0)
          for (int q = 0; q < 9; ++q) v += src[(size_t)q * L + k];
        else
          v = src[(size_t)(e == 1 ? 5 : e + 4) * L + k];
      }
      A[k * (RT + 1) + r] = v;
    }
  }
  __syncthreads();
  const int r = tid & (RT - 1);
  const size_t item = (size_t)((r0 + r) / kBR) * kBlockEdges + e;
  T* out = K + item * (size_t)nval * kBR + ((r0 + r) & (kBR - 1));
  for (int v = tid / RT; v < nval; v += blockDim.x / RT) {
    double s = 0.0;
    for (int q = vptr[v]; q < vptr[v + 1]; ++q) s = fma(vg[q], A[vk[q] * (RT + 1) + r], s);
    out[(size_t)v * kBR] = (T)s;
  }
}

struct BlockPlan {
  int TS = 0, nb = 0, rounds = 0, ntile = 0, nval = 0;
  std::vector<int> table, tkind;
  std::vector<int> va, vb;  // fields of every value of an item, in order
};

// Range size with the fewest padded values (the larger one on a tie: fewer reads of d per value),
// among those that leave at most kBlockMaxWarps ranges.
bool plan_sizes(int P, BlockPlan& pl) {
  long long best = -1;
  for (int ts : {4, 5, 6, 7}) {
    const int nb = (P + ts - 1) / ts;
    if (nb > kBlockMaxWarps) continue;
    const long long nv = (long long)nb * (nb - 1) / 2 * ts * ts + (long long)nb * ts * (ts + 1) / 2;
    if (best < 0 || nv <= best) {
      best = nv;
      pl.TS = ts;
      pl.nb = nb;
    }
  }
  if (best < 0) return false;
  pl.nval = (int)best;
  pl.rounds = pl.nb;  // odd: each with one diagonal tile; even: nb - 1 of pairs and one of diagonals
  pl.ntile = pl.nb * (pl.nb + 1) / 2;
  return true;
}

void plan_tables(BlockPlan& pl) {
  const int nb = pl.nb, odd = nb & 1, n = odd ? nb : nb - 1;
  pl.table.assign((size_t)pl.rounds * nb, 0);
  int s = 0;
  auto put = [&](int r, int a, int b) {
    const int ts = pl.TS;
    if (a == b) {
      pl.table[(size_t)r * nb + a] = s | a << 16 | 2 << 24;
      for (int i = 0; i < ts; ++i)
        for (int j = i; j < ts; ++j) {
          pl.va.push_back(a * ts + i);
          pl.vb.push_back(a * ts + j);
        }
    } else {
      pl.table[(size_t)r * nb + a] = s | b << 16;
      pl.table[(size_t)r * nb + b] = s | a << 16 | 1 << 24;
      for (int i = 0; i < ts; ++i)
        for (int j = 0; j < ts; ++j) {
          pl.va.push_back(a * ts + i);
          pl.vb.push_back(b * ts + j);
        }
    }
    pl.tkind.push_back(a == b);
    ++s;
  };
  for (int r = 0; r < n; ++r)
    for (int a = 0; a < n; ++a) {
      const int b = (r - a + n) % n;
      if (a < b) put(r, a, b);
      else if (a == b) odd ? put(r, a, a) : put(r, a, nb - 1);
    }
  if (!odd)
    for (int a = 0; a < nb; ++a) put(nb - 1, a, a);
}

size_t block_smem(const BlockPlan& pl, int elem, int slots) {
  const size_t head = 16 * (size_t)slots + 16 + 4 * (size_t)(pl.rounds * pl.nb + pl.ntile);
  return (size_t)slots * pl.TS * pl.TS * kBR * elem + ((head + 15) & ~(size_t)15) +
         (size_t)pl.nb * pl.TS * kBLd * elem;
}

// Ring slots, a power of two.  CTAs per SM so that about 28 warps are resident (12 ranges of fields:
// 2, 5: 4, 3: 7), their rings sharing some 200 KB; one that is alone on its SM (from 14 ranges on)
// has to fit its differences and tables beside the ring (FP64 P = 126, 18 ranges: 8 slots, not 16;
// n = 24 144 us against the pair kernel's 1060).  0 where two slots do not fit.
int block_slots(const BlockPlan& pl, int elem) {
  const size_t slot = (size_t)pl.TS * pl.TS * kBR * elem;
  const size_t want = (200 * 1024) / std::max(1, std::min(8, 28 / (pl.nb + 1)));
  const size_t most = smem_optin_max();
  int slots = 2;
  if (block_smem(pl, elem, slots) > most) return 0;
  while (slots < 32 && 2 * slots * slot <= want && block_smem(pl, elem, 2 * slots) <= most) slots *= 2;
  return slots;
}

template <typename T>
void (*block_kernel(int ts))(BlockArgs, const int*, const int*, const T*, const T*, T*, const int*, int*) {
  switch (ts) {
    case 4: return block_edge_kernel<T, 4>;
    case 5: return block_edge_kernel<T, 5>;
    case 6: return block_edge_kernel<T, 6>;
    default: return block_edge_kernel<T, 7>;
  }
}

template <typename T, int RT>
int run_assemble(const System& s, const BlockOp& op, const int* vptr, const int* vk,
                 const double* vg, T* K, cudaStream_t st) {
  auto kern = block_assemble_kernel<T, RT>;
  const size_t smem = sizeof(double) * (size_t)s.L * (RT + 1);
  SG_TRY(ensure_smem((const void*)kern, smem));
  kern<<<dim3((unsigned)(op.row_tiles * (kBR / RT)), kBlockEdges), 512, smem, st>>>(
      s.N, s.pat.m, s.L, op.nval, s.rowptr.p, s.stack.p, vptr, vk, vg, K);
  return check_launch("block_assemble");
}

}  // namespace

size_t block_scratch_elems(const System& s) { return (size_t)kBlockEdges * s.N * s.P; }

// Bytes of the block-stencil operator's tiles for this system, 0 where the form does not apply.
// Where a system has few fields and few nodes its two launches take longer than the pair kernel's
// one (n = 16, P = 6: 14 us a call against 11; n = 50, P = 15: 14.5 against 15.2), so it takes
// P >= 10 or 300 k values.
size_t block_op_bytes(const System& s, int elem) {
  BlockPlan pl;
  if (s.pat.m < 4 || !plan_sizes(s.P, pl) || block_slots(pl, elem) == 0) return 0;
  if ((unsigned long long)s.N * (unsigned long long)s.P >= (1ull << 31)) return 0;
  if (sizeof(double) * (size_t)s.L * 9 > smem_optin_max()) return 0;
  const size_t tiles = ((size_t)s.N - 2 * (s.pat.m + 1) + kBR - 1) / kBR;
  if (s.P < 10 && (size_t)s.N * kBlockEdges * pl.nval < 300000) return 0;
  return tiles * kBlockEdges * (size_t)pl.nval * kBR * elem;
}

// One allocation holds the tiles, the products of an application, and the tables (those of the
// assembly too), which one copy brings, and a mixed system's FP32 tiles are the FP64 ones rounded.
// Bound: allocations and copies, each of which waits for the stream, on small meshes; the assembly's
// multiply-adds on large ones.  Setup of 64 systems of 64 x 64 (P = 35, five levels) 1.69 -> 1.59 s, of
// one of 256 x 256 (P = 84, FP32) 219 -> 206 ms, against ten allocations, five copies and two assemblies.
int build_block_op(System& s, BlockOp& op, int elem, cudaStream_t st) {
  BlockPlan pl;
  if (block_op_bytes(s, elem) == 0 || !plan_sizes(s.P, pl))
    return fail(SG_ERR_ARG, "block operator: unsupported sizes");
  plan_tables(pl);
  op.elem = elem;
  op.TS = pl.TS;
  op.nb = pl.nb;
  op.rounds = pl.rounds;
  op.ntile = pl.ntile;
  op.nval = pl.nval;
  op.row_tiles = (s.N - 2 * (s.pat.m + 1) + kBR - 1) / kBR;
  op.slots = block_slots(pl, elem);
  op.smem = block_smem(pl, elem, op.slots);
  // triples of every field pair a <= b, in k order, then of every value
  const auto pair_of = [&](const Triple& t) { return (size_t)t.a * s.P + t.b; };
  std::vector<int> first((size_t)s.P * s.P + 1, 0);
  for (const Triple& t : s.triples)
    if (t.a <= t.b) ++first[pair_of(t) + 1];
  for (size_t i = 1; i < first.size(); ++i) first[i] += first[i - 1];
  std::vector<const Triple*> order(first.back());
  std::vector<int> next(first.begin(), first.end() - 1);
  for (const Triple& t : s.triples)
    if (t.a <= t.b) order[next[pair_of(t)]++] = &t;
  // tables: vg; then as ints table, tkind, the error word, vptr, vk
  const size_t nent = order.size(), ntab = pl.table.size();
  std::vector<double> host(nent + (ntab + pl.ntile + 1 + (pl.nval + 1) + nent + 1) / 2, 0.0);
  int* const ints = reinterpret_cast<int*>(host.data() + nent);
  std::copy(pl.table.begin(), pl.table.end(), ints);
  std::copy(pl.tkind.begin(), pl.tkind.end(), ints + ntab);
  int* const vptr = ints + ntab + pl.ntile + 1;
  int* const vk = vptr + pl.nval + 1;
  int q = 0;
  for (int v = 0; v < pl.nval; ++v) {
    const int a = pl.va[v], b = pl.vb[v];
    if (a < s.P && b < s.P) {
      const size_t i = (size_t)a * s.P + b;
      for (int e = first[i]; e < first[i + 1]; ++e, ++q) {
        host[q] = order[e]->g;
        vk[q] = order[e]->k;
      }
    }
    vptr[v + 1] = q;
  }
  const size_t total = (size_t)op.row_tiles * kBlockEdges * pl.nval * kBR;
  const size_t scratch = (block_scratch_elems(s) * elem + 15) & ~(size_t)15;
  SG_TRY(op.mem.alloc(total * elem + scratch + host.size() * sizeof(double)));
  op.k = op.mem.p;
  op.f = op.mem.p + total * elem;
  double* const dg = reinterpret_cast<double*>(op.mem.p + total * elem + scratch);
  op.table = reinterpret_cast<int*>(dg + nent);
  op.tkind = op.table + ntab;
  op.err = op.tkind + pl.ntile;
  const int *dptr = op.err + 1, *dk = dptr + pl.nval + 1;
  SG_CUDA(cudaMemcpyAsync(dg, host.data(), host.size() * sizeof(double), cudaMemcpyHostToDevice, st));
  const bool wide = sizeof(double) * (size_t)s.L * 17 > smem_optin_max();
  if (elem == 8)
    SG_TRY(wide ? (run_assemble<double, 8>(s, op, dptr, dk, dg, (double*)op.k, st))
                : (run_assemble<double, 16>(s, op, dptr, dk, dg, (double*)op.k, st)));
  else if (s.block64.ready)  // the values of the FP64 operator, rounded (the same tiles)
    SG_TRY(launch_cast_f32((const double*)s.block64.k, (float*)op.k, total, st));
  else
    SG_TRY(wide ? (run_assemble<float, 8>(s, op, dptr, dk, dg, (float*)op.k, st))
                : (run_assemble<float, 16>(s, op, dptr, dk, dg, (float*)op.k, st)));
  SG_CUDA(cudaStreamSynchronize(st));  // (the copy's source goes)
  const void* kern = elem == 8 ? (const void*)block_kernel<double>(op.TS) : (const void*)block_kernel<float>(op.TS);
  SG_TRY(ensure_smem(kern, op.smem));
  int dev = 0, sms = 0, per_sm = 0;
  SG_CUDA(cudaGetDevice(&dev));
  SG_CUDA(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
  SG_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, (op.nb + 1) * 32, op.smem));
  op.grid = std::max(1, std::min(op.row_tiles * kBlockEdges, sms * std::max(1, per_sm)));
  op.bytes = total * elem;
  op.ready = true;
  return SG_OK;
}

void free_block_op(BlockOp& op) {
  op.mem.release();
  op.ready = false;
}

template <typename T>
int launch_block_op(const System& s, const BlockOp& op, const T* X, T* Y, T alpha, const T* B,
                    T beta, T* F, cudaStream_t st, const int* done) {
  if (!op.ready || F == nullptr) return fail(SG_ERR_ARG, "block operator not built");
  const BlockArgs g{s.N, s.pat.m, s.P, op.nb, op.rounds, op.ntile, op.row_tiles, op.slots,
                    (long long)op.nval * kBR, op.bytes > ((size_t)64 << 20) ? 1 : 0,
                    test_block_fail()};
  auto kern = block_kernel<T>(op.TS);
  TimeScope ts(s.timer, sizeof(T) == 8 ? K_APPLY_F64 : K_APPLY_LOWP, st);
  SG_TRY(launch_pdl(kern, dim3(op.grid), dim3((op.nb + 1) * 32), op.smem, st, g, (const int*)op.table,
                    (const int*)op.tkind, (const T*)op.k, X, F, done, op.err));
  // 16-byte accesses where every row starts on one
  constexpr int kV = 16 / sizeof(T);
  const auto addr = [](const void* p) { return reinterpret_cast<unsigned long long>(p); };
  const bool vec = s.P % kV == 0 && ((addr(X) | addr(Y) | addr(B) | addr(F)) & 15) == 0;
  const size_t n = (size_t)s.N * s.P / (vec ? kV : 1);
  const int grid = (int)std::min<size_t>((n + 255) / 256, 152 * 16);
  return launch_pdl(vec ? block_sum_kernel<T, kV> : block_sum_kernel<T, 1>, dim3(grid), dim3(256), 0, st,
                    s.N, s.pat.m, s.P, (const T*)F, X, Y, alpha, B, beta, done);
}

template int launch_block_op<double>(const System&, const BlockOp&, const double*, double*, double,
                                     const double*, double, double*, cudaStream_t, const int*);
template int launch_block_op<float>(const System&, const BlockOp&, const float*, float*, float,
                                    const float*, float, float*, cudaStream_t, const int*);

}  // namespace sg
