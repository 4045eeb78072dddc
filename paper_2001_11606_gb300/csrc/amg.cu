// amg.cu -- aggregation algebraic multigrid preconditioner (row a5 of the hot
// path) and its V-cycle (inside row a6).
//
// The paper preconditions GMRES with hypre's BoomerAMG, set up once at the
// start of each step and reused in every outer iteration (Sec. 3.2).  This is
// a GPU-native aggregation AMG on the symmetric operator B = V A:
//
//   strength   j is a strong neighbour of i if |B_ij| >= theta sqrt(B_ii B_jj)
//   aggregates Luby-style maximal independent set of the strength graph with
//              fixed hashed priorities (roots), every other node joins the
//              root it is most strongly coupled to; rows without strong
//              neighbours stay unaggregated (left to the smoother)
//   transfer   piecewise-constant prolongation P (tentative), R = P^T
//   Galerkin   B_c = P^T B P: each coarse entry is the sum of the fine entries
//              that map to it, summed in a fixed order (deterministic)
//   smoother   Chebyshev on D^{-1} B with the interval [lmax/8, lmax],
//              lmax from Gershgorin; the coarsest level gets a Chebyshev solve
//              over its whole Gershgorin interval
//
// The V-cycle uses the same polynomial before and after the coarse
// correction, so it is a symmetric positive-definite preconditioner for CG.
//
// Everything runs on the device.  Aggregates and the coarse sparsity are built
// from the first step's operator and kept (config.amg_rebuild = 1 rebuilds
// them every step); the Galerkin values are recomputed every step.
#include <cuda_runtime.h>

#include <algorithm>
#include <vector>

#include <cooperative_groups.h>

#include "common.cuh"
#include "sliced.cuh"

namespace cg = cooperative_groups;

namespace sphrt {

sph_rt_status exclusive_scan(sph_rt *s, const int64_t *in, int64_t n, int64_t *out);
template <typename MT, typename VT>
sph_rt_status cheb_apply(sph_rt *s, const CsrView<MT> &A, const VT *r, VT *z, VT *d, VT *tmp,
                         int degree, const ChebCoef *cf, const Scalars *sc, bool first_done);
sph_rt_status launch_cheb_slots(sph_rt *s, int first, const double *gersh_dev,
                                const std::vector<int> &mode, const std::vector<int> &degree);

constexpr int kUndecided = 1, kRoot = 2, kNonroot = 0, kIsolated = 3;
constexpr int kHash = 4096;        // shared hash-table slots per coarse row
constexpr int kCoarseTarget = 512;  // stop coarsening at or below this many rows
constexpr int kMaxLevels = 12;
static_assert(1 + kMaxLevels <= kChebSlots, "one Chebyshev slot per AMG level");

}  // namespace sphrt

// Source indices of Galerkin sums over a level's entries (k < nnz for an
// off-diagonal entry, nnz + i for a diagonal): 32 bits while nnz + n fits
// (below 2^31 - 1, or unless config.index64), else 64 bits.  Exactly one of
// the two is set.
struct SrcList {
  int32_t *i32 = nullptr;
  int64_t *i64 = nullptr;
};

struct SphLevel {
  int64_t n = 0, nnz = 0;
  // operator (level 0 borrows the fine operator; others own theirs)
  int64_t *ptr = nullptr;
  int32_t *col = nullptr;
  double *val = nullptr, *diag = nullptr, *invdiag = nullptr;
  float *val32 = nullptr, *diag32 = nullptr, *invdiag32 = nullptr;
  // transfer to the next level
  int32_t *agg = nullptr;       // [n] coarse row of each row, -1 if unaggregated
  int64_t *agg_ptr = nullptr;   // [nc+1] members of each coarse row
  int32_t *agg_mem = nullptr;
  int64_t *seg_ptr = nullptr;   // [nnz_c + nc + 1] Galerkin contributions per coarse target
  SrcList seg_src;              // source: k < nnz (off-diagonal entry) or nnz + i (diagonal)
  // vectors of the V-cycle
  double *r = nullptr, *z = nullptr, *res = nullptr, *d = nullptr, *t = nullptr;
  float *r32 = nullptr, *z32 = nullptr, *res32 = nullptr, *d32 = nullptr, *t32 = nullptr;
  int W = 32, U = 4;
  // finest level only: A P (P = this level's aggregation), by fine row
  int64_t nnz_ap = 0;
  int64_t *ap_ptr = nullptr;    // [n + 1]
  int32_t *ap_col = nullptr;    // [nnz_ap] aggregate (next-level row)
  int64_t *ap_seg_ptr = nullptr;  // [nnz_ap + 1] sources of each A P entry
  SrcList ap_seg_src;             // source: k < nnz (off-diagonal entry) or nnz + i (diagonal)
  int64_t *apg_ptr = nullptr;     // [nnz_c + nc + 1] next level's Galerkin sums over A P entries
  int32_t *apg_src = nullptr;     // (P^T (A P): each A P entry (i, K) adds to (agg[i], K))
  double *ap_val = nullptr;     // [nnz_ap], or in slice order [ap_sl.padded]
  float *ap_val32 = nullptr;
  // A P in slices, where the operator is (ap_ptr and ap_col then only describe its
  // rows): ap_pos is each operator entry's place within its row's A P entries
  SlicedRowsData ap_sl;
  uint16_t *ap_pos = nullptr;
  int ap_most = 0;              // most A P entries of a row
  // finest level, mixed form with the V-cycle's CG product (fine_post_smooth = 0):
  // the CG's FP32 search direction p, its product q = B p and w = B z
  float *p32 = nullptr, *q32 = nullptr, *w32 = nullptr;
  std::vector<void *> owned;
};

namespace sphrt {

// Level buffers come from the handle's caching allocator and go back to it
// when the hierarchy is released (after a stream synchronisation).
static void *lvl_alloc(sph_rt *s, SphLevel *L, size_t bytes) {
  void *p = dalloc_bytes(s, bytes > 0 ? bytes : 16);
  if (p) L->owned.push_back(p);
  return p;
}
template <typename T>
static T *lalloc(sph_rt *s, SphLevel *L, size_t count) {
  return static_cast<T *>(lvl_alloc(s, L, sizeof(T) * (count > 0 ? count : 1)));
}
// scratch buffer of one set-up phase
template <typename T>
static T *scratch(sph_rt *s, size_t count) {
  return static_cast<T *>(dalloc_bytes(s, sizeof(T) * (count > 0 ? count : 1)));
}

void amg_release(sph_rt *s) {
  if (!s->levels.empty() && s->cuda_ready) cudaStreamSynchronize(s->stream);
  for (SphLevel *L : s->levels) {
    for (void *p : L->owned) dfree(s, p);
    delete L;
  }
  s->levels.clear();
  s->amg_ready = false;
}

static int gcap(const sph_rt *s, int64_t n, int per_block) {
  int64_t g = ceil_div(n > 0 ? n : 1, per_block);
  int64_t cap = (int64_t)s->num_sms * 8;
  if (cap > kMaxRedBlocks) cap = kMaxRedBlocks;
  return (int)(g < cap ? g : cap);
}

__device__ __forceinline__ uint32_t hash_u32(uint32_t x) {  // integer mixer (Wang-style)
  x = (x ^ 61u) ^ (x >> 16);
  x *= 9u;
  x ^= x >> 4;
  x *= 0x27d4eb2du;
  x ^= x >> 15;
  return x;
}
// priority order: larger hash wins, ties by larger index
__device__ __forceinline__ bool beats(uint32_t i, uint32_t j) {
  uint32_t hi = hash_u32(i), hj = hash_u32(j);
  return hi > hj || (hi == hj && i > j);
}

// ---------------------------------------------------------------------------
// strength and aggregation
// ---------------------------------------------------------------------------
// A warp per row: the row's entries 32 at a time (coalesced), the count of
// strong entries by ballot.
__global__ void strength_kernel(int64_t n, const int64_t *ptr, const int32_t *col,
                                const double *val, const double *diag, double theta2,
                                uint8_t *strong, int *state) {
  const int lane = threadIdx.x & 31;
  const int64_t warp = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
  for (int64_t i = warp; i < n; i += nwarps) {
    int cnt = 0;
    const double di = diag[i];
    const int64_t e = ptr[i + 1];
    for (int64_t k0 = ptr[i]; k0 < e; k0 += 32) {
      const int64_t k = k0 + lane;
      bool st = false;
      if (k < e) {
        const int32_t j = col[k];
        // |B_ij| >= theta sqrt(B_ii B_jj), squared: no FP64 square root per entry
        st = j != i && val[k] * val[k] >= theta2 * (di * diag[j]);
        strong[k] = st;
      }
      cnt += __popc(__ballot_sync(0xffffffffu, st));
    }
    if (lane == 0) state[i] = cnt > 0 ? kUndecided : kIsolated;
  }
}

// The MIS passes and the assignment with a warp per row: the row's entries
// 32 at a time (coalesced), decisions by ballot, the assignment's strongest
// root by a warp arg-max under the same order (largest |B_ij|, then smallest
// j; the columns of a row are distinct, so the choice is unique).
__global__ void mis_select_kernel(int64_t n, const int64_t *ptr, const int32_t *col,
                                  const uint8_t *strong, const int *state, uint8_t *cand) {
  const int lane = threadIdx.x & 31;
  const int64_t warp = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
  for (int64_t i = warp; i < n; i += nwarps) {
    uint8_t c = 0;
    if (state[i] == kUndecided) {
      c = 1;
      const int64_t e = ptr[i + 1];
      for (int64_t k0 = ptr[i]; k0 < e; k0 += 32) {
        const int64_t k = k0 + lane;
        bool block = false;
        if (k < e && strong[k]) {
          const int32_t j = col[k];
          const int sj = state[j];
          block = sj == kRoot || (sj == kUndecided && beats((uint32_t)j, (uint32_t)i));
        }
        if (__ballot_sync(0xffffffffu, block)) {
          c = 0;
          break;
        }
      }
    }
    if (lane == 0) cand[i] = c;
  }
}

__global__ void mis_apply_kernel(int64_t n, const uint8_t *cand, int *state) {
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x)
    if (cand[i]) state[i] = kRoot;
}

__global__ void mis_mark_kernel(int64_t n, const int64_t *ptr, const int32_t *col,
                                const uint8_t *strong, int *state, unsigned *undecided) {
  const int lane = threadIdx.x & 31;
  const int64_t warp = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
  unsigned left = 0;
  for (int64_t i = warp; i < n; i += nwarps) {
    if (state[i] != kUndecided) continue;  // warp-uniform
    bool nr = false;
    const int64_t e = ptr[i + 1];
    for (int64_t k0 = ptr[i]; k0 < e && !nr; k0 += 32) {
      const int64_t k = k0 + lane;
      const bool hit = k < e && strong[k] && state[col[k]] == kRoot;
      nr = __ballot_sync(0xffffffffu, hit) != 0;
    }
    if (lane == 0) {
      if (nr) state[i] = kNonroot;
      else ++left;
    }
  }
  if (left) atomicAdd(undecided, left);
}

__global__ void root_flag_kernel(int64_t n, const int *state, int64_t *flag) {
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x)
    flag[i] = state[i] == kRoot ? 1 : 0;
}

__global__ void assign_kernel(int64_t n, const int64_t *ptr, const int32_t *col, const double *val,
                              const uint8_t *strong, const int *state, const int64_t *root_id,
                              int32_t *agg, unsigned *members) {
  const int lane = threadIdx.x & 31;
  const int64_t warp = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
  for (int64_t i = warp; i < n; i += nwarps) {
    const int st = state[i];
    int32_t a = -1;
    if (st == kRoot) {
      a = (int32_t)root_id[i];
    } else if (st == kNonroot) {
      double best = -1.0;
      int32_t bj = -1;
      const int64_t e = ptr[i + 1];
      for (int64_t k = ptr[i] + lane; k < e; k += 32) {
        const int32_t j = col[k];
        if (!strong[k] || state[j] != kRoot) continue;
        const double v = fabs(val[k]);
        if (v > best || (v == best && j < bj)) {
          best = v;
          bj = j;
        }
      }
      for (int o = 16; o > 0; o >>= 1) {
        const double ov = __shfl_xor_sync(0xffffffffu, best, o);
        const int32_t oj = __shfl_xor_sync(0xffffffffu, bj, o);
        if (oj >= 0 && (bj < 0 || ov > best || (ov == best && oj < bj))) {
          best = ov;
          bj = oj;
        }
      }
      a = bj >= 0 ? (int32_t)root_id[bj] : -1;
    }
    if (lane == 0) {
      agg[i] = a;
      if (a >= 0) atomicAdd(&members[a], 1u);
    }
  }
}

// counting-sort scatter + per-segment insertion sort (shared by the member
// lists and the Galerkin contribution lists): orders each segment by value
// S: the item index type (int32_t, or int64_t for more than 2^31 - 1 items)
template <typename S>
__global__ void bucket_scatter_kernel(int64_t n, const int32_t *bucket, const int64_t *start,
                                      unsigned *cursor, S *out) {
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x) {
    int32_t b = bucket[i];
    if (b < 0) continue;
    int64_t at = start[b] + atomicAdd(&cursor[b], 1u);
    out[at] = (S)i;
  }
}
// Buckets of up to kSmallBucket items are insertion-sorted by one thread
// (bucket_sort_kernel); larger ones, where a quadratic sort in one thread
// would dominate the set-up, by a warp (bucket_rank_kernel).
constexpr int kSmallBucket = 32;
// largest bucket the warp sort stages in shared memory (32 KB a block)
template <typename S>
constexpr int rank_bucket() { return 4096 / (int)sizeof(S); }
template <typename S>
__device__ __forceinline__ void insertion_sort(S *a, int64_t c) {
  for (int64_t t = 1; t < c; ++t) {
    S v = a[t];
    int64_t u = t - 1;
    while (u >= 0 && a[u] > v) {
      a[u + 1] = a[u];
      --u;
    }
    a[u + 1] = v;
  }
}
// A thread per small bucket, sorted in the thread's slice of shared memory
// (one read and one write of the bucket in global memory); 64-bit items, for
// the rare levels past 2^31 sources, are sorted in place.
template <typename S>
__global__ void __launch_bounds__(kBlock) bucket_sort_kernel(int64_t nb, const int64_t *start,
                                                             S *out) {
  __shared__ int32_t stage[kSmallBucket][kBlock];  // item q of thread t at [q][t]
  for (int64_t b = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; b < nb;
       b += (int64_t)gridDim.x * blockDim.x) {
    const int64_t s0 = start[b], c = start[b + 1] - s0;
    if (c < 2 || c > kSmallBucket) continue;
    if (sizeof(S) != sizeof(int32_t)) {
      insertion_sort(out + s0, c);
      continue;
    }
    for (int q = 0; q < (int)c; ++q) stage[q][threadIdx.x] = (int32_t)out[s0 + q];
    for (int t = 1; t < (int)c; ++t) {
      const int32_t v = stage[t][threadIdx.x];
      int u = t - 1;
      while (u >= 0 && stage[u][threadIdx.x] > v) {
        stage[u + 1][threadIdx.x] = stage[u][threadIdx.x];
        --u;
      }
      stage[u + 1][threadIdx.x] = v;
    }
    for (int q = 0; q < (int)c; ++q) out[s0 + q] = stage[q][threadIdx.x];
  }
}
// A warp takes 32 consecutive buckets and sorts each larger one in turn: the
// items (distinct indices) are staged in shared memory and each is written at
// its rank, the number of smaller items.  Buckets beyond rank_bucket items
// (not met by the aggregation levels, whose sources per target are a few
// hundred at most) fall back to one thread.
template <typename S>
__global__ void bucket_rank_kernel(int64_t nb, const int64_t *start, S *out) {
  constexpr int kRankBucket = rank_bucket<S>();
  __shared__ S stage[kWarpsPerBlock][kRankBucket];
  S *sm = stage[threadIdx.x >> 5];
  const int lane = threadIdx.x & 31;
  const int64_t warp = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
  for (int64_t b0 = warp * 32; b0 < nb; b0 += nwarps * 32) {
    const int64_t b = b0 + lane;
    const int64_t c = b < nb ? start[b + 1] - start[b] : 0;
    unsigned m = __ballot_sync(0xffffffffu, c > kSmallBucket);
    while (m) {
      const int t = __ffs(m) - 1;
      m &= m - 1;
      const int64_t bb = b0 + t;
      const int64_t s0 = start[bb], cc = start[bb + 1] - s0;
      if (cc > kRankBucket) {
        if (lane == 0) insertion_sort(out + s0, cc);
        __syncwarp();
        continue;
      }
      for (int64_t k = lane; k < cc; k += 32) sm[k] = out[s0 + k];
      __syncwarp();
      for (int64_t k = lane; k < cc; k += 32) {
        const S v = sm[k];
        int rank = 0;
        for (int q = 0; q < (int)cc; ++q) rank += sm[q] < v;
        out[s0 + rank] = v;
      }
      __syncwarp();
    }
  }
}

__global__ void u32_to_i64_kernel(int64_t n, const unsigned *in, int64_t *out) {
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x)
    out[i] = in[i];
}

// ---------------------------------------------------------------------------
// coarse sparsity: one block per coarse row, shared-memory hash of the coarse
// columns reached from the members' rows, then sorted.  agg == nullptr: the rows'
// columns are coarse already (the rows of A P) and no targets are wanted.
// ---------------------------------------------------------------------------
template <bool FILL>
__global__ void coarse_struct_kernel(int64_t nc, const int64_t *agg_ptr, const int32_t *agg_mem,
                                     const int64_t *ptr, const int32_t *col, const int32_t *agg,
                                     int64_t *ccount, const int64_t *cptr, int32_t *ccol,
                                     int32_t *tgt, int64_t nnz_c, int32_t *tgt_diag,
                                     int *overflow) {
  __shared__ int32_t table[kHash];
  __shared__ int32_t keys[kHash / 2];
  __shared__ int nkeys;
  for (int64_t I = blockIdx.x; I < nc; I += gridDim.x) {
    for (int t = threadIdx.x; t < kHash; t += blockDim.x) table[t] = 0x7fffffff;
    if (threadIdx.x == 0) nkeys = 0;
    __syncthreads();
    const int64_t m0 = agg_ptr[I], m1 = agg_ptr[I + 1];
    // insert
    for (int64_t m = m0; m < m1; ++m) {
      int32_t i = agg_mem[m];
      for (int64_t k = ptr[i] + threadIdx.x; k < ptr[i + 1]; k += blockDim.x) {
        const int32_t J = agg ? agg[col[k]] : col[k];
        if (J < 0 || J == (int32_t)I) continue;
        uint32_t hsh = hash_u32((uint32_t)J) & (kHash - 1);
        for (int probe = 0; probe < kHash; ++probe) {
          int32_t prev = atomicCAS(&table[hsh], 0x7fffffff, J);
          if (prev == 0x7fffffff) {
            atomicAdd(&nkeys, 1);
            break;
          }
          if (prev == J) break;
          hsh = (hsh + 1) & (kHash - 1);
        }
      }
    }
    __syncthreads();
    int cnt = nkeys;
    if (cnt > kHash / 2) {  // too wide for the table's load factor: give up on this level
      if (threadIdx.x == 0) atomicExch(overflow, 1);
      __syncthreads();
      continue;
    }
    // compact the keys (any order), pad to a power of two and sort ascending
    __shared__ int ncomp;
    if (threadIdx.x == 0) ncomp = 0;
    __syncthreads();
    for (int t = threadIdx.x; t < kHash; t += blockDim.x) {
      int32_t v = table[t];
      if (v != 0x7fffffff) keys[atomicAdd(&ncomp, 1)] = v;
    }
    int P2 = 1;
    while (P2 < cnt) P2 <<= 1;
    __syncthreads();
    for (int t = cnt + threadIdx.x; t < P2; t += blockDim.x) keys[t] = 0x7fffffff;
    __syncthreads();
    for (int k = 2; k <= P2; k <<= 1) {
      for (int j = k >> 1; j > 0; j >>= 1) {
        for (int t = threadIdx.x; t < P2; t += blockDim.x) {
          int u = t ^ j;
          if (u > t) {
            int32_t a = keys[t], b = keys[u];
            bool up = (t & k) == 0;
            if ((a > b) == up) {
              keys[t] = b;
              keys[u] = a;
            }
          }
        }
        __syncthreads();
      }
    }
    if (!FILL) {
      if (threadIdx.x == 0) ccount[I] = cnt;
    } else {
      const int64_t base = cptr[I];
      for (int t = threadIdx.x; t < cnt; t += blockDim.x) ccol[base + t] = keys[t];
      for (int64_t m = m0; m < m1 && tgt; ++m) {
        int32_t i = agg_mem[m];
        if (threadIdx.x == 0) tgt_diag[i] = (int32_t)(nnz_c + I);
        for (int64_t k = ptr[i] + threadIdx.x; k < ptr[i + 1]; k += blockDim.x) {
          int32_t J = agg[col[k]];
          int32_t tg = -1;
          if (J == (int32_t)I) {
            tg = (int32_t)(nnz_c + I);
          } else if (J >= 0) {
            int lo = 0, hi = cnt;  // lower_bound
            while (lo < hi) {
              int mid = (lo + hi) >> 1;
              if (keys[mid] < J) lo = mid + 1;
              else hi = mid;
            }
            tg = (int32_t)(base + lo);
          }
          tgt[k] = tg;
        }
      }
    }
    __syncthreads();
  }
}

// The same from the rows of A P with a warp per coarse row: an aggregate of ~6
// rows has ~190 A P entries and ~50 distinct columns, too few for a block and its
// 4096-slot table.  The members' entries are walked 32 at a time into a small hash
// table, and the distinct columns sorted by the warp and written at off[I] (room
// for all the members' entries); they are compacted once the counts are known, so
// the rows are hashed once.  *wide: a row has more than kWarpCols columns; the
// block kernels above then do the level.  (Both passes of the block kernels, over
// the operator's own entries, took 3.5 ms for the levels of 97 x 96 x 91 particles;
// this takes 0.28.)
constexpr int kWarpTable = 1024, kWarpCols = 512;
__global__ void member_bound_kernel(int64_t nc, const int64_t *agg_ptr, const int32_t *agg_mem,
                                    const int64_t *ap_ptr, int64_t *bound) {
  for (int64_t I = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; I < nc;
       I += (int64_t)gridDim.x * blockDim.x) {
    int64_t b = 0;
    for (int64_t m = agg_ptr[I]; m < agg_ptr[I + 1]; ++m) {
      const int32_t i = agg_mem[m];
      b += ap_ptr[i + 1] - ap_ptr[i];
    }
    bound[I] = b;
  }
}
constexpr int kCoarseRowWarps = 4;
__global__ void __launch_bounds__(32 * kCoarseRowWarps)
    coarse_rows_kernel(int64_t nc, const int64_t *agg_ptr, const int32_t *agg_mem,
                       const int64_t *ap_ptr, const int32_t *ap_col, const int64_t *off,
                       int32_t *cols, int64_t *ccount, int *wide) {
  __shared__ int32_t table_sh[kCoarseRowWarps][kWarpTable];
  __shared__ int32_t keys_sh[kCoarseRowWarps][kWarpCols];
  constexpr int32_t kFree = 0x7fffffff;
  int32_t *table = table_sh[threadIdx.x >> 5], *keys = keys_sh[threadIdx.x >> 5];
  const int lane = threadIdx.x & 31;
  const unsigned lt = (1u << lane) - 1u;
  const int64_t warp = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
  for (int t = lane; t < kWarpTable; t += 32) table[t] = kFree;
  __syncwarp();
  for (int64_t I = warp; I < nc; I += nwarps) {
    int cnt = 0;  // distinct columns so far (warp-uniform)
    for (int64_t m = agg_ptr[I]; m < agg_ptr[I + 1] && cnt <= kWarpCols; ++m) {
      const int32_t i = agg_mem[m];
      const int64_t e = ap_ptr[i + 1];
      for (int64_t k0 = ap_ptr[i]; k0 < e && cnt <= kWarpCols; k0 += 32) {
        const int64_t k = k0 + lane;
        const int32_t J = k < e ? ap_col[k] : (int32_t)I;
        bool fresh = false;
        if (J != (int32_t)I) {
          // at most kWarpCols + 32 of the kWarpTable slots are ever used
          uint32_t h = hash_u32((uint32_t)J) & (kWarpTable - 1);
          for (int probe = 0; probe < kWarpTable; ++probe) {
            const int32_t prev = atomicCAS(&table[h], kFree, J);
            fresh = prev == kFree;
            if (fresh || prev == J) break;
            h = (h + 1) & (kWarpTable - 1);
          }
        }
        const unsigned mask = __ballot_sync(0xffffffffu, fresh);
        const int at = cnt + __popc(mask & lt);
        if (fresh && at < kWarpCols) keys[at] = J;
        cnt += __popc(mask);
      }
    }
    __syncwarp();
    if (cnt > kWarpCols) {
      if (lane == 0) {
        *wide = 1;
        ccount[I] = 0;
      }
      for (int t = lane; t < kWarpTable; t += 32) table[t] = kFree;
      __syncwarp();
      continue;
    }
    int P2 = 32;
    while (P2 < cnt) P2 <<= 1;
    for (int t = cnt + lane; t < P2; t += 32) keys[t] = kFree;
    __syncwarp();
    for (int k = 2; k <= P2; k <<= 1)
      for (int j = k >> 1; j > 0; j >>= 1) {
        for (int t = lane; t < P2; t += 32) {
          const int u = t ^ j;
          if (u > t) {
            const int32_t a = keys[t], b = keys[u];
            if ((a > b) == ((t & k) == 0)) {
              keys[t] = b;
              keys[u] = a;
            }
          }
        }
        __syncwarp();
      }
    for (int t = lane; t < cnt; t += 32) cols[off[I] + t] = keys[t];
    if (lane == 0) ccount[I] = cnt;
    // clear the table for the next row
    for (int t = lane; t < kWarpTable; t += 32) table[t] = kFree;
    __syncwarp();
  }
}
// rows of `cnt` entries at in[off[i]] to out[ptr[i]], a warp per row
__global__ void compact_rows_kernel(int64_t n, const int64_t *off, const int32_t *in,
                                    const int64_t *ptr, int32_t *out) {
  const int lane = threadIdx.x & 31;
  const int64_t warp = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
  for (int64_t i = warp; i < n; i += nwarps) {
    const int64_t b = ptr[i], c = ptr[i + 1] - b, o = off[i];
    for (int64_t t = lane; t < c; t += 32) out[b + t] = in[o + t];
  }
}
// where ap_structure wrote row i's aggregates
__global__ void ap_offset_kernel(int64_t n, const int64_t *ptr, int64_t *off) {
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x)
    off[i] = ptr[i] + i;
}

// targets of the fine diagonal entries of unaggregated rows stay -1
__global__ void fill_i32_kernel(int64_t n, int32_t v, int32_t *a) {
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x)
    a[i] = v;
}

__global__ void target_count_kernel(int64_t nsrc, const int32_t *tgt, unsigned *cnt) {
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < nsrc;
       i += (int64_t)gridDim.x * blockDim.x) {
    int32_t t = tgt[i];
    if (t >= 0) atomicAdd(&cnt[t], 1u);
  }
}

// Galerkin values: thread per coarse target, fixed-order sum of its sources
// (8 source indices loaded before their gathers, so the gathers overlap).  A
// warp adds as many slots of a batch as its longest segment has left (most
// A P targets have 3-4 sources): the additions a lane skips would add +0.0,
// and a sum that starts at +0.0 is unchanged by them, so the result is that of
// adding all 8 slots.
// T: the hierarchy's value type (FP32 in the mixed form: its sums are formed
// from the FP32 fine values directly).
// S: the source index type (SrcList).
template <typename T, typename S>
__global__ void galerkin_kernel(int64_t nnz_c, int64_t nc, const int64_t *seg_ptr,
                                const S *seg_src, int64_t nnz_f, const T *val_f,
                                const T *diag_f, T *val_c, T *diag_c, T *invdiag_c) {
  constexpr int G = 8;
  for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < nnz_c + nc;
       t += (int64_t)gridDim.x * blockDim.x) {
    const unsigned mask = __activemask();
    T acc = T(0);
    const int64_t u1 = seg_ptr[t + 1];
    for (int64_t u = seg_ptr[t];; u += G) {
      const int64_t left = u1 - u;
      const int m = __reduce_max_sync(mask, left <= 0 ? 0 : (left < G ? (int)left : G));
      if (m == 0) break;  // uniform over the lanes of `mask`
      S src[G];
#pragma unroll
      for (int g = 0; g < G; ++g) src[g] = u + g < u1 ? __ldg(seg_src + u + g) : S(-1);
      T v[G];
#pragma unroll
      for (int g = 0; g < G; ++g)
        v[g] = src[g] < 0 ? T(0) : (src[g] < nnz_f ? __ldg(val_f + src[g]) : __ldg(diag_f + (src[g] - nnz_f)));
#pragma unroll 1
      for (int g = 0; g < m; ++g) {
        acc += v[0];  // sources in order; a shorter segment's padding adds +0.0
#pragma unroll
        for (int q = 0; q + 1 < G; ++q) v[q] = v[q + 1];
      }
    }
    if (t < nnz_c) {
      val_c[t] = acc;
    } else {
      diag_c[t - nnz_c] = acc;
      invdiag_c[t - nnz_c] = T(1) / acc;
    }
  }
}

// Gershgorin bounds of D^{-1} A, max_i sum_j |A_ij| / A_ii, of all levels in one
// launch: row tiles (one FP64 addition an entry, the quotients on all lanes), the
// maxima (of non-negative values, so ordered like their bit patterns, and the same
// in any order) by atomics.  The finest level's bound was reduced by the assembly.
// (One launch per level with a thread per row took 27 us a step for four levels
// under 8.6e4 particles, 275 for seven under 1.3e6; this takes 12 and
// 168.)
template <typename T>
struct GershLevels {
  int count;  // levels 1 .. count - 1
  struct {
    int64_t n;
    const int64_t *ptr;
    const T *val, *diag;
  } L[kMaxLevels];
};
template <typename T>
__global__ void gersh_kernel(const __grid_constant__ GershLevels<T> G, const double *fine,
                             double *out) {
  constexpr int W = 4, U = 8;
  const int lane = threadIdx.x & 31, sub = lane % W, own = tile_own_row<W>(lane);
  if (blockIdx.x == 0 && threadIdx.x == 0) out[0] = *fine;
  for (int l = 1; l < G.count; ++l) {
    const int64_t *__restrict__ ptr = G.L[l].ptr;
    const T *__restrict__ val = G.L[l].val;
    double g = 0.0;
    int64_t r0, r1;
    warp_rows<W>(G.L[l].n, r0, r1);
    for (int64_t base = r0; base < r1; base += 32) {
      const int rows = (int)(r1 - base < 32 ? r1 - base : 32);
      int64_t b = 0, e = 0;
      if (own < rows) {
        b = ptr[base + own];
        e = ptr[base + own + 1];
      }
      const double s = tile_tree<W, 1, double>(0, rows, sub, [&](int t) -> double {
        const int64_t rb = __shfl_sync(0xffffffffu, b, t, W);
        const int64_t re = __shfl_sync(0xffffffffu, e, t, W);
        double acc = 0.0;
        for (int64_t k = rb + sub; k < re; k += W * U) {
          T v[U];
#pragma unroll
          for (int u = 0; u < U; ++u) v[u] = k + u * W < re ? __ldg(val + k + u * W) : T(0);
#pragma unroll
          for (int u = 0; u < U; ++u)
            if (k + u * W < re) acc += fabs(widen(v[u]));
        }
        __syncwarp();
        return acc;
      });
      if (own < rows) g = max_bits(g, quotient(s, widen(G.L[l].diag[base + own])));
    }
    g = warp_max_bits(g);
    if ((threadIdx.x & 31) == 0 && g > 0.0)
      atomicMax(reinterpret_cast<unsigned long long *>(out + l),
                (unsigned long long)__double_as_longlong(g));
  }
}

template <typename S, typename D>
__global__ void convert_kernel(int64_t n, const S *in, D *out) {
  pdl_wait();
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x)
    out[i] = (D)in[i];
}

// ---------------------------------------------------------------------------
// V-cycle kernels
// ---------------------------------------------------------------------------
// One sweep, two names (finest level vs coarse levels in profiles); the coarse one
// loads its row operands before the row sums, as in cheb_step_kernel.
template <int W, int U, typename MT, typename VT>
__global__ void __launch_bounds__(kBlock, kCoarseMinBlocks)
    resid_level_kernel(CsrView<MT> A, const VT *r, const VT *z, VT *res, const Scalars *sc) {
  pdl_wait();
  if (sc && sc->done) return;
  const int own = tile_own_row<W>(threadIdx.x & 31);
  int64_t r0, r1;
  warp_rows<W>(A.n, r0, r1);
  for (int64_t base = r0; base < r1; base += 32) {
    const int rows = (int)(r1 - base < 32 ? r1 - base : 32);
    const int64_t i = base + own;
    const bool active = own < rows;
    VT ri = VT(0), dg = VT(0), zi = VT(0);
    if (active) {
      ri = r[i];
      dg = (VT)A.diag[i];
      zi = z[i];
    }
    const VT s = tile_row_sums<W, U, MT, VT>(base, rows, A.ptr, A.col, A.val, z);
    if (active) res[i] = ri - fmadd(dg, zi, s);
  }
}
template <typename Rows, typename VT>
__global__ void __launch_bounds__(kBlock, Rows::kMinBlocks)
    fine_resid_level_kernel(Rows A, const VT *r, const VT *z, VT *res, const Scalars *sc,
                            int *wflag) {
  pdl_wait();
  if (sc && sc->done) {
    mark_work(wflag, 0);
    return;
  }
  mark_work(wflag, 1);
  A.each(
      z, [&](int64_t i) { return Ops3<VT>{r[i], (VT)A.A.diag[i], z[i]}; },
      [&](int64_t i, VT s, const Ops3<VT> &o) { res[i] = o.a - fmadd(o.b, o.c, s); });
}

// Sum of res over the members [m0, m1) of an aggregate, in member order.
// Aggregates have ~6 members: 8 member indices are loaded before their
// gathers, so an aggregate costs two dependent round trips instead of two per
// member.
template <typename VT>
__device__ __forceinline__ VT aggregate_sum(int64_t m0, int64_t m1, const int32_t *agg_mem,
                                            const VT *res) {
  constexpr int G = 8;
  VT acc = 0;
  for (int64_t m = m0; m < m1; m += G) {
    int32_t j[G];
#pragma unroll
    for (int g = 0; g < G; ++g) j[g] = m + g < m1 ? agg_mem[m + g] : -1;
    VT v[G];
#pragma unroll
    for (int g = 0; g < G; ++g) v[g] = j[g] >= 0 ? res[j[g]] : VT(0);
#pragma unroll
    for (int g = 0; g < G; ++g)
      if (j[g] >= 0) acc += v[g];
  }
  return acc;
}

template <typename VT>
__global__ void restrict_kernel(int64_t nc, const int64_t *agg_ptr, const int32_t *agg_mem,
                                const VT *res, VT *rc, const Scalars *sc) {
  pdl_wait();
  if (sc && sc->done) return;
  for (int64_t I = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; I < nc;
       I += (int64_t)gridDim.x * blockDim.x) {
    const VT acc = aggregate_sum(agg_ptr[I], agg_ptr[I + 1], agg_mem, res);
    rc[I] = acc;
  }
}

// Restriction fused with the next level's zero-guess smoother start
// (cheb_init_zero_kernel's arithmetic): rc = P^T res; d_c = z_c = D_c^{-1} rc / theta_c.
template <typename MT, typename VT>
__global__ void restrict_init_kernel(int64_t nc, const int64_t *agg_ptr, const int32_t *agg_mem,
                                     const VT *res, VT *rc, const MT *invdiag_c,
                                     const ChebCoef *cf_c, VT *d_c, VT *z_c, const Scalars *sc) {
  pdl_wait();
  if (sc && sc->done) return;
  const double inv_theta = cf_c->inv_theta;
  for (int64_t I = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; I < nc;
       I += (int64_t)gridDim.x * blockDim.x) {
    const VT acc = aggregate_sum(agg_ptr[I], agg_ptr[I + 1], agg_mem, res);
    rc[I] = acc;
    VT di = (VT)(inv_theta * (double)invdiag_c[I] * (double)acc);
    d_c[I] = di;
    z_c[I] = di;
  }
}

// Levels without A P (operators of at most kTailMaxNnz entries: a few microseconds
// of work each, bound by launches and by chains of dependent loads).
// Going down: the residual r - A z of an aggregate's rows, summed in member order
// (and the next level's zero-guess smoother start, INIT), in one launch: a warp per
// coarse row, W lanes per member row.  The row sums and the order of the members
// are those of resid_level_kernel and restrict_kernel, bit for bit.
template <int W, int U, typename T, bool INIT>
__global__ void __launch_bounds__(kBlock, kCoarseMinBlocks)
    resid_restrict_kernel(CsrView<T> A, const T *r, const T *z, int64_t nc,
                          const int64_t *agg_ptr, const int32_t *agg_mem, T *rc,
                          const T *invdiag_c, const ChebCoef *cf_c, T *d_c, T *z_c,
                          const Scalars *sc, int *wflag) {
  pdl_wait();
  if (sc && sc->done) {
    mark_work(wflag, 0);
    return;
  }
  mark_work(wflag, 1);
  constexpr int G = 32 / W;
  const int lane = threadIdx.x & 31, sub = lane % W, g = lane / W;
  const int64_t warp = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
  for (int64_t I = warp; I < nc; I += nwarps) {
    const int64_t m1 = agg_ptr[I + 1];
    T acc = T(0);
    for (int64_t mb = agg_ptr[I]; mb < m1; mb += G) {
      const bool active = mb + g < m1;
      const int32_t i = active ? agg_mem[mb + g] : 0;
      const int64_t b = active ? __ldg(A.ptr + i) : 0, e = active ? __ldg(A.ptr + i + 1) : 0;
      T ri = T(0), dg = T(0), zi = T(0);
      if (active && sub == 0) {
        ri = r[i];
        dg = A.diag[i];
        zi = z[i];
      }
      const T s = row_reduce<W>(row_dot_n<W, U, T, T>(b, e, A.col, A.val, GatherVec<T>{z}, sub,
                                                      tile_nmax<W>(b, e, sub)));
      const T res = ri - fmadd(dg, zi, s);  // of the group's row, in its first lane
      const int members = (int)(m1 - mb < G ? m1 - mb : G);
      for (int q = 0; q < members; ++q) acc += __shfl_sync(0xffffffffu, res, q * W);
    }
    if (lane == 0) {
      rc[I] = acc;
      if (INIT) {
        const T di = (T)(cf_c->inv_theta * (double)invdiag_c[I] * (double)acc);
        d_c[I] = di;
        z_c[I] = di;
      }
    }
  }
}

// Going up: the prolongation folded into the first post-smoothing step, z' = z + P e
// formed as it is gathered; z_out = z' + c2 D^{-1} (r - A z') in one launch (the
// cluster tail's arithmetic, bit for bit).
// DOT (finest level, degree 1): also the preconditioned inner product of DotFuse.
template <int W, int U, typename T, bool DOT>
__global__ void __launch_bounds__(kBlock, kCoarseMinBlocks)
    prolong_cheb_kernel(CsrView<T> A, const T *r, const T *z, const int32_t *agg, const T *ec,
                        T *z_out, T *d, const ChebCoef *cf, const Scalars *sc, int *wflag,
                        const DotFuse df) {
  pdl_wait();
  if (sc && sc->done) {
    mark_work(wflag, 0);
    return;
  }
  mark_work(wflag, 1);
  const T c2 = (T)cf->inv_theta;
  auto corrected = [&](int32_t c) {
    const T zc = __ldg(z + c);
    const int32_t a = __ldg(agg + c);
    return a >= 0 ? zc + __ldg(ec + a) : zc;
  };
  const int own = tile_own_row<W>(threadIdx.x & 31);
  int64_t r0, r1;
  warp_rows<W>(A.n, r0, r1);
  double da = 0.0, db = 0.0;
  for (int64_t base = r0; base < r1; base += 32) {
    const int rows = (int)(r1 - base < 32 ? r1 - base : 32);
    const int64_t i = base + own;
    const bool active = own < rows;
    T ri = T(0), zi = T(0), dg = T(0), idg = T(0);
    if (active) {
      ri = r[i];
      zi = corrected((int32_t)i);
      dg = A.diag[i];
      idg = A.invdiag[i];
    }
    const T s = tile_row_sums_of<W, U, T, T>(base, rows, A.ptr, A.col, A.val, corrected);
    if (active) {
      const T res = ri - fmadd(dg, zi, s);
      const T di = (c2 * idg) * res;
      const T zo = zi + di;
      d[i] = di;
      z_out[i] = zo;
      if (DOT) {
        const double rd = df.r[i], zn = widen(zo);
        if (df.flex) {
          if (!df.first) db += rd * df.z64[i];
          df.z64[i] = zn;
        }
        da += rd * zn;
      }
    }
  }
  if (DOT) {
    double part[2] = {da, db}, out[2];
    block_sums(part);
    const bool mx[2] = {false, false};
    if (last_block_combine<2>(part, df.partials, &df.sc->counter, out, mx) && threadIdx.x == 0) {
      Scalars *w = df.sc;
      if (!df.first) w->beta = (df.flex ? out[0] - out[1] : out[0]) / w->rho;
      w->rho = out[0];
    }
  }
}

// Coarsest level: the whole Chebyshev solve (zero guess, `degree` steps over
// [lo, hi]) in ONE block with the level's operator AND vectors staged in
// shared memory, so every step is a few shared-memory passes instead of a
// separate launch.  Used when the level fits (coarse_smem_bytes <= 200 KiB).
__host__ inline size_t coarse_smem_bytes(int64_t n, int64_t nnz, size_t mt, size_t vt) {
  size_t b = (size_t)nnz * (mt + 4) + (size_t)(n + 1) * 4 + (size_t)n * (2 * mt + 4 * vt);
  return (b + 15) & ~(size_t)15;
}
constexpr size_t kCoarseSmemMax = 200 * 1024;

// Body of the coarsest-level solve for one block (blockDim.x threads, the
// shared-memory buffer of coarse_smem_bytes(n, nnz, sizeof(VT), sizeof(VT)));
// also run by one block of the cluster-resident V-cycle tail.  MT / GT: type
// of the level's operator / vectors in global memory; VT: the type the solve
// is staged and computed in (the operator is converted when it is staged).
template <typename MT, typename VT, typename GT = VT>
__device__ void coarse_cheb_body(const CsrView<MT> &A, const GT *r_g, GT *z_g, const ChebCoef *cf,
                                 int degree, unsigned char *smem_raw) {
  const int n = (int)A.n, nnz = (int)A.nnz;
  // layout: values, diag, invdiag | r, z0, z1, d (all VT) | cols, ptr (int32)
  VT *val = reinterpret_cast<VT *>(smem_raw);
  VT *dg = val + nnz, *idg = dg + n;
  VT *r = reinterpret_cast<VT *>(idg + n);
  VT *zb0 = r + n, *zb1 = zb0 + n, *d = zb1 + n;
  int *col = reinterpret_cast<int *>(d + n);
  int *ptr = col + nnz;
  const int64_t base = A.ptr[0];
  const double inv_theta = cf->inv_theta;
  // the step coefficients, staged once: a global load per step would put an
  // L2 round trip on the critical path of every step
  __shared__ VT cs1[kChebMaxDeg], cs2[kChebMaxDeg];
  for (int k = threadIdx.x; k < degree && k < kChebMaxDeg; k += blockDim.x) {
    cs1[k] = (VT)cf->c1[k];
    cs2[k] = (VT)cf->c2[k];
  }
  for (int k = threadIdx.x; k < nnz; k += blockDim.x) {
    val[k] = (VT)A.val[base + k];
    col[k] = A.col[base + k];
  }
  for (int i = threadIdx.x; i <= n; i += blockDim.x) ptr[i] = (int)(A.ptr[i] - base);
  for (int i = threadIdx.x; i < n; i += blockDim.x) {
    dg[i] = (VT)A.diag[i];
    idg[i] = (VT)A.invdiag[i];
    VT ri = (VT)r_g[i];
    r[i] = ri;
    VT di = (VT)(inv_theta * (double)A.invdiag[i] * (double)ri);
    d[i] = di;
    zb0[i] = di;
  }
  __syncthreads();
  VT *zin = zb0, *zout = zb1;
  for (int k = 1; k < degree; ++k) {
    const VT c1 = cs1[k], c2 = cs2[k];
    for (int i = threadIdx.x; i < n; i += blockDim.x) {  // thread per row: no shuffles
      // 8 column / value loads, then 8 gathers in flight, summed in entry order
      VT s = 0;
      const int e = ptr[i + 1];
      for (int kk = ptr[i]; kk < e; kk += 8) {
        int cc[8];
        VT vv[8], zz[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) {
          cc[u] = kk + u < e ? col[kk + u] : -1;
          vv[u] = kk + u < e ? val[kk + u] : VT(0);
        }
#pragma unroll
        for (int u = 0; u < 8; ++u) zz[u] = cc[u] >= 0 ? zin[cc[u]] : VT(0);
#pragma unroll
        for (int u = 0; u < 8; ++u)
          if (cc[u] >= 0) s = fmadd(vv[u], zz[u], s);
      }
      VT res = r[i] - fmadd((VT)dg[i], zin[i], s);
      VT di = fmadd(c1, d[i], (c2 * (VT)idg[i]) * res);
      d[i] = di;
      zout[i] = zin[i] + di;
    }
    __syncthreads();
    VT *t = zin;
    zin = zout;
    zout = t;
  }
  for (int i = threadIdx.x; i < n; i += blockDim.x) z_g[i] = (GT)zin[i];
}

template <typename MT, typename VT, typename GT>
__global__ void __launch_bounds__(1024) coarse_cheb_kernel(CsrView<MT> A, const GT *r_g, GT *z_g,
                                                           const ChebCoef *cf, int degree,
                                                           const Scalars *sc) {
  pdl_wait();
  if (sc && sc->done) return;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  coarse_cheb_body<MT, VT, GT>(A, r_g, z_g, cf, degree, smem_raw);
}

// ---------------------------------------------------------------------------
// A P of the finest level.  After the coarse correction e_c, the first
// post-smoothing step needs r - A (z_pre + P e_c) = res - (A P) e_c, where
// res = r - A z_pre is the residual already formed before the restriction.
// A P has one entry per (fine row, distinct aggregate among the row's own
// and its columns' aggregates) -- about a sixth of A's entries -- so that
// step reads A P instead of A (and absorbs the prolongation).  Its entries
// are kept in first-occurrence order along the row (own aggregate first).
// ---------------------------------------------------------------------------
// structure, pass 1 (per fine row, one thread): distinct aggregates written
// uncompacted at tmp[ptr[i] + i ..], relative positions in ap_map / ap_dmap
__global__ void ap_structure_kernel(int64_t n, const int64_t *ptr, const int32_t *col,
                                    const int32_t *agg, int32_t *tmp, int64_t *cnt,
                                    int32_t *ap_map, int32_t *ap_dmap) {
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x) {
    int32_t *keys = tmp + ptr[i] + i;
    int32_t m = 0;
    const int32_t a0 = agg[i];
    if (a0 >= 0) keys[m++] = a0;
    ap_dmap[i] = a0 >= 0 ? 0 : -1;
    for (int64_t k = ptr[i]; k < ptr[i + 1]; ++k) {
      const int32_t K = agg[col[k]];
      int32_t pos = -1;
      if (K >= 0) {
        for (int32_t q = 0; q < m; ++q)
          if (keys[q] == K) {
            pos = q;
            break;
          }
        if (pos < 0) {
          pos = m;
          keys[m++] = K;
        }
      }
      ap_map[k] = pos;
    }
    cnt[i] = m;
  }
}
// The same pass with a warp per row: the row's entries are read 32 at a time
// (coalesced), equal aggregates within a batch are grouped with match_any, and
// a batch's new aggregates are appended in lane order after the keys of the
// earlier batches, which the warp keeps in shared memory -- so keys, positions
// and counts are exactly those of ap_structure_kernel.  A row with more than
// kApWarpKeys distinct aggregates sets *overflow; the caller then runs
// ap_structure_kernel instead.
constexpr int kApWarpKeys = 128;
__global__ void ap_structure_warp_kernel(int64_t n, const int64_t *ptr, const int32_t *col,
                                         const int32_t *agg, int32_t *tmp, int64_t *cnt,
                                         int32_t *ap_map, int32_t *ap_dmap, int *overflow) {
  __shared__ int32_t keys_sh[kWarpsPerBlock][kApWarpKeys];
  int32_t *ks = keys_sh[threadIdx.x >> 5];
  const int lane = threadIdx.x & 31;
  const unsigned lt = (1u << lane) - 1u;
  const int64_t warp = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
  for (int64_t i = warp; i < n; i += nwarps) {
    const int32_t a0 = agg[i];
    int m = 0;  // keys so far (warp-uniform)
    if (a0 >= 0) {
      if (lane == 0) ks[0] = a0;
      m = 1;
    }
    if (lane == 0) ap_dmap[i] = a0 >= 0 ? 0 : -1;
    __syncwarp();
    bool over = false;
    const int64_t b = ptr[i], e = ptr[i + 1];
    for (int64_t k0 = b; k0 < e; k0 += 32) {
      const int64_t k = k0 + lane;
      const bool valid = k < e;
      const int32_t K = valid ? agg[col[k]] : -1;
      int pos = -1;
      if (K >= 0)
        for (int q = 0; q < m; ++q)
          if (ks[q] == K) {
            pos = q;
            break;
          }
      // first lane of each group of equal new aggregates appends it
      const unsigned peers = __match_any_sync(0xffffffffu, K);
      const int leader = __ffs(peers) - 1;
      const bool fresh = K >= 0 && pos < 0;
      const bool adds = fresh && lane == leader;
      const unsigned newmask = __ballot_sync(0xffffffffu, adds);
      int mine = adds ? m + __popc(newmask & lt) : -1;
      if (adds && mine < kApWarpKeys) ks[mine] = K;
      mine = __shfl_sync(0xffffffffu, mine, leader);
      if (fresh) pos = mine;
      m += __popc(newmask);
      if (m > kApWarpKeys) {  // warp-uniform; the keys past the list were not kept
        over = true;
        break;
      }
      __syncwarp();
      if (valid) ap_map[k] = pos;
    }
    if (over) {
      if (lane == 0) *overflow = 1;
      continue;
    }
    int32_t *keys = tmp + b + i;
    for (int q = lane; q < m; q += 32) keys[q] = ks[q];
    if (lane == 0) cnt[i] = m;
    __syncwarp();
  }
}
// pass 2 (CSR rows only: the sources of each A P entry are then sorted by it):
// make the positions absolute, a warp per row
__global__ void ap_absolute_kernel(int64_t n, const int64_t *ptr, const int64_t *ap_ptr,
                                   int32_t *ap_map, int32_t *ap_dmap) {
  const int lane = threadIdx.x & 31;
  const int64_t warp = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
  for (int64_t i = warp; i < n; i += nwarps) {
    const int32_t b = (int32_t)ap_ptr[i];
    if (lane == 0 && ap_dmap[i] >= 0) ap_dmap[i] += b;
    const int64_t e = ptr[i + 1];
    for (int64_t k = ptr[i] + lane; k < e; k += 32)
      if (ap_map[k] >= 0) ap_map[k] += b;
  }
}
// The values (every step) are fixed-order sums of each entry's sources, the
// same gather-sum as the Galerkin product (galerkin_kernel).  The next
// level's operator P^T A P = P^T (A P) is then summed from the A P entries
// (about a sixth as many sources as A's entries): entry (i, K) of A P adds to
// coarse entry (agg[i], K), the diagonal when K = agg[i].
__global__ void ap_galerkin_target_kernel(int64_t n, const int64_t *ap_ptr, const int32_t *ap_col,
                                          const int32_t *agg, int64_t nnz_c, const int64_t *cptr,
                                          const int32_t *ccol, int32_t *tgt, int *missing) {
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x) {
    const int32_t I = agg[i];
    for (int64_t q = ap_ptr[i]; q < ap_ptr[i + 1]; ++q) {
      const int32_t K = ap_col[q];
      int64_t t = -1;
      if (I >= 0) {
        if (K == I) {
          t = nnz_c + I;
        } else {  // binary search in the sorted coarse row I
          int64_t lo = cptr[I], hi = cptr[I + 1];
          while (lo < hi) {
            const int64_t mid = (lo + hi) / 2;
            if (ccol[mid] < K) lo = mid + 1; else hi = mid;
          }
          if (lo < cptr[I + 1] && ccol[lo] == K) t = lo;
          else *missing = 1;
        }
      }
      tgt[q] = (int32_t)t;
    }
  }
}

// The same targets for A P in slices: tgt is in slice order (padding stays -1).
__global__ void ap_sliced_target_kernel(int64_t n, const int64_t *ap_ptr, const int32_t *ap_col,
                                        SlicedRowsData ap, const int32_t *agg, int64_t nnz_c,
                                        const int64_t *cptr, const int32_t *ccol, int32_t *tgt,
                                        int *missing) {
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x) {
    const int32_t I = agg[i];
    if (I < 0) continue;
    const int q0 = ap.place[i];
    const int64_t k0 = ap.ptr[i / kBlock * kWarpsPerBlock + q0 / 32] + q0 % 32;
    const int64_t b = ap_ptr[i], c0 = cptr[I], c1 = cptr[I + 1];
    for (int64_t q = b; q < ap_ptr[i + 1]; ++q) {
      const int32_t K = ap_col[q];
      int64_t t = nnz_c + I;
      if (K != I) {  // binary search in the sorted coarse row I
        int64_t lo = c0, hi = c1;
        while (lo < hi) {
          const int64_t mid = (lo + hi) / 2;
          if (ccol[mid] < K) lo = mid + 1; else hi = mid;
        }
        t = lo;
        if (lo >= c1 || ccol[lo] != K) {
          *missing = 1;
          t = -1;
        }
      }
      tgt[k0 + (q - b) * 32] = (int32_t)t;
    }
  }
}

// First post-smoothing step of a level with the prolongation folded in:
// z = z_pre + P e_c, res2 = res - (A P) e_c (= r - A z), d = c2 D^{-1} res2
// (step 0 from a nonzero guess), z_out = z + d.  z_out may be z_pre.
// DOT (finest level, smoother degree 1, where this is the V-cycle's last
// sweep): also the preconditioned inner product of DotFuse over the new z.
// Finest level (Rows over A P):
template <typename Rows, typename VT, bool DOT>
__global__ void __launch_bounds__(kBlock, Rows::kMinBlocks)
    fine_post_ap_kernel(Rows A, const int32_t *agg, const VT *ec, const VT *z_pre, const VT *res,
                        const VT *invdiag, const ChebCoef *cf, VT *d, VT *z_out,
                        const Scalars *sc, int *wflag, const DotFuse df) {
  pdl_wait();
  if (sc && sc->done) {
    mark_work(wflag, 0);
    return;
  }
  mark_work(wflag, 1);
  const VT c2 = (VT)cf->inv_theta;
  double da = 0.0, db = 0.0;  // (r, z) and (r, z_old) partials (DOT)
  A.each(
      ec,
      [&](int64_t i) {
        const int32_t a = agg[i];
        return Ops3<VT>{z_pre[i] + (a >= 0 ? ec[a] : VT(0)), c2 * invdiag[i], res[i]};
      },
      [&](int64_t i, VT s, const Ops3<VT> &o) {
        const VT di = o.b * (o.c - s);
        const VT zo = o.a + di;
        d[i] = di;
        z_out[i] = zo;
        if (DOT) {
          const double ri = df.r[i], zn = widen(zo);
          if (df.flex) {
            if (!df.first) db += ri * df.z64[i];
            df.z64[i] = zn;
          }
          da += ri * zn;
        }
      });
  if (DOT) {
    double part[2] = {da, db}, out[2];
    block_sums(part);
    const bool mx[2] = {false, false};
    if (last_block_combine<2>(part, df.partials, &df.sc->counter, out, mx) && threadIdx.x == 0) {
      Scalars *w = df.sc;
      if (!df.first) w->beta = (df.flex ? out[0] - out[1] : out[0]) / w->rho;
      w->rho = out[0];
    }
  }
}
// coarser levels (row operands before the row sums)
template <int W, int U, typename MT, typename VT>
__global__ void __launch_bounds__(kBlock, kCoarseMinBlocks)
    post_ap_kernel(int64_t n, const int64_t *ap_ptr, const int32_t *ap_col, const MT *ap_val,
                   const int32_t *agg, const VT *ec, const VT *z_pre, const VT *res,
                   const MT *invdiag, const ChebCoef *cf, VT *d, VT *z_out, const Scalars *sc) {
  pdl_wait();
  if (sc && sc->done) return;
  const VT c2 = (VT)cf->inv_theta;
  const int own = tile_own_row<W>(threadIdx.x & 31);
  int64_t r0, r1;
  warp_rows<W>(n, r0, r1);
  for (int64_t base = r0; base < r1; base += 32) {
    const int rows = (int)(r1 - base < 32 ? r1 - base : 32);
    const int64_t i = base + own;
    const bool active = own < rows;
    VT zp = VT(0), rs = VT(0), idg = VT(0), pe = VT(0);
    if (active) {
      zp = z_pre[i];
      rs = res[i];
      idg = (VT)invdiag[i];
      const int32_t a = agg[i];
      pe = a >= 0 ? ec[a] : VT(0);
    }
    const VT s = tile_row_sums<W, U, MT, VT>(base, rows, ap_ptr, ap_col, ap_val, ec);
    if (active) {
      const VT zi = zp + pe;
      const VT di = (c2 * idg) * (rs - s);
      d[i] = di;
      z_out[i] = zi + di;
    }
  }
}

// ---------------------------------------------------------------------------
// The finest level without post-smoothing, for the CG whose product comes from
// the V-cycle (config.fine_post_smooth = 0).  With the zero-guess smoother
// start z_pre = c0 D^{-1} r, the residual res = r - B z_pre (the V-cycle's
// first sweep) and the coarse correction e_c, the preconditioned residual is
// z = z_pre + P e_c, and
//   B z = B z_pre + (B P) e_c = (r - res) + (res - res2) = r - res2,
// res2 = res - (A P) e_c -- the A P sweep gives B z without a sweep of B.  The
// CG then needs no product sweep of its own: q = B p = B z + beta q_old.
// The sweep also forms the iteration's inner products, so alpha and beta are
// known when it ends (one reduction per iteration):
//   a = (r, z), b = (r, z_old), c = (z, B z), d = (z, q_old), e = (p_old, B z)
//   beta = (a - b) / rho_old     (flexible, Polak-Ribiere: the V-cycle without
//                                 post-smoothing is not symmetric)
//   (p, q) = (z + beta p_old, B z + beta q_old) = c + beta (d + e) + beta^2 (p_old, q_old)
//   alpha = a / (p, q)
// first = 1 (the first iteration of a solve): p = z, beta = 0, (p, q) = c.
// ---------------------------------------------------------------------------
__device__ __forceinline__ void fcg_scalars(const double (&o)[5], int first, Scalars *sc) {
  const double a = o[0];
  double beta = 0.0, pq = o[2];
  if (!first) {
    beta = (a - o[1]) / sc->rho;
    pq = o[2] + beta * (o[3] + o[4]) + beta * beta * sc->pq;
  }
  sc->beta = beta;
  sc->rho = a;
  sc->pq = pq;
  sc->pfirst = first;
  if (!(pq > 0.0) || !(pq < 1e308) || !(a == a)) {  // loss of definiteness or NaN
    sc->breakdown = 1;
    sc->done = 1;
  } else {
    sc->alpha = a / pq;
  }
}

// Row epilogue shared by the two forms of the last sweep: z and B z of row i
// and the five inner-product partials (zo, qo, po: the previous z, q, p).
template <typename VT>
__device__ __forceinline__ void fcg_row(int64_t i, VT zn, VT wn, VT r, VT zo, VT qo, VT po, VT *z,
                                        VT *w, int first, double (&acc)[5]) {
  const double ri = widen(r), zd = widen(zn), wd = widen(wn);
  acc[0] += ri * zd;
  acc[2] += zd * wd;
  if (!first) {
    acc[1] += ri * widen(zo);
    acc[3] += zd * widen(qo);
    acc[4] += widen(po) * wd;
  }
  z[i] = zn;
  w[i] = wn;
}

template <typename VT>
__device__ __forceinline__ void fcg_reduce(double (&acc)[5], int first, Scalars *sc,
                                           double *partials, const LoopCond &cond) {
  double out[5];
  block_sums(acc);
  const bool mx[5] = {false, false, false, false, false};
  if (last_block_combine<5>(acc, partials, &sc->counter, out, mx) && threadIdx.x == 0) {
    fcg_scalars(out, first, sc);
    loop_cond_set(cond, sc);
  }
}

// The A P sweep: res2 = res - (A P) e_c, z = z_pre + P e_c, B z = r - res2.
// (five FP64 partials on top of the row tile: compiled for the resident blocks
// per SM at which the register file holds them without spilling -- 4 with FP32
// vectors (64 registers), 3 with FP64 ones (72))
template <typename VT>
__host__ __device__ constexpr int fcg_min_blocks() {
  return sizeof(VT) == sizeof(float) ? 4 : 3;
}
template <typename Rows, typename VT>
__global__ void __launch_bounds__(kBlock, fcg_min_blocks<VT>())
    fine_ap_cg_kernel(Rows A, const int32_t *agg, const VT *ec, const VT *z_pre, const VT *res,
                      const VT *r, VT *z, VT *w, const VT *p, const VT *q, int first, Scalars *sc,
                      double *partials, int *wflag, const LoopCond cond) {
  pdl_wait();
  if (sc->done) {
    loop_cond_skip(cond, sc);
    mark_work(wflag, 0);
    return;
  }
  mark_work(wflag, 1);
  double acc[5] = {0.0, 0.0, 0.0, 0.0, 0.0};
  A.each(
      ec,
      [&](int64_t i) {
        const int32_t a = agg[i];
        const VT pe = a >= 0 ? ec[a] : VT(0);
        return Ops7<VT>{z_pre[i] + pe, res[i], r[i], first ? VT(0) : z[i],
                        first ? VT(0) : q[i], first ? VT(0) : p[i]};
      },
      [&](int64_t i, VT s, const Ops7<VT> &o) {
        const VT res2 = o.b - s;
        fcg_row<VT>(i, o.a, o.c - res2, o.c, o.d, o.e, o.f, z, w, first, acc);
      });
  fcg_reduce<VT>(acc, first, sc, partials, cond);
}

// Without A P (operators below the A P threshold): z = z_pre + P e_c into t,
// then B z by a sweep of B.
template <typename VT>
__global__ void fcg_prolong_kernel(int64_t n, const int32_t *agg, const VT *ec, const VT *z_pre,
                                   VT *t, const Scalars *sc) {
  pdl_wait();
  if (sc->done) return;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x) {
    const int32_t a = agg[i];
    t[i] = z_pre[i] + (a >= 0 ? ec[a] : VT(0));
  }
}
template <int W, int U, typename MT, typename VT>
__global__ void __launch_bounds__(kBlock, fcg_min_blocks<VT>())
    fcg_spmv_dot_kernel(CsrView<MT> A, const VT *t, const VT *r, VT *z, VT *w, const VT *p,
                        const VT *q, int first, Scalars *sc, double *partials, int *wflag,
                        const LoopCond cond) {
  pdl_wait();
  if (sc->done) {
    loop_cond_skip(cond, sc);
    mark_work(wflag, 0);
    return;
  }
  mark_work(wflag, 1);
  const int own = tile_own_row<W>(threadIdx.x & 31);
  int64_t r0, r1;
  warp_rows<W>(A.n, r0, r1);
  double acc[5] = {0.0, 0.0, 0.0, 0.0, 0.0};
  for (int64_t base = r0; base < r1; base += 32) {
    const int rows = (int)(r1 - base < 32 ? r1 - base : 32);
    const int64_t i = base + own;
    const VT s = tile_row_sums<W, U, MT, VT>(base, rows, A.ptr, A.col, A.val, t);
    if (own < rows) {
      const VT ti = t[i];
      fcg_row<VT>(i, ti, fmadd((VT)A.diag[i], ti, s), r[i], first ? VT(0) : z[i],
                  first ? VT(0) : q[i], first ? VT(0) : p[i], z, w, first, acc);
    }
  }
  fcg_reduce<VT>(acc, first, sc, partials, cond);
}

// ---------------------------------------------------------------------------
// Cluster-resident V-cycle tail: the levels from `tail_level` down (small
// operators that live in L2) run as ONE launch of one thread-block cluster.
// Phases that depend on other rows are separated by cluster barriers instead
// of kernel boundaries, so a small level costs a few barrier round trips
// instead of several launches.  Rows of a level are split into contiguous
// ranges, one per block; every phase repeats the arithmetic of the per-level
// kernels exactly (same W-lane row sums, same update expressions, same
// restriction order), so the result is bitwise that of the launched V-cycle.
// Vectors written inside the launch are read with L2 (.cg) loads.  All
// control flow is uniform over the cluster: every block passes every barrier.
// ---------------------------------------------------------------------------
template <typename T>
struct TailLevel {
  CsrView<T> A;
  const int32_t *agg;      // [n] row of the next level (-1: unaggregated)
  const int64_t *agg_ptr;  // [n_next + 1] members of each next-level row
  const int32_t *agg_mem;
  T *r, *z, *res, *d, *t;
  const ChebCoef *cf;
  int deg;
};
template <typename T>
struct TailParams {
  int nlev;        // levels in the tail; the last one is the coarsest
  int coarse_smem; // 1: the coarsest solve runs in block 0 from shared memory
  int coarse_fp32; // 1: that solve is staged and computed in FP32
  TailLevel<T> L[kMaxLevels];
};

template <int W, typename MT, typename VT>
__device__ __forceinline__ VT row_dot_cg(int64_t beg, int64_t end, const int32_t *__restrict__ col,
                                         const MT *__restrict__ val, const VT *x, int sub) {
  constexpr int U = 4;
  VT s = VT(0);
  for (int64_t k = beg + sub; k < end; k += (int64_t)W * U) {
    int32_t c[U];
    MT v[U];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int64_t kk = k + (int64_t)u * W;
      c[u] = kk < end ? __ldg(col + kk) : -1;
      v[u] = kk < end ? __ldg(val + kk) : MT(0);
    }
#pragma unroll
    for (int u = 0; u < U; ++u)
      if (c[u] >= 0) s = fmadd((VT)v[u], __ldcg(x + c[u]), s);
  }
  return s;
}

// f(i, s) for the rows [r0, r1) of this block, s = sum_j A_ij x_j (off-diagonal)
template <int W, typename T, typename F>
__device__ __forceinline__ void tail_rows(const CsrView<T> &A, const T *x, int64_t r0, int64_t r1,
                                          F &&f) {
  const int sub = threadIdx.x % W;
  const int64_t grp = threadIdx.x / W, ngrp = blockDim.x / W;
  for (int64_t wb = r0 + warp_first_group<W>(grp); wb < r1; wb += ngrp) {
    const int64_t i = wb + group_in_warp<W>(grp);
    const bool active = i < r1;
    T s = active ? row_dot_cg<W, T, T>(__ldg(A.ptr + i), __ldg(A.ptr + i + 1), A.col, A.val, x,
                                       sub)
                 : T(0);
    s = row_reduce<W>(s);
    if (active && sub == 0) f(i, s);
  }
}
template <typename T, typename F>
__device__ __forceinline__ void tail_rows_w(const CsrView<T> &A, const T *x, int64_t r0,
                                            int64_t r1, F &&f) {
  if (A.W <= 4)
    tail_rows<4>(A, x, r0, r1, f);
  else
    tail_rows<8>(A, x, r0, r1, f);
}

// Chebyshev step k of a level (cheb_step_kernel's arithmetic) on this block's rows
template <typename T>
__device__ __forceinline__ void tail_cheb_step(const TailLevel<T> &L, const T *zin, T *zout,
                                               int k, int64_t r0, int64_t r1) {
  const double c1 = k > 0 ? L.cf->c1[k] : 0.0, c2 = k > 0 ? L.cf->c2[k] : L.cf->inv_theta;
  const T vc1 = (T)c1, vc2 = (T)c2;
  tail_rows_w(L.A, zin, r0, r1, [&](int64_t i, T s) {
    T zi = __ldcg(zin + i);
    T res = __ldcg(L.r + i) - fmadd((T)L.A.diag[i], zi, s);
    T di = (vc2 * (T)L.A.invdiag[i]) * res;
    if (k > 0) di = fmadd(vc1, __ldcg(L.d + i), di);
    L.d[i] = di;
    zout[i] = zi + di;
  });
}

template <typename T>
__global__ void __launch_bounds__(1024, 1) vcycle_tail_kernel(const __grid_constant__ TailParams<T> P,
                                                              const Scalars *sc) {
  if (sc && sc->done) return;  // uniform: nothing in this launch writes `done`
  extern __shared__ __align__(16) unsigned char smem_raw[];
  cg::cluster_group cl = cg::this_cluster();
  const int64_t cb = cl.block_rank(), nb = cl.num_blocks();
  auto lo = [&](int64_t n) { return n * cb / nb; };
  auto hi = [&](int64_t n) { return n * (cb + 1) / nb; };
  // Chebyshev from a zero guess over `deg` steps, result in z (cheb_apply's ping-pong)
  auto cheb_zero = [&](const TailLevel<T> &L, int deg) {
    T *bufs[2] = {L.z, L.t};
    const int w0 = (deg - 1) % 2;
    const int64_t r0 = lo(L.A.n), r1 = hi(L.A.n);
    const double inv_theta = L.cf->inv_theta;
    for (int64_t i = r0 + threadIdx.x; i < r1; i += blockDim.x) {
      T di = (T)(inv_theta * (double)L.A.invdiag[i] * (double)__ldcg(L.r + i));
      L.d[i] = di;
      bufs[w0][i] = di;
    }
    cl.sync();
    int at = w0;
    for (int k = 1; k < deg; ++k) {
      tail_cheb_step(L, bufs[at], bufs[at ^ 1], k, r0, r1);
      cl.sync();
      at ^= 1;
    }
  };
  const int last = P.nlev - 1;
  // down: pre-smoothing, residual, restriction
  for (int l = 0; l < last; ++l) {
    const TailLevel<T> &L = P.L[l];
    const TailLevel<T> &C = P.L[l + 1];
    cheb_zero(L, L.deg);
    const int64_t r0 = lo(L.A.n), r1 = hi(L.A.n);
    tail_rows_w(L.A, L.z, r0, r1, [&](int64_t i, T s) {
      L.res[i] = __ldcg(L.r + i) - fmadd((T)L.A.diag[i], __ldcg(L.z + i), s);
    });
    cl.sync();
    for (int64_t I = lo(C.A.n) + threadIdx.x; I < hi(C.A.n); I += blockDim.x) {
      T acc = 0;
      for (int64_t m = L.agg_ptr[I]; m < L.agg_ptr[I + 1]; ++m) acc += __ldcg(L.res + L.agg_mem[m]);
      C.r[I] = acc;
    }
    cl.sync();
  }
  // coarsest level
  {
    const TailLevel<T> &L = P.L[last];
    if (P.coarse_smem) {
      if (cb == 0) {
        if (P.coarse_fp32)
          coarse_cheb_body<T, float, T>(L.A, L.r, L.z, L.cf, L.deg, smem_raw);
        else
          coarse_cheb_body<T, T, T>(L.A, L.r, L.z, L.cf, L.deg, smem_raw);
      }
      cl.sync();
    } else {
      cheb_zero(L, L.deg);
    }
  }
  // up: prolongation, post-smoothing from the corrected guess
  for (int l = last - 1; l >= 0; --l) {
    const TailLevel<T> &L = P.L[l];
    const TailLevel<T> &C = P.L[l + 1];
    const int64_t r0 = lo(L.A.n), r1 = hi(L.A.n);
    for (int64_t i = r0 + threadIdx.x; i < r1; i += blockDim.x) {
      int32_t a = L.agg[i];
      if (a >= 0) L.z[i] = __ldcg(L.z + i) + __ldcg(C.z + a);
    }
    cl.sync();
    T *bufs[2] = {L.z, L.t};
    const int w0 = (L.deg - 1) % 2;
    if (w0 == 0) {  // the guess is read from bufs[1]
      for (int64_t i = r0 + threadIdx.x; i < r1; i += blockDim.x) L.t[i] = __ldcg(L.z + i);
      cl.sync();
    }
    tail_cheb_step(L, bufs[w0 ^ 1], bufs[w0], 0, r0, r1);
    cl.sync();
    int at = w0;
    for (int k = 1; k < L.deg; ++k) {
      tail_cheb_step(L, bufs[at], bufs[at ^ 1], k, r0, r1);
      cl.sync();
      at ^= 1;
    }
  }
}

// ---------------------------------------------------------------------------
// host: structure
// ---------------------------------------------------------------------------
CsrView<double> fine_view(const sph_rt *s);
sph_rt_status launch_assembly(sph_rt *s, double dt, double *gersh_out);


// bucket sort of ids by bucket[i] into (start, out); nb buckets
template <typename S>
static sph_rt_status bucket_sort(sph_rt *s, SphLevel *owner, int64_t nitems,
                                 const int32_t *bucket, int64_t nb, int64_t **start_out,
                                 S **out_out, int64_t *total_out) {
  unsigned *cnt = scratch<unsigned>(s, nb + 1), *cur = scratch<unsigned>(s, nb + 1);
  int64_t *cnt64 = scratch<int64_t>(s, nb + 1);
  if (!cnt || !cur || !cnt64) return SPH_RT_ENOMEM;
  int64_t *start = lalloc<int64_t>(s, owner, nb + 1);
  if (!start) return SPH_RT_ENOMEM;
  SPH_CUDA(s, cudaMemsetAsync(cnt, 0, sizeof(unsigned) * (nb + 1), s->stream));
  SPH_CUDA(s, cudaMemsetAsync(cur, 0, sizeof(unsigned) * (nb + 1), s->stream));
  target_count_kernel<<<gcap(s, nitems, kBlock), kBlock, 0, s->stream>>>(nitems, bucket, cnt);
  SPH_LAUNCHED(s);
  u32_to_i64_kernel<<<gcap(s, nb, kBlock), kBlock, 0, s->stream>>>(nb, cnt, cnt64);
  SPH_LAUNCHED(s);
  sph_rt_status rc = exclusive_scan(s, cnt64, nb, start);
  if (rc) return rc;
  int64_t total = 0;
  SPH_CUDA(s, cudaMemcpyAsync(&total, start + nb, sizeof(int64_t), cudaMemcpyDeviceToHost, s->stream));
  SPH_CUDA(s, cudaStreamSynchronize(s->stream));
  S *out = lalloc<S>(s, owner, total);
  if (!out) return SPH_RT_ENOMEM;
  bucket_scatter_kernel<S><<<gcap(s, nitems, kBlock), kBlock, 0, s->stream>>>(nitems, bucket,
                                                                             start, cur, out);
  SPH_LAUNCHED(s);
  bucket_sort_kernel<S><<<gcap(s, nb, kBlock), kBlock, 0, s->stream>>>(nb, start, out);
  SPH_LAUNCHED(s);
  bucket_rank_kernel<S><<<gcap(s, ceil_div(nb, 32), kWarpsPerBlock), kBlock, 0, s->stream>>>(
      nb, start, out);
  SPH_LAUNCHED(s);
  SPH_CUDA(s, cudaStreamSynchronize(s->stream));
  dfree(s, cnt);
  dfree(s, cur);
  dfree(s, cnt64);
  *start_out = start;
  *out_out = out;
  if (total_out) *total_out = total;
  return SPH_RT_OK;
}

// Galerkin source lists over nitems = nnz + n sources: 64-bit indices when
// they do not fit 32 bits (or config.index64), else 32-bit.
static sph_rt_status source_sort(sph_rt *s, SphLevel *owner, int64_t nitems,
                                 const int32_t *bucket, int64_t nb, int64_t **start_out,
                                 SrcList *out) {
  *out = SrcList{};
  if (s->cfg.index64 || nitems >= ((int64_t)1 << 31) - 1)
    return bucket_sort<int64_t>(s, owner, nitems, bucket, nb, start_out, &out->i64, nullptr);
  return bucket_sort<int32_t>(s, owner, nitems, bucket, nb, start_out, &out->i32, nullptr);
}

template <typename T>
static sph_rt_status launch_galerkin(sph_rt *s, int64_t nnz_c, int64_t nc, const int64_t *seg_ptr,
                            const SrcList &src, int64_t nnz_f, const T *val_f, const T *diag_f,
                            T *val_c, T *diag_c, T *invdiag_c) {
  const int g = gcap(s, nnz_c + nc, kBlock);
  if (src.i64)
    galerkin_kernel<T, int64_t><<<g, kBlock, 0, s->stream>>>(nnz_c, nc, seg_ptr, src.i64, nnz_f,
                                                             val_f, diag_f, val_c, diag_c,
                                                             invdiag_c);
  else
    galerkin_kernel<T, int32_t><<<g, kBlock, 0, s->stream>>>(nnz_c, nc, seg_ptr, src.i32, nnz_f,
                                                             val_f, diag_f, val_c, diag_c,
                                                             invdiag_c);
  SPH_LAUNCHED(s);
  return SPH_RT_OK;
}

__global__ void max_len_kernel(int64_t n, const int32_t *len, int *most) {
  int m = 0;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x)
    m = max(m, len[i]);
  m = __reduce_max_sync(0xffffffffu, m);
  if ((threadIdx.x & 31) == 0) atomicMax(most, m);
}

// Slices of the finest level's A P from its CSR rows.  Where they have no dictionary
// within the caps, the set-up fails as it does without memory for them, and amg_setup
// starts again from CSR rows.
static void *take_level(sph_rt *s, void *L, size_t bytes) {
  return lvl_alloc(s, static_cast<SphLevel *>(L), bytes);
}
static sph_rt_status build_ap_slices(sph_rt *s, SphLevel *L) {
  bool ok = false;
  sph_rt_status rc = sliced_build(s, L->n, L->ap_ptr, L->ap_col, nullptr, take_level, L, &L->ap_sl,
                                  nullptr, &ok);
  if (rc) return rc;
  int *most = scratch<int>(s, 1);
  if (!most) return SPH_RT_ENOMEM;
  SPH_CUDA(s, cudaMemsetAsync(most, 0, sizeof(int), s->stream));
  if (ok) {
    max_len_kernel<<<gcap(s, L->n, kBlock), kBlock, 0, s->stream>>>(L->n, L->ap_sl.len, most);
    SPH_LAUNCHED(s);
  }
  SPH_CUDA(s, cudaMemcpyAsync(&L->ap_most, most, sizeof(int), cudaMemcpyDeviceToHost, s->stream));
  SPH_CUDA(s, cudaStreamSynchronize(s->stream));
  dfree(s, most);
  if (!ok || L->ap_most >= kNoPlace || s->test_refuse_ap)
    return set_error(s, SPH_RT_ENOMEM, "A P does not fit the sliced layout");
  const size_t size = (size_t)L->ap_sl.padded + 1;
  if (s->cfg.precision == SPH_RT_MIXED)
    L->ap_val32 = lalloc<float>(s, L, size);
  else
    L->ap_val = lalloc<double>(s, L, size);
  return L->ap_val || L->ap_val32 ? SPH_RT_OK : SPH_RT_ENOMEM;
}

// structure of A P of the last level so far (see ap_structure_kernel)
static sph_rt_status build_ap(sph_rt *s) {
  const size_t l = s->levels.size() - 1;
  SphLevel *L = s->levels[l];
  const int64_t n = L->n;
  int32_t *tmp = scratch<int32_t>(s, (size_t)(L->nnz + n));
  int64_t *cnt = scratch<int64_t>(s, (size_t)n + 1);
  // target A P entry of each source: off-diagonal entries, then the diagonals
  int32_t *map = scratch<int32_t>(s, (size_t)(L->nnz + n));
  L->ap_ptr = lalloc<int64_t>(s, L, n + 1);
  if (!tmp || !cnt || !map || !L->ap_ptr) return SPH_RT_ENOMEM;
  int32_t *dmap = map + L->nnz;
  int *ovf = scratch<int>(s, 1);
  if (!ovf) return SPH_RT_ENOMEM;
  SPH_CUDA(s, cudaMemsetAsync(ovf, 0, sizeof(int), s->stream));
  ap_structure_warp_kernel<<<gcap(s, n, kWarpsPerBlock), kBlock, 0, s->stream>>>(
      n, L->ptr, L->col, L->agg, tmp, cnt, map, dmap, ovf);
  SPH_LAUNCHED(s);
  int h_ovf = 0;
  SPH_CUDA(s, cudaMemcpyAsync(&h_ovf, ovf, sizeof(int), cudaMemcpyDeviceToHost, s->stream));
  SPH_CUDA(s, cudaStreamSynchronize(s->stream));
  dfree(s, ovf);
  if (h_ovf) {  // a row with more distinct aggregates than the warp keeps: one thread a row
    ap_structure_kernel<<<gcap(s, n, kBlock), kBlock, 0, s->stream>>>(n, L->ptr, L->col, L->agg,
                                                                      tmp, cnt, map, dmap);
    SPH_LAUNCHED(s);
  }
  sph_rt_status rc;
  const bool sliced = l == 0 && s->sl.ptr != nullptr;
  if (sliced) {  // the relative places, before they are made absolute
    L->ap_pos = lalloc<uint16_t>(s, L, (size_t)s->sl.padded + 1);
    if (!L->ap_pos) return SPH_RT_ENOMEM;
    if ((rc = sliced_places(s, map, L->ap_pos))) return rc;
  }
  if ((rc = exclusive_scan(s, cnt, n, L->ap_ptr))) return rc;
  int64_t total = 0;
  SPH_CUDA(s, cudaMemcpyAsync(&total, L->ap_ptr + n, sizeof(int64_t), cudaMemcpyDeviceToHost,
                              s->stream));
  SPH_CUDA(s, cudaStreamSynchronize(s->stream));
  if (total >= ((int64_t)1 << 31)) return set_error(s, SPH_RT_EINVAL, "A P too large");
  L->nnz_ap = total;
  L->ap_col = lalloc<int32_t>(s, L, (size_t)total);
  if (!L->ap_col) return SPH_RT_ENOMEM;
  const int gw = gcap(s, n, kWarpsPerBlock);  // a warp per row
  ap_offset_kernel<<<gcap(s, n, kBlock), kBlock, 0, s->stream>>>(n, L->ptr, cnt);
  SPH_LAUNCHED(s);
  compact_rows_kernel<<<gw, kBlock, 0, s->stream>>>(n, cnt, tmp, L->ap_ptr, L->ap_col);
  SPH_LAUNCHED(s);
  if (sliced) {
    if ((rc = build_ap_slices(s, L))) return rc;
  } else {
    L->ap_val = lalloc<double>(s, L, (size_t)total);
    if (!L->ap_val) return SPH_RT_ENOMEM;
    if (s->cfg.precision == SPH_RT_MIXED && !(L->ap_val32 = lalloc<float>(s, L, (size_t)total)))
      return SPH_RT_ENOMEM;
    ap_absolute_kernel<<<gw, kBlock, 0, s->stream>>>(n, L->ptr, L->ap_ptr, map, dmap);
    SPH_LAUNCHED(s);
    // sources of each A P entry in increasing source order
    if ((rc = source_sort(s, L, L->nnz + n, map, total, &L->ap_seg_ptr, &L->ap_seg_src)))
      return rc;
  }
  SPH_CUDA(s, cudaStreamSynchronize(s->stream));
  dfree(s, tmp);
  dfree(s, cnt);
  dfree(s, map);
  return SPH_RT_OK;
}

// The next level's sparsity from the rows of A P.  *overflow: a coarse row is too
// wide for the block kernel's table too (the level is then not built).
static sph_rt_status coarse_from_ap(sph_rt *s, SphLevel *L, SphLevel *C, int64_t *ccount,
                                    int *overflow) {
  const int64_t nc = C->n;
  cudaStream_t st = s->stream;
  int64_t *bound = scratch<int64_t>(s, nc), *off = scratch<int64_t>(s, nc + 1);
  int32_t *cols = scratch<int32_t>(s, (size_t)L->nnz_ap + 1);
  int *flags = scratch<int>(s, 2);  // wide, overflow
  if (!bound || !off || !cols || !flags) return SPH_RT_ENOMEM;
  SPH_CUDA(s, cudaMemsetAsync(flags, 0, 2 * sizeof(int), st));
  member_bound_kernel<<<gcap(s, nc, kBlock), kBlock, 0, st>>>(nc, L->agg_ptr, L->agg_mem,
                                                             L->ap_ptr, bound);
  SPH_LAUNCHED(s);
  sph_rt_status rc = exclusive_scan(s, bound, nc, off);
  if (rc) return rc;
  coarse_rows_kernel<<<(int)std::min<int64_t>(ceil_div(nc, kCoarseRowWarps), s->num_sms * 9),
                       32 * kCoarseRowWarps, 0, st>>>(nc, L->agg_ptr, L->agg_mem, L->ap_ptr,
                                                      L->ap_col, off, cols, ccount, flags);
  SPH_LAUNCHED(s);
  int hf[2] = {0, 0};
  SPH_CUDA(s, cudaMemcpyAsync(hf, flags, sizeof hf, cudaMemcpyDeviceToHost, st));
  SPH_CUDA(s, cudaStreamSynchronize(st));
  const int gb = (int)std::min<int64_t>(nc, (int64_t)s->num_sms * 16);
  if (hf[0]) {
    coarse_struct_kernel<false><<<gb, kBlock, 0, st>>>(nc, L->agg_ptr, L->agg_mem, L->ap_ptr,
                                                       L->ap_col, nullptr, ccount, nullptr, nullptr,
                                                       nullptr, 0, nullptr, flags + 1);
    SPH_LAUNCHED(s);
    SPH_CUDA(s, cudaMemcpyAsync(hf, flags, sizeof hf, cudaMemcpyDeviceToHost, st));
    SPH_CUDA(s, cudaStreamSynchronize(st));
  }
  *overflow = hf[1];
  if (!hf[1]) {
    if ((rc = exclusive_scan(s, ccount, nc, C->ptr))) return rc;
    SPH_CUDA(s, cudaMemcpyAsync(&C->nnz, C->ptr + nc, sizeof(int64_t), cudaMemcpyDeviceToHost, st));
    SPH_CUDA(s, cudaStreamSynchronize(st));
    C->col = lalloc<int32_t>(s, C, C->nnz);
    if (!C->col) return SPH_RT_ENOMEM;
    if (hf[0])
      coarse_struct_kernel<true><<<gb, kBlock, 0, st>>>(nc, L->agg_ptr, L->agg_mem, L->ap_ptr,
                                                        L->ap_col, nullptr, nullptr, C->ptr, C->col,
                                                        nullptr, C->nnz, nullptr, flags + 1);
    else
      compact_rows_kernel<<<gcap(s, nc, kWarpsPerBlock), kBlock, 0, st>>>(nc, off, cols, C->ptr,
                                                                          C->col);
    SPH_LAUNCHED(s);
  }
  SPH_CUDA(s, cudaStreamSynchronize(st));
  dfree(s, bound);
  dfree(s, off);
  dfree(s, cols);
  dfree(s, flags);
  return SPH_RT_OK;
}

// values and vectors of a coarse level
static sph_rt_status coarse_storage(sph_rt *s, SphLevel *C) {
  const int64_t nc = C->n;
  C->val = lalloc<double>(s, C, C->nnz);
  C->diag = lalloc<double>(s, C, nc);
  C->invdiag = lalloc<double>(s, C, nc);
  C->r = lalloc<double>(s, C, nc);
  C->z = lalloc<double>(s, C, nc);
  C->res = lalloc<double>(s, C, nc);
  C->d = lalloc<double>(s, C, nc);
  C->t = lalloc<double>(s, C, nc);
  if (!C->val || !C->diag || !C->invdiag || !C->r || !C->z || !C->res || !C->d || !C->t)
    return SPH_RT_ENOMEM;
  {
    RowShape sh = shape_for_mean(nc ? (double)C->nnz / (double)nc : 0.0);
    C->W = sh.W;
    C->U = sh.U;
  }
  return SPH_RT_OK;
}

// Lists of the next level's sums over A P entries.
static sph_rt_status build_apg(sph_rt *s, SphLevel *L, SphLevel *C) {
  const int64_t n = L->n, total = L->nnz_ap;
  sph_rt_status rc;
  // next level's Galerkin sources: the A P entries of its members' rows, numbered
  // as they are stored
  const int64_t stored = L->ap_sl.ptr ? L->ap_sl.padded : total;
  int32_t *tgt = scratch<int32_t>(s, (size_t)stored + 1);
  int *missing = scratch<int>(s, 1);
  if (!tgt || !missing) return SPH_RT_ENOMEM;
  SPH_CUDA(s, cudaMemsetAsync(missing, 0, sizeof(int), s->stream));
  if (L->ap_sl.ptr) {
    fill_i32_kernel<<<gcap(s, stored, kBlock), kBlock, 0, s->stream>>>(stored, -1, tgt);
    SPH_LAUNCHED(s);
    ap_sliced_target_kernel<<<gcap(s, n, kBlock), kBlock, 0, s->stream>>>(
        n, L->ap_ptr, L->ap_col, L->ap_sl, L->agg, C->nnz, C->ptr, C->col, tgt, missing);
  } else {
    ap_galerkin_target_kernel<<<gcap(s, n, kBlock), kBlock, 0, s->stream>>>(
        n, L->ap_ptr, L->ap_col, L->agg, C->nnz, C->ptr, C->col, tgt, missing);
  }
  SPH_LAUNCHED(s);
  if ((rc = bucket_sort<int32_t>(s, L, stored, tgt, C->nnz + C->n, &L->apg_ptr, &L->apg_src,
                                 nullptr)))
    return rc;
  int miss = 0;
  SPH_CUDA(s, cudaMemcpyAsync(&miss, missing, sizeof(int), cudaMemcpyDeviceToHost, s->stream));
  SPH_CUDA(s, cudaStreamSynchronize(s->stream));
  dfree(s, tgt);
  dfree(s, missing);
  if (miss) return set_error(s, SPH_RT_EDEVICE, "A P entry outside the coarse sparsity");
  return SPH_RT_OK;
}

// Aggregate level L and build the next level's sparsity plus the Galerkin
// contribution lists: through A P on the levels above kTailMaxNnz entries (~a
// third of the sources, and no list over the operator's own entries), else from
// the level's entries.  Returns the new level in *next (nullptr: stop).
static sph_rt_status coarsen(sph_rt *s, SphLevel *L, SphLevel **next) {
  *next = nullptr;
  const int64_t n = L->n, nnz = L->nnz;
  cudaStream_t st = s->stream;
  uint8_t *strong = scratch<uint8_t>(s, nnz), *cand = scratch<uint8_t>(s, n);
  int *state = scratch<int>(s, n);
  int64_t *flag = scratch<int64_t>(s, n), *root_id = scratch<int64_t>(s, n + 1);
  unsigned *undec = scratch<unsigned>(s, 1), *members = nullptr;
  if (!strong || !cand || !state || !flag || !root_id || !undec) return SPH_RT_ENOMEM;
  auto cleanup = [&]() {
    cudaStreamSynchronize(s->stream);
    dfree(s, strong);
    dfree(s, cand);
    dfree(s, state);
    dfree(s, flag);
    dfree(s, root_id);
    dfree(s, undec);
    if (members) dfree(s, members);
  };
  const int g = gcap(s, n, kBlock);
  const int gw = gcap(s, n, kWarpsPerBlock);  // a warp per row
  strength_kernel<<<gw, kBlock, 0, st>>>(n, L->ptr, L->col, L->val, L->diag,
                                        s->cfg.amg_theta * s->cfg.amg_theta,
                                        strong, state);
  SPH_LAUNCHED(s);
  for (int round = 0; round < 200; ++round) {
    mis_select_kernel<<<gw, kBlock, 0, st>>>(n, L->ptr, L->col, strong, state, cand);
    SPH_LAUNCHED(s);
    mis_apply_kernel<<<g, kBlock, 0, st>>>(n, cand, state);
    SPH_LAUNCHED(s);
    SPH_CUDA(s, cudaMemsetAsync(undec, 0, sizeof(unsigned), st));
    mis_mark_kernel<<<gw, kBlock, 0, st>>>(n, L->ptr, L->col, strong, state, undec);
    SPH_LAUNCHED(s);
    unsigned left = 0;
    SPH_CUDA(s, cudaMemcpyAsync(&left, undec, sizeof(unsigned), cudaMemcpyDeviceToHost, st));
    SPH_CUDA(s, cudaStreamSynchronize(st));
    if (left == 0) break;
  }
  root_flag_kernel<<<g, kBlock, 0, st>>>(n, state, flag);
  SPH_LAUNCHED(s);
  sph_rt_status rc = exclusive_scan(s, flag, n, root_id);
  if (rc) return cleanup(), rc;
  int64_t nc = 0;
  SPH_CUDA(s, cudaMemcpyAsync(&nc, root_id + n, sizeof(int64_t), cudaMemcpyDeviceToHost, st));
  SPH_CUDA(s, cudaStreamSynchronize(st));
  if (nc == 0 || nc * 10 > n * 9) {  // nothing to coarsen, or coarsening too slow
    cleanup();
    return SPH_RT_OK;
  }
  members = scratch<unsigned>(s, nc);
  if (!members) return cleanup(), SPH_RT_ENOMEM;
  SPH_CUDA(s, cudaMemsetAsync(members, 0, sizeof(unsigned) * nc, st));
  L->agg = lalloc<int32_t>(s, L, n);
  if (!L->agg) return cleanup(), SPH_RT_ENOMEM;
  assign_kernel<<<gw, kBlock, 0, st>>>(n, L->ptr, L->col, L->val, strong, state, root_id, L->agg,
                                      members);
  SPH_LAUNCHED(s);
  cleanup();
  members = nullptr;
  // member lists of the coarse rows
  int64_t tot = 0;
  if ((rc = bucket_sort<int32_t>(s, L, n, L->agg, nc, &L->agg_ptr, &L->agg_mem, &tot))) return rc;

  SphLevel *C = new SphLevel();
  C->n = nc;
  // coarse sparsity: count, scan, fill (+ Galerkin targets of every fine entry)
  int64_t *ccount = lalloc<int64_t>(s, C, nc);
  C->ptr = lalloc<int64_t>(s, C, nc + 1);
  if (!ccount || !C->ptr) return SPH_RT_ENOMEM;
  auto drop = [&]() {  // stop coarsening here
    for (void *p : C->owned) dfree(s, p);
    delete C;
    return SPH_RT_OK;
  };
  if (nnz > kTailMaxNnz) {
    if ((rc = build_ap(s))) return rc;
    int ovf = 0;
    if ((rc = coarse_from_ap(s, L, C, ccount, &ovf))) return rc;
    if (ovf) return drop();
    if ((rc = build_apg(s, L, C))) return rc;
    if ((rc = coarse_storage(s, C))) return rc;
    *next = C;
    return SPH_RT_OK;
  }
  int *overflow = scratch<int>(s, 1);
  if (!overflow) return SPH_RT_ENOMEM;
  SPH_CUDA(s, cudaMemsetAsync(overflow, 0, sizeof(int), st));
  int gb = (int)std::min<int64_t>(nc, (int64_t)s->num_sms * 16);
  coarse_struct_kernel<false><<<gb, kBlock, 0, st>>>(nc, L->agg_ptr, L->agg_mem, L->ptr, L->col,
                                                     L->agg, ccount, nullptr, nullptr, nullptr, 0,
                                                     nullptr, overflow);
  SPH_LAUNCHED(s);
  int ovf = 0;
  SPH_CUDA(s, cudaMemcpyAsync(&ovf, overflow, sizeof(int), cudaMemcpyDeviceToHost, st));
  SPH_CUDA(s, cudaStreamSynchronize(st));
  if (ovf) {
    dfree(s, overflow);
    return drop();
  }
  if ((rc = exclusive_scan(s, ccount, nc, C->ptr))) return rc;
  SPH_CUDA(s, cudaMemcpyAsync(&C->nnz, C->ptr + nc, sizeof(int64_t), cudaMemcpyDeviceToHost, st));
  SPH_CUDA(s, cudaStreamSynchronize(st));
  C->col = lalloc<int32_t>(s, C, C->nnz);
  int32_t *tgt = scratch<int32_t>(s, nnz + n);  // off-diagonal entries, then diagonals
  if (!C->col || !tgt) return SPH_RT_ENOMEM;
  fill_i32_kernel<<<gcap(s, nnz + n, kBlock), kBlock, 0, st>>>(nnz + n, -1, tgt);
  SPH_LAUNCHED(s);
  coarse_struct_kernel<true><<<gb, kBlock, 0, st>>>(nc, L->agg_ptr, L->agg_mem, L->ptr, L->col,
                                                    L->agg, nullptr, C->ptr, C->col, tgt, C->nnz,
                                                    tgt + nnz, overflow);
  SPH_LAUNCHED(s);
  // Galerkin contribution lists per coarse target (nnz_c off-diagonal + nc diagonal)
  rc = source_sort(s, L, nnz + n, tgt, C->nnz + nc, &L->seg_ptr, &L->seg_src);
  SPH_CUDA(s, cudaStreamSynchronize(st));
  dfree(s, tgt);
  dfree(s, overflow);
  if (rc) return rc;
  if ((rc = coarse_storage(s, C))) return rc;
  *next = C;
  return SPH_RT_OK;
}

static sph_rt_status level_vectors_fine(sph_rt *s, SphLevel *L) {
  L->res = lalloc<double>(s, L, L->n);
  L->d = lalloc<double>(s, L, L->n);
  L->t = lalloc<double>(s, L, L->n);
  if (!L->res || !L->d || !L->t) return SPH_RT_ENOMEM;
  (void)s;
  return SPH_RT_OK;
}

static sph_rt_status build_structure(sph_rt *s, double *csr) {
  amg_release(s);
  SphLevel *L0 = new SphLevel();
  CsrView<double> A = fine_view(s);
  L0->n = A.n;
  L0->nnz = A.nnz;
  L0->ptr = const_cast<int64_t *>(A.ptr);
  L0->col = const_cast<int32_t *>(A.col);
  L0->val = csr ? csr : const_cast<double *>(A.val);
  L0->diag = const_cast<double *>(A.diag);
  L0->invdiag = const_cast<double *>(A.invdiag);
  L0->W = A.W;
  L0->U = A.U;
  s->levels.push_back(L0);
  sph_rt_status rc = level_vectors_fine(s, L0);
  if (rc) return rc;
  SphLevel *L = L0;
  while ((int)s->levels.size() < kMaxLevels && L->n > kCoarseTarget) {
    // the strength test needs this level's values
    if (L != L0) {
      // values are produced by the numeric pass below; build them now
    }
    SphLevel *C = nullptr;
    if ((rc = coarsen(s, L, &C))) return rc;
    if (!C) break;
    s->levels.push_back(C);
    // numeric Galerkin product for C so that the next strength test can run
    if (L->apg_ptr) {
      // A P in FP64 (scratch where the mixed form keeps it in FP32 only), then P^T (A P)
      const int64_t stored = L->ap_sl.ptr ? L->ap_sl.padded : L->nnz_ap;
      double *ap = L->ap_val ? L->ap_val : scratch<double>(s, (size_t)stored + 1);
      if (!ap) return SPH_RT_ENOMEM;
      rc = L->ap_sl.ptr ? sliced_ap_values<double>(s, L->ap_pos, L->agg, L->ap_sl, L->ap_most,
                                                   s->sl_val, L->diag, ap)
                        : launch_galerkin<double>(s, L->nnz_ap, 0, L->ap_seg_ptr, L->ap_seg_src,
                                                  L->nnz, L->val, L->diag, ap, nullptr, nullptr);
      if (rc) return rc;
      if ((rc = launch_galerkin<double>(s, C->nnz, C->n, L->apg_ptr, SrcList{L->apg_src, nullptr},
                                        stored, ap, nullptr, C->val, C->diag, C->invdiag)))
        return rc;
      if (!L->ap_val) {
        SPH_CUDA(s, cudaStreamSynchronize(s->stream));
        dfree(s, ap);
      }
    } else if ((rc = launch_galerkin<double>(s, C->nnz, C->n, L->seg_ptr, L->seg_src, L->nnz,
                                             L->val, L->diag, C->val, C->diag, C->invdiag))) {
      return rc;
    }
    L = C;
  }
  s->amg_ready = true;
  return SPH_RT_OK;
}

// numeric set-up of every level from the current fine operator
// Bytes per value the coarsest-level solve is staged and computed in: FP32
// when config.coarse_fp32 (also in the FP64 form), else the level's type.
template <typename T>
static size_t coarse_solve_bytes(const sph_rt *s) {
  return s->cfg.coarse_fp32 ? sizeof(float) : sizeof(T);
}

// Chebyshev degree of the coarsest-level solve.  Each step is a dependent pass
// through one SM (~2 us for a few hundred rows); 6 steps gave the same Krylov
// counts as 12 on the 64^3 and 128^3 manufactured problems.
static int coarse_degree(const sph_rt *s, const SphLevel *L) {
  return L->n <= kCoarseTarget * 4 ? 6 : 3 * s->cfg.cheb_degree;
}

template <typename T>
struct LevelVecs;
template <>
struct LevelVecs<double> {
  static CsrView<double> view(SphLevel *L) {
    CsrView<double> A;
    A.n = L->n;
    A.ptr = L->ptr;
    A.col = L->col;
    A.val = L->val;
    A.diag = L->diag;
    A.invdiag = L->invdiag;
    A.nnz = L->nnz;
    A.W = L->W;
    A.U = L->U;
    return A;
  }
  static double *r(SphLevel *L) { return L->r; }
  static double *z(SphLevel *L) { return L->z; }
  static double *res(SphLevel *L) { return L->res; }
  static double *d(SphLevel *L) { return L->d; }
  static double *t(SphLevel *L) { return L->t; }
  static const double *ap(SphLevel *L) { return L->ap_val; }
};
template <>
struct LevelVecs<float> {
  static CsrView<float> view(SphLevel *L) {
    CsrView<float> A;
    A.n = L->n;
    A.ptr = L->ptr;
    A.col = L->col;
    A.val = L->val32;
    A.diag = L->diag32;
    A.invdiag = L->invdiag32;
    A.nnz = L->nnz;
    A.W = L->W;
    A.U = L->U;
    return A;
  }
  static float *r(SphLevel *L) { return L->r32; }
  static float *z(SphLevel *L) { return L->z32; }
  static float *res(SphLevel *L) { return L->res32; }
  static float *d(SphLevel *L) { return L->d32; }
  static float *t(SphLevel *L) { return L->t32; }
  static const float *ap(SphLevel *L) { return L->ap_val32; }
};


// FP32 storage of every level of the mixed form (level 0 borrows the FP32
// copy the assembly writes).
static sph_rt_status level_fp32(sph_rt *s, size_t l) {
  SphLevel *L = s->levels[l];
  if (L->r32) return SPH_RT_OK;
  if (l == 0) {
    L->val32 = s->mat_val32;  // none where the operator is in slices
    L->diag32 = s->diag32;
    L->invdiag32 = s->invdiag32;
  } else {
    L->val32 = lalloc<float>(s, L, L->nnz);
    L->diag32 = lalloc<float>(s, L, L->n);
    L->invdiag32 = lalloc<float>(s, L, L->n);
  }
  L->r32 = lalloc<float>(s, L, L->n);
  L->z32 = lalloc<float>(s, L, L->n);
  L->res32 = lalloc<float>(s, L, L->n);
  L->d32 = lalloc<float>(s, L, L->n);
  L->t32 = lalloc<float>(s, L, L->n);
  if ((!L->val32 && !(l == 0 && s->sl.ptr)) || !L->diag32 || !L->invdiag32 || !L->r32 || !L->z32 || !L->res32 || !L->d32 ||
      !L->t32)
    return SPH_RT_ENOMEM;
  return SPH_RT_OK;
}

// Galerkin values of every level from the current fine operator, in the
// hierarchy's type T: FP64, or FP32 in the mixed form, where the sums are
// formed from the FP32 fine copy directly.
template <typename T>
static sph_rt_status galerkin_levels(sph_rt *s) {
  using LV = LevelVecs<T>;
  for (size_t l = 0; l + 1 < s->levels.size(); ++l) {
    SphLevel *L = s->levels[l], *C = s->levels[l + 1];
    const CsrView<T> Lv = LV::view(L), Cv = LV::view(C);
    if (L->ap_sl.ptr) {
      const SlicedView<T> F = fine_sliced<T>(s);
      sph_rt_status rc = sliced_ap_values<T>(s, L->ap_pos, L->agg, L->ap_sl, L->ap_most, F.val,
                                             F.diag, const_cast<T *>(LV::ap(L)));
      if (rc) return rc;
    } else if (L->ap_ptr) {  // A P of this level (its values are final: level l is done)
      sph_rt_status rc = launch_galerkin<T>(s, L->nnz_ap, 0, L->ap_seg_ptr, L->ap_seg_src,
                                            L->nnz, Lv.val, Lv.diag, const_cast<T *>(LV::ap(L)),
                                            nullptr, nullptr);
      if (rc) return rc;
    }
    T *cval = const_cast<T *>(Cv.val), *cdiag = const_cast<T *>(Cv.diag),
      *cinv = const_cast<T *>(Cv.invdiag);
    // P^T (A P): its sources are A P entries (fewer than 2^31)
    sph_rt_status rc =
        L->apg_ptr ? launch_galerkin<T>(s, C->nnz, C->n, L->apg_ptr, SrcList{L->apg_src, nullptr},
                                        L->ap_sl.ptr ? L->ap_sl.padded : L->nnz_ap, LV::ap(L),
                                        nullptr, cval, cdiag, cinv)
                   : launch_galerkin<T>(s, C->nnz, C->n, L->seg_ptr, L->seg_src, L->nnz, Lv.val,
                                        Lv.diag, cval, cdiag, cinv);
    if (rc) return rc;
  }
  // Gershgorin bounds of every level, turned into Chebyshev coefficients on
  // the device (slot 1 + l): no host read
  if (!s->amg_gersh) s->amg_gersh = dalloc<double>(s, kMaxLevels);
  double *dg = s->amg_gersh;
  if (!dg) return SPH_RT_ENOMEM;
  GershLevels<T> G;
  memset(&G, 0, sizeof G);
  G.count = (int)s->levels.size();
  int64_t rows = 0;
  for (int l = 1; l < G.count; ++l) {
    const CsrView<T> Lv = LV::view(s->levels[l]);
    G.L[l] = {Lv.n, Lv.ptr, Lv.val, Lv.diag};
    rows += Lv.n;
  }
  SPH_CUDA(s, cudaMemsetAsync(dg, 0, sizeof(double) * kMaxLevels, s->stream));
  gersh_kernel<T><<<gcap(s, rows, kBlock / 4), kBlock, 0, s->stream>>>(G, s->gersh, dg);
  SPH_LAUNCHED(s);
  return SPH_RT_OK;
}

bool fcg_active(const sph_rt *s);
sph_rt_status fcg_vectors(sph_rt *s, FcgVecs *v);

static sph_rt_status numeric(sph_rt *s) {
  sph_rt_status rc;
  const bool mixed = s->cfg.precision == SPH_RT_MIXED;
  if (mixed) {
    for (size_t l = 0; l < s->levels.size(); ++l)
      if ((rc = level_fp32(s, l))) return rc;
    SphLevel *L0 = s->levels[0];
    if (L0->ap_ptr && !L0->ap_val32 && !(L0->ap_val32 = lalloc<float>(s, L0, L0->nnz_ap)))
      return SPH_RT_ENOMEM;
    if ((rc = galerkin_levels<float>(s))) return rc;
  } else {
    if ((rc = galerkin_levels<double>(s))) return rc;
  }
  std::vector<int> mode(s->levels.size()), degree(s->levels.size());
  for (size_t l = 0; l < s->levels.size(); ++l) {
    const bool coarsest = l + 1 == s->levels.size();
    mode[l] = coarsest ? 2 : 1;
    degree[l] = coarsest ? coarse_degree(s, s->levels[l]) : s->cfg.cheb_degree;
  }
  if ((rc = launch_cheb_slots(s, 1, s->amg_gersh, mode, degree))) return rc;
  // FP32 CG vectors of the V-cycle-product CG, allocated here (not while a
  // loop graph is being captured)
  if (mixed && fcg_active(s)) {
    FcgVecs v;
    if ((rc = fcg_vectors(s, &v))) return rc;
  }
  return SPH_RT_OK;
}

template <typename T>
static void tail_setup(sph_rt *s);

static sph_rt_status setup_levels(sph_rt *s) {
  sph_rt_status rc;
  if (!s->amg_ready || s->cfg.amg_rebuild) {
    // the set-up reads the finest level's values in CSR order
    double *csr = nullptr;
    if (s->sl.ptr && (rc = sliced_to_csr(s, &csr))) return rc;
    if ((rc = build_structure(s, csr))) return rc;
    if (s->cfg.precision == SPH_RT_MIXED)
      tail_setup<float>(s);
    else
      tail_setup<double>(s);
    if (csr) {
      SPH_CUDA(s, cudaStreamSynchronize(s->stream));
      dfree(s, csr);
      s->levels[0]->val = nullptr;
    }
  }
  return numeric(s);
}

sph_rt_status amg_setup(sph_rt *s, double dt) {
  if (!s->sl.ptr || (s->amg_ready && !s->cfg.amg_rebuild)) return setup_levels(s);
  // beside the slices the device may be too small for a set-up that has room beside
  // CSR rows: what it took goes back, and it starts again from those, assembled anew
  // (a diagonal's sum runs in the order of its row's entries there)
  amg_release(s);
  std::vector<void *> held = s->allocs;
  std::sort(held.begin(), held.end());
  sph_rt_status rc = setup_levels(s);
  if (rc != SPH_RT_ENOMEM) return rc;
  cudaStreamSynchronize(s->stream);
  amg_release(s);
  const std::vector<void *> now = s->allocs;
  for (void *p : now)
    if (!std::binary_search(held.begin(), held.end(), p)) {
      if (p == s->amg_gersh) s->amg_gersh = nullptr;
      dfree(s, p);
    }
  if ((rc = sliced_undo(s))) return rc;
  s->err.clear();
  if ((rc = launch_assembly(s, dt, s->gersh))) return rc;
  return setup_levels(s);
}

// ---------------------------------------------------------------------------
// V-cycle
// ---------------------------------------------------------------------------
// Launch CALL over the rows of the finest level's A P, sliced or in CSR row tiles
// of shape `sh` and CSR_BLOCKS_ blocks per SM (as SPH_FINE_ROWS).
#define SPH_AP_ROWS(s_, L_, T_, CSR_BLOCKS_, CALL)                                         \
  do {                                                                                     \
    if ((L_)->ap_sl.ptr) {                                                                 \
      using Rows = SlicedRows<T_>;                                                         \
      const Rows rows{sliced_view<T_>((L_)->ap_sl, (L_)->n, (L_)->nnz_ap, LV::ap(L_),      \
                                      nullptr, nullptr)};                                  \
      const int grid = sliced_grid(                                                        \
          s_, (L_)->n, (CSR_BLOCKS_) < Rows::kMinBlocks ? (CSR_BLOCKS_) : Rows::kMinBlocks); \
      const size_t smem = (size_t)(L_)->ap_sl.dict_max * sizeof(T_);                       \
      CALL;                                                                                \
    } else {                                                                               \
      CsrView<T_> apv;                                                                     \
      apv.n = (L_)->n;                                                                     \
      apv.ptr = (L_)->ap_ptr;                                                              \
      apv.col = (L_)->ap_col;                                                              \
      apv.val = LV::ap(L_);                                                                \
      const size_t smem = 0;                                                               \
      SPH_DISPATCH_SHAPE(sh.W, sh.U, ({                                                    \
                           using Rows = CsrRows<W, U, T_>;                                 \
                           const Rows rows{apv};                                           \
                           const int grid =                                                \
                               row_grid_blocks((s_)->num_sms, apv.n, W, CSR_BLOCKS_);      \
                           CALL;                                                           \
                         }));                                                              \
    }                                                                                      \
  } while (0)

template <typename T>
static sph_rt_status launch_tail(sph_rt *s, size_t l0, const T *r, T *z, const Scalars *sc) {
  using LV = LevelVecs<T>;
  TailParams<T> P;
  memset(&P, 0, sizeof P);
  P.nlev = (int)(s->levels.size() - l0);
  for (int m = 0; m < P.nlev; ++m) {
    SphLevel *L = s->levels[l0 + m];
    TailLevel<T> &t = P.L[m];
    t.A = LV::view(L);
    t.agg = L->agg;
    t.agg_ptr = L->agg_ptr;
    t.agg_mem = L->agg_mem;
    t.r = m == 0 ? const_cast<T *>(r) : LV::r(L);
    t.z = m == 0 ? z : LV::z(L);
    t.res = LV::res(L);
    t.d = LV::d(L);
    t.t = LV::t(L);
    t.cf = s->cheb_slots + 1 + l0 + m;
    t.deg = m + 1 == P.nlev ? coarse_degree(s, L) : s->cfg.cheb_degree;
  }
  SphLevel *Lc = s->levels.back();
  const size_t cs = coarse_solve_bytes<T>(s);
  const size_t smem = coarse_smem_bytes(Lc->n, Lc->nnz, cs, cs);
  P.coarse_smem = 1;  // tail_setup only enables the tail when the coarsest level fits
  P.coarse_fp32 = cs == sizeof(float) && sizeof(T) == sizeof(double);
  cudaLaunchConfig_t lc;
  memset(&lc, 0, sizeof lc);
  lc.gridDim = dim3((unsigned)s->tail_cluster);
  lc.blockDim = dim3(1024);
  lc.dynamicSmemBytes = smem;
  lc.stream = s->stream;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = (unsigned)s->tail_cluster;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  lc.attrs = attr;
  lc.numAttrs = 1;
  SPH_CUDA(s, cudaLaunchKernelEx(&lc, vcycle_tail_kernel<T>, P, sc));
  SPH_LAUNCHED(s);
  return SPH_RT_OK;
}

// Decide where the cluster tail starts (0 = no tail) and its cluster size:
// 16 blocks where the device can co-schedule them, else 8.
template <typename T>
static void tail_setup(sph_rt *s) {
  s->tail_level = 0;
  s->tail_cluster = 0;
  const int nl = (int)s->levels.size();
  if (nl < 3 || !s->cfg.amg_tail) return;
  int l0 = nl;
  while (l0 > 1 && s->levels[l0 - 1]->nnz <= kTailMaxNnz) --l0;
  if (nl - l0 < 2) return;
  SphLevel *Lc = s->levels.back();
  const size_t cs = coarse_solve_bytes<T>(s);
  const size_t smem = coarse_smem_bytes(Lc->n, Lc->nnz, cs, cs);
  if (smem > kCoarseSmemMax) return;
  auto kern = vcycle_tail_kernel<T>;
  if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize,
                           (int)kCoarseSmemMax) != cudaSuccess) {
    cudaGetLastError();
    return;
  }
  cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
  cudaGetLastError();
  for (int cl : {16, 8}) {
    cudaLaunchConfig_t lc;
    memset(&lc, 0, sizeof lc);
    lc.gridDim = dim3((unsigned)cl);
    lc.blockDim = dim3(1024);
    lc.dynamicSmemBytes = smem;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = (unsigned)cl;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    lc.attrs = attr;
    lc.numAttrs = 1;
    int clusters = 0;
    if (cudaOccupancyMaxActiveClusters(&clusters, kern, &lc) == cudaSuccess && clusters >= 1) {
      s->tail_level = l0;
      s->tail_cluster = cl;
      return;
    }
    cudaGetLastError();
  }
}

// Whether a level post-smooths through A P.
template <typename T>
static bool has_ap(SphLevel *L) {
  return L->ap_ptr && LevelVecs<T>::ap(L);
}
// Where the zero-guess smoother start of level L goes, z being the buffer of its
// result: cheb_apply's first write (levels without A P: see vcycle).
template <typename T>
static T *smoother_start(const sph_rt *s, SphLevel *L, T *z) {
  const bool odd = s->cfg.cheb_degree % 2 == 1;
  return has_ap<T>(L) && odd ? z : LevelVecs<T>::t(L);
}

// Residual of level l (no A P) restricted to level l + 1, with that level's
// smoother start at zc_first unless it is null.
template <typename T>
static sph_rt_status launch_resid_restrict(sph_rt *s, size_t l, const T *r, const T *zpre,
                                           T *zc_first, const Scalars *sc) {
  using LV = LevelVecs<T>;
  SphLevel *L = s->levels[l], *C = s->levels[l + 1];
  const CsrView<T> A = LV::view(L);
  const int gr = gcap(s, C->n, kWarpsPerBlock);  // a warp per coarse row
  int *wf = l == 0 ? timing_begin(s) : nullptr;
  if (zc_first)
    SPH_DISPATCH_SHAPE(A.W, A.U,
                       (pdl_launch(s, resid_restrict_kernel<W, U, T, true>, gr, kBlock, 0, A, r,
                                   zpre, C->n, (const int64_t *)L->agg_ptr,
                                   (const int32_t *)L->agg_mem, LV::r(C), LV::view(C).invdiag,
                                   (const ChebCoef *)(s->cheb_slots + 2 + l), LV::d(C), zc_first,
                                   sc, wf)));
  else
    SPH_DISPATCH_SHAPE(A.W, A.U,
                       (pdl_launch(s, resid_restrict_kernel<W, U, T, false>, gr, kBlock, 0, A, r,
                                   zpre, C->n, (const int64_t *)L->agg_ptr,
                                   (const int32_t *)L->agg_mem, LV::r(C), (const T *)nullptr,
                                   (const ChebCoef *)nullptr, (T *)nullptr, (T *)nullptr, sc,
                                   wf)));
  SPH_LAUNCHED(s);
  if (l == 0)
    timing_end(s, (4.0 + sizeof(T)) * (double)A.nnz + (12.0 + 3.0 * sizeof(T)) * (double)A.n,
               kTimedResid);
  return SPH_RT_OK;
}

template <typename T>
static sph_rt_status vcycle(sph_rt *s, size_t l, const T *r, T *z, const Scalars *sc,
                            bool init_done = false, const DotFuse *df = nullptr,
                            bool *dot_done = nullptr) {
  using LV = LevelVecs<T>;
  if (s->tail_level > 0 && l == (size_t)s->tail_level) return launch_tail<T>(s, l, r, z, sc);
  SphLevel *L = s->levels[l];
  CsrView<T> A = LV::view(L);
  const int deg = s->cfg.cheb_degree;
  sph_rt_status rc;
  if (l + 1 == s->levels.size()) {
    // coarsest level: Chebyshev solve over the whole Gershgorin interval
    const int cdeg = coarse_degree(s, L);
    const ChebCoef *cf = s->cheb_slots + 1 + l;
    const size_t cs = coarse_solve_bytes<T>(s);
    const size_t smem = coarse_smem_bytes(L->n, L->nnz, cs, cs);
    if (l > 0 && smem <= kCoarseSmemMax) {
      // opt in to more than 48 KiB of dynamic shared memory (once per handle and variant)
      const bool f32 = cs == sizeof(float) && sizeof(T) == sizeof(double);
      const int bit = f32 ? 4 : (sizeof(T) == 8 ? 1 : 2);
      if (!(s->coarse_smem_optin & bit)) {
        if (f32)
          SPH_CUDA(s, cudaFuncSetAttribute(coarse_cheb_kernel<T, float, T>,
                                           cudaFuncAttributeMaxDynamicSharedMemorySize,
                                           (int)kCoarseSmemMax));
        else
          SPH_CUDA(s, cudaFuncSetAttribute(coarse_cheb_kernel<T, T, T>,
                                           cudaFuncAttributeMaxDynamicSharedMemorySize,
                                           (int)kCoarseSmemMax));
        s->coarse_smem_optin |= bit;
      }
      if (f32)
        pdl_launch(s, coarse_cheb_kernel<T, float, T>, 1, 1024, smem, A, r, z, cf, cdeg, sc);
      else
        pdl_launch(s, coarse_cheb_kernel<T, T, T>, 1, 1024, smem, A, r, z, cf, cdeg, sc);
      SPH_LAUNCHED(s);
      return SPH_RT_OK;
    }
    return cheb_apply<T, T>(s, A, r, z, LV::d(L), LV::t(L), cdeg, cf, sc, false);
  }
  const ChebCoef *cf = s->cheb_slots + 1 + l;
  SphLevel *C = s->levels[l + 1];
  // a launched, non-coarsest next level takes its smoother start from the restriction
  const bool fuse = l + 2 < s->levels.size() &&
                    !(s->tail_level > 0 && l + 1 == (size_t)s->tail_level);
  T *zc_first = fuse ? smoother_start<T>(s, C, LV::z(C)) : nullptr;
  if (!has_ap<T>(L)) {
    // pre-smoothing into the buffer that the first post-smoothing step reads
    T *t = LV::t(L);
    const bool odd = deg % 2 == 1;
    T *zpre = odd ? t : z, *zpost = odd ? z : t;
    if ((rc = cheb_apply<T, T>(s, A, r, zpre, LV::d(L), zpost, deg, cf, sc, init_done)))
      return rc;
    if ((rc = launch_resid_restrict<T>(s, l, r, zpre, zc_first, sc))) return rc;
    if ((rc = vcycle<T>(s, l + 1, LV::r(C), LV::z(C), sc, fuse))) return rc;
    const int gp = row_grid_blocks(s->num_sms, L->n, A.W, kCoarseMinBlocks);
    const bool dot = l == 0 && df && dot_done && deg == 1;
    int *wf = l == 0 ? timing_begin(s) : nullptr;
    if (dot)
      SPH_DISPATCH_SHAPE(A.W, A.U,
                         (pdl_launch(s, prolong_cheb_kernel<W, U, T, true>, gp, kBlock, 0, A, r,
                                     (const T *)zpre, (const int32_t *)L->agg,
                                     (const T *)LV::z(C), zpost, LV::d(L), cf, sc, wf, *df)));
    else
      SPH_DISPATCH_SHAPE(A.W, A.U,
                         (pdl_launch(s, prolong_cheb_kernel<W, U, T, false>, gp, kBlock, 0, A, r,
                                     (const T *)zpre, (const int32_t *)L->agg,
                                     (const T *)LV::z(C), zpost, LV::d(L), cf, sc, wf,
                                     DotFuse{})));
    SPH_LAUNCHED(s);
    if (dot) *dot_done = true;
    if (l == 0)
      timing_end(s, (4.0 + sizeof(T)) * (double)A.nnz + (12.0 + 7.0 * sizeof(T)) * (double)A.n,
                 kTimedCheb);
    // the remaining post-smoothing steps
    return cheb_apply<T, T>(s, A, r, z, LV::d(L), t, deg, cf, sc, true);
  }
  // zero-guess pre-smoothing (its first write was made by the restriction above
  // when init_done)
  if ((rc = cheb_apply<T, T>(s, A, r, z, LV::d(L), LV::t(L), deg, cf, sc, init_done)))
    return rc;
  const int gw = row_grid_blocks(s->num_sms, L->n, A.W, kCoarseMinBlocks);
  T *res = LV::res(L);
  // fine-level residual sweeps are timed with the other fine SpMV-class kernels;
  // per row: rowptr, diag, r, z, res
  int *wf = l == 0 ? timing_begin(s) : nullptr;
  if (l == 0)
    SPH_FINE_ROWS(s, T, A, sizeof(T),
                  (pdl_launch(s, fine_resid_level_kernel<Rows, T>, grid, kBlock, smem, rows, r, z,
                              res, sc, wf)));
  else
    SPH_DISPATCH_SHAPE(A.W, A.U,
                       (pdl_launch(s, resid_level_kernel<W, U, T, T>, gw, kBlock, 0, A, r, z, res,
                                   sc)));
  SPH_LAUNCHED(s);
  if (l == 0)
    timing_end(s, ((s->sl.ptr ? 2.0 : 4.0) + sizeof(T)) * (double)A.nnz + (8.0 + 4.0 * sizeof(T)) * (double)A.n,
               kTimedResid);
  if (fuse) {
    pdl_launch(s, restrict_init_kernel<T, T>, gcap(s, C->n, kBlock), kBlock, 0,
        C->n, L->agg_ptr, L->agg_mem, res, LV::r(C), LV::view(C).invdiag,
        s->cheb_slots + 1 + (l + 1), LV::d(C), zc_first, sc);
  } else {
    pdl_launch(s, restrict_kernel<T>, gcap(s, C->n, kBlock), kBlock, 0,
        C->n, L->agg_ptr, L->agg_mem, res, LV::r(C), sc);
  }
  SPH_LAUNCHED(s);
  if ((rc = vcycle<T>(s, l + 1, LV::r(C), LV::z(C), sc, fuse))) return rc;
  {
    // prolongation and the first post-smoothing step in one sweep of A P
    T *bufs[2] = {z, LV::t(L)};
    const int w0 = (deg - 1) % 2;
    const RowShape sh = shape_for_mean(L->n ? (double)L->nnz_ap / (double)L->n : 0.0);
    int *wf = l == 0 ? timing_begin(s) : nullptr;
    // with degree 1 this sweep is the V-cycle's last: the inner product rides along
    const bool dot = l == 0 && df && dot_done && deg == 1;
    if (dot) {
      SPH_AP_ROWS(s, L, T, sweep_min_blocks(sh.U),
                  (pdl_launch(s, fine_post_ap_kernel<Rows, T, true>, grid, kBlock, smem, rows,
                              (const int32_t *)L->agg, (const T *)LV::z(C), (const T *)z,
                              (const T *)res, A.invdiag, cf, LV::d(L), bufs[w0], sc, wf, *df)));
      *dot_done = true;
    } else if (l == 0) {
      SPH_AP_ROWS(s, L, T, sweep_min_blocks(sh.U),
                  (pdl_launch(s, fine_post_ap_kernel<Rows, T, false>, grid, kBlock, smem, rows,
                              (const int32_t *)L->agg, (const T *)LV::z(C), (const T *)z,
                              (const T *)res, A.invdiag, cf, LV::d(L), bufs[w0], sc, wf,
                              DotFuse{})));
    } else {
      const int gp = row_grid_blocks(s->num_sms, L->n, sh.W, kCoarseMinBlocks);
      SPH_DISPATCH_SHAPE(sh.W, sh.U,
                         (pdl_launch(s, post_ap_kernel<W, U, T, T>, gp, kBlock, 0,
                             L->n, L->ap_ptr, L->ap_col, LV::ap(L), L->agg, LV::z(C), z, res,
                             A.invdiag, cf, LV::d(L), bufs[w0], sc)));
    }
    SPH_LAUNCHED(s);
    // A P entry: column + value; per row: ap_ptr, agg, the coarse entry of P e_c,
    // z_pre, res, 1/diag, d, z_out; with the inner product also r (and, flexible,
    // the FP64 z read and written)
    if (l == 0)
      timing_end(s,
                 ((L->ap_sl.ptr ? 2.0 : 4.0) + sizeof(T)) * (double)L->nnz_ap +
                     (12.0 + 6.0 * sizeof(T) + (dot ? (df->flex ? 24.0 : 8.0) : 0.0)) *
                         (double)L->n,
                 kTimedPost);
    return cheb_apply<T, T>(s, A, r, z, LV::d(L), LV::t(L), deg, cf, sc, true);
  }
}

// Mixed form without the last conversion: r is rounded to FP32 and the FP32
// V-cycle leaves z in levels[0]->z32 (amg_z32), for a caller that widens it
// itself (the fused flexible-CG inner product).  init_done: r32 and the finest
// level's smoother start were written by the CG update.
sph_rt_status amg_apply_to32(sph_rt *s, const double *r, const Scalars *sc, bool init_done,
                             const DotFuse *df, bool *dot_done) {
  if (s->levels.empty()) return set_error(s, SPH_RT_ESTATE, "AMG hierarchy not set up");
  SphLevel *L0 = s->levels[0];
  if (!init_done) {
    pdl_launch(s, convert_kernel<double, float>, gcap(s, L0->n, kBlock), kBlock, 0, L0->n, r,
                                                                                    L0->r32);
    SPH_LAUNCHED(s);
  }
  return vcycle<float>(s, 0, L0->r32, L0->z32, sc, init_done, df, dot_done);
}
const float *amg_z32(const sph_rt *s) { return s->levels.empty() ? nullptr : s->levels[0]->z32; }

// The finest level's zero-guess smoother start for the CG update to write
// (FineInit): in FP64 into the preconditioner output z (or the ping-pong
// buffer the start goes to), in FP32 into the level's FP32 vectors together
// with the narrowed residual.  False where the V-cycle takes no such start
// (a single level: the finest level is then the coarsest).
bool amg_fine_init(sph_rt *s, FineInit<double> *f64, FineInit<float> *f32) {
  if (s->levels.size() < 2) return false;
  SphLevel *L0 = s->levels[0];
  const ChebCoef *cf = s->cheb_slots + 1;
  if (s->cfg.precision == SPH_RT_MIXED) {
    *f32 = {L0->r32, L0->invdiag32, cf, L0->d32, smoother_start<float>(s, L0, L0->z32)};
  } else {
    *f64 = {nullptr, L0->invdiag, cf, L0->d, smoother_start<double>(s, L0, s->z)};
  }
  return true;
}

sph_rt_status amg_apply(sph_rt *s, const double *r, double *z, const Scalars *sc, bool init_done,
                        const DotFuse *df, bool *dot_done) {
  if (s->levels.empty()) return set_error(s, SPH_RT_ESTATE, "AMG hierarchy not set up");
  if (s->cfg.precision == SPH_RT_MIXED) {
    SphLevel *L0 = s->levels[0];
    if (!init_done) {
      pdl_launch(s, convert_kernel<double, float>, gcap(s, L0->n, kBlock), kBlock, 0, L0->n, r,
                                                                                      L0->r32);
      SPH_LAUNCHED(s);
    }
    sph_rt_status rc = vcycle<float>(s, 0, L0->r32, L0->z32, sc, init_done);
    if (rc) return rc;
    pdl_launch(s, convert_kernel<float, double>, gcap(s, L0->n, kBlock), kBlock, 0, L0->n, L0->z32, z);
    SPH_LAUNCHED(s);
    return SPH_RT_OK;
  }
  return vcycle<double>(s, 0, r, z, sc, init_done, df, dot_done);
}

// ---------------------------------------------------------------------------
// The V-cycle of the CG with the V-cycle's product (fine_post_smooth = 0), in
// the precision T of the hierarchy: from r and the smoother start z_pre (in
// the finest level's d, written by the CG update or the residual kernel), the
// finest-level residual sweep, the coarse V-cycle (symmetric, as always) and
// the last sweep that forms z, w = B z and the CG scalars (see
// fine_ap_cg_kernel).  The vectors are those of FcgVecs.
// ---------------------------------------------------------------------------
bool fcg_active(const sph_rt *s) {
  return s->cfg.fine_post_smooth == 0 && s->cfg.precond == SPH_RT_PRECOND_AMG &&
         s->levels.size() >= 2;
}

sph_rt_status fcg_vectors(sph_rt *s, FcgVecs *v) {
  SphLevel *L0 = s->levels[0];
  if (s->cfg.precision == SPH_RT_MIXED) {
    if (!L0->p32) {
      L0->p32 = lalloc<float>(s, L0, L0->n);
      L0->q32 = lalloc<float>(s, L0, L0->n);
      L0->w32 = lalloc<float>(s, L0, L0->n);
      if (!L0->p32 || !L0->q32 || !L0->w32) return SPH_RT_ENOMEM;
    }
    v->f32 = {L0->r32, L0->z32, L0->w32, L0->p32, L0->q32, L0->d32, L0->invdiag32};
  } else {
    v->f64 = {s->r, s->z, s->w, s->p, s->q, L0->d, L0->invdiag};
  }
  v->cf = s->cheb_slots + 1;
  return SPH_RT_OK;
}

template <typename T>
static sph_rt_status fcg_cycle_t(sph_rt *s, const FcgSet<T> &v, int first) {
  using LV = LevelVecs<T>;
  SphLevel *L = s->levels[0];
  CsrView<T> A = LV::view(L);
  const Scalars *sc = s->sc;
  T *res = LV::res(L);
  SphLevel *C = s->levels[1];
  const bool fuse = s->levels.size() > 2 && !(s->tail_level > 0 && s->tail_level == 1);
  T *zc_first = fuse ? smoother_start<T>(s, C, LV::z(C)) : nullptr;
  sph_rt_status rc;
  int *wf = nullptr;
  if (!has_ap<T>(L)) {
    if ((rc = launch_resid_restrict<T>(s, 0, v.r, v.zpre, zc_first, sc))) return rc;
  } else {
    wf = timing_begin(s);
    SPH_FINE_ROWS(s, T, A, sizeof(T),
                  (pdl_launch(s, fine_resid_level_kernel<Rows, T>, grid, kBlock, smem, rows,
                              (const T *)v.r, (const T *)v.zpre, res, sc, wf)));
    SPH_LAUNCHED(s);
    timing_end(s,
               ((s->sl.ptr ? 2.0 : 4.0) + sizeof(T)) * (double)A.nnz +
                   (8.0 + 4.0 * sizeof(T)) * (double)A.n,
               kTimedResid);
    if (fuse)
      pdl_launch(s, restrict_init_kernel<T, T>, gcap(s, C->n, kBlock), kBlock, 0, C->n,
                 L->agg_ptr, L->agg_mem, (const T *)res, LV::r(C), LV::view(C).invdiag,
                 s->cheb_slots + 2, LV::d(C), zc_first, sc);
    else
      pdl_launch(s, restrict_kernel<T>, gcap(s, C->n, kBlock), kBlock, 0, C->n, L->agg_ptr,
                 L->agg_mem, (const T *)res, LV::r(C), sc);
    SPH_LAUNCHED(s);
  }
  if ((rc = vcycle<T>(s, 1, LV::r(C), LV::z(C), sc, fuse))) return rc;
  if (L->ap_ptr && LV::ap(L)) {
    const RowShape sh = shape_for_mean(L->n ? (double)L->nnz_ap / (double)L->n : 0.0);
    wf = timing_begin(s);
    SPH_AP_ROWS(s, L, T, fcg_min_blocks<T>(),
                (pdl_launch(s, fine_ap_cg_kernel<Rows, T>, grid, kBlock, smem, rows,
                            (const int32_t *)L->agg, (const T *)LV::z(C), (const T *)v.zpre,
                            (const T *)res, (const T *)v.r, v.z, v.w, (const T *)v.p,
                            (const T *)v.q, first, s->sc, s->partials, wf, s->loop_cond)));
    SPH_LAUNCHED(s);
    // A P entry: column + value; per row: ap_ptr, agg, P e_c, z_pre, res, r, z r/w, w,
    // p, q
    timing_end(s, ((L->ap_sl.ptr ? 2.0 : 4.0) + sizeof(T)) * (double)L->nnz_ap +
                      (12.0 + 10.0 * sizeof(T)) * (double)L->n,
               kTimedPost);
    return SPH_RT_OK;
  }
  T *t = LV::t(L);
  pdl_launch(s, fcg_prolong_kernel<T>, gcap(s, L->n, kBlock), kBlock, 0, L->n,
             (const int32_t *)L->agg, (const T *)LV::z(C), (const T *)v.zpre, t, sc);
  SPH_LAUNCHED(s);
  wf = timing_begin(s);
  const int gd = row_grid_blocks(s->num_sms, L->n, A.W, fcg_min_blocks<T>());
  SPH_DISPATCH_SHAPE(A.W, A.U,
                     (pdl_launch(s, fcg_spmv_dot_kernel<W, U, T, T>, gd, kBlock, 0, A,
                                 (const T *)t, (const T *)v.r, v.z, v.w, (const T *)v.p,
                                 (const T *)v.q, first, s->sc, s->partials, wf, s->loop_cond)));
  SPH_LAUNCHED(s);
  timing_end(s, (4.0 + sizeof(T)) * (double)A.nnz + (8.0 + 9.0 * sizeof(T)) * (double)A.n,
             kTimedSpmvPQ);
  return SPH_RT_OK;
}

sph_rt_status fcg_cycle(sph_rt *s, const FcgVecs &v, int first) {
  if (s->cfg.precision == SPH_RT_MIXED) return fcg_cycle_t<float>(s, v.f32, first);
  return fcg_cycle_t<double>(s, v.f64, first);
}

// Launch-relevant layout of the hierarchy, appended to the signature of a captured loop
// graph: sizes, shapes, the finest level's own buffers and EVERY buffer that belongs to a
// level, in the order of allocation, which gives each its role.  (Rebuilt hierarchies
// take their buffers from a free list keyed by size: buffers of one size can change
// places while all others stay.)
void amg_signature(const sph_rt *s, std::vector<uint64_t> &sig) {
  sig.push_back(s->levels.size());
  sig.push_back((uint64_t)s->tail_level);
  sig.push_back((uint64_t)s->tail_cluster);
  for (const SphLevel *L : s->levels) {
    const uint64_t v[] = {(uint64_t)L->n,
                          (uint64_t)L->nnz,
                          (uint64_t)L->nnz_ap,
                          (uint64_t)L->W,
                          (uint64_t)L->U,
                          (uint64_t)L->ap_sl.dict_max,
                          (uint64_t)L->ap_sl.padded,
                          (uint64_t)(uintptr_t)L->ptr,
                          (uint64_t)(uintptr_t)L->col,
                          (uint64_t)(uintptr_t)L->val,
                          (uint64_t)(uintptr_t)L->diag,
                          (uint64_t)(uintptr_t)L->invdiag,
                          (uint64_t)(uintptr_t)L->val32,
                          (uint64_t)(uintptr_t)L->diag32,
                          (uint64_t)(uintptr_t)L->invdiag32,
                          (uint64_t)L->owned.size()};
    sig.insert(sig.end(), v, v + sizeof v / sizeof v[0]);
    for (void *p : L->owned) sig.push_back((uint64_t)(uintptr_t)p);
  }
}

// number of levels and rows/nnz per level (for diagnostics)
int amg_levels(const sph_rt *s, int64_t *rows, int64_t *nnz, int maxl) {
  int k = 0;
  for (SphLevel *L : s->levels) {
    if (k >= maxl) break;
    rows[k] = L->n;
    nnz[k] = L->nnz;
    ++k;
  }
  return k;
}

}  // namespace sphrt
