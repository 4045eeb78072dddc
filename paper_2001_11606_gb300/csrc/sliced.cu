// sliced.cu -- sliced operators of the finest level (layout and reasons at
// SlicedView in common.cuh): building the slices and dictionaries from CSR rows,
// moving arrays between the two orders, and the values of A P.
#include <cuda_runtime.h>

#include <vector>

#include "common.cuh"
#include "sliced.cuh"

namespace sphrt {

sph_rt_status exclusive_scan(sph_rt *s, const int64_t *in, int64_t n, int64_t *out);

// A group's columns are collected as 32-column words: a hash table of kWordTable
// keys, at most kWordCap of them used.
constexpr int kWordTable = 2048;
constexpr int kWordCap = 1024;
// largest dictionary: a block stages it in FP64 beside its own shared memory (up to
// 7.2 KB: the assembly), and the two stay within the 48 KB of any launch
constexpr int kDictCap = 5120;

static int blocks_for(const sph_rt *s, int64_t n, int per_block, int per_sm) {
  const int64_t g = ceil_div(n > 0 ? n : 1, per_block), cap = (int64_t)s->num_sms * per_sm;
  return (int)(g < cap ? g : cap);
}

// Rows worth slicing: a block takes 256 rows, so the layout needs kSliceMinGroups
// groups per SM to spread them evenly, and A P is formed from it (amg.cu), so the
// level must be one that has A P.  FP64 steps in ms, row tiles and slices, at 1.2, 2.0,
// 3.0, 5.0 and 16 groups per SM: 240 entries a row (3-D) 1.05 1.27, 2.14 2.17, 3.08 3.19,
// 4.49 4.47, 11.2 9.7; 104 entries 1.18 1.20, 1.57 1.58, 1.84 1.77 and, at 26 groups,
// 10.0 8.7; 25 entries (2-D) 1.32 1.24, 1.72 1.66, 2.00 1.97.  The long rows set the line:
// below two groups they lose up to a fifth, between two and four up to 7 % (616 groups on
// 608 resident blocks), from five on nothing.  Mixed steps gain 4-30 % from two groups on.
// The first step of a set pays 0.1-2 ms for building them.
// A set holds ~36 bytes per entry in CSR rows; building the slices takes ~19 more and
// the AMG set-up its lists: a set that has less than kSliceBytes of the device per
// entry stays in CSR rows.  Sizes alone decide, never the memory that happens to be
// free: the two layouts add a row in different orders, and the same set is to give the
// same bits in every run.
static bool sliced_wanted(const sph_rt *s) {
  constexpr double kSliceBytes = 125.0;
  if (s->n_int < (int64_t)kSliceMinGroups * s->num_sms * kBlock || s->nnz_mat <= kTailMaxNnz)
    return false;
  if (s->nnz_mat <= (int64_t)500000000) return true;  // 63 GB, of the 284 of a GB300
  size_t free_b = 0, total_b = 0;
  return cudaMemGetInfo(&free_b, &total_b) == cudaSuccess &&
         kSliceBytes * (double)s->nnz_mat <= (double)total_b;
}

// ---------------------------------------------------------------------------
// structure
// ---------------------------------------------------------------------------
// One block per group: the rows by eighths of their length, longest first (ties by
// row), and the widths of the group's slices (their longest row).
__global__ void __launch_bounds__(kBlock)
    slice_order_kernel(int64_t n, const int64_t *ptr, uint8_t *order, uint8_t *place, int32_t *len,
                       int64_t *width32) {
  __shared__ int l_sh[kBlock];
  const int64_t groups = ceil_div(n, kBlock), slices = ceil_div(n, 32);
  for (int64_t g = blockIdx.x; g < groups; g += gridDim.x) {
    const int64_t i = g * kBlock + threadIdx.x;
    const int l = i < n ? (int)(ptr[i + 1] - ptr[i]) : -1;
    __syncthreads();
    l_sh[threadIdx.x] = l;
    __syncthreads();
    int rank = 0;
    const int l8 = l >> 3;  // -1 past the last row: last
    for (int t = 0; t < kBlock; ++t) {
      const int o8 = l_sh[t] >> 3;
      rank += o8 > l8 || (o8 == l8 && t < (int)threadIdx.x);
    }
    if (i < n) {
      order[g * kBlock + rank] = (uint8_t)threadIdx.x;
      place[i] = (uint8_t)rank;
      len[g * kBlock + rank] = l;
    }
    __syncthreads();
    l_sh[rank] = l > 0 ? l : 0;
    __syncthreads();
    const int w = __reduce_max_sync(0xffffffffu, l_sh[threadIdx.x]);
    if (threadIdx.x % 32 == 0 && i / 32 < slices) width32[i / 32] = (int64_t)w * 32;
  }
}

// One block per group: the words (32 columns each) its rows touch, ascending,
// with their column masks; counts of words and columns.  *refused is set when
// a group has more than the caps.
__global__ void __launch_bounds__(kBlock)
    dict_words_kernel(int64_t n, const int64_t *ptr, const int32_t *col, int32_t *word_key,
                      uint32_t *word_mask, int32_t *nwords, int64_t *ncols, int *most,
                      int *refused) {
  __shared__ int32_t key[kWordTable];
  __shared__ uint32_t mask[kWordTable];
  __shared__ unsigned long long item[kWordCap];  // key << 32 | mask, for the sort
  __shared__ int used, total;
  const int64_t groups = ceil_div(n, kBlock);
  for (int64_t g = blockIdx.x; g < groups; g += gridDim.x) {
    for (int t = threadIdx.x; t < kWordTable; t += kBlock) {
      key[t] = -1;
      mask[t] = 0u;
    }
    if (threadIdx.x == 0) used = total = 0;
    __syncthreads();
    const int64_t r0 = g * kBlock, r1 = r0 + kBlock < n ? r0 + kBlock : n;
    const int64_t k1 = ptr[r1];
    for (int64_t k = ptr[r0] + threadIdx.x; k < k1; k += kBlock) {
      const int32_t c = col[k], w = c >> 5;
      const uint32_t bit = 1u << (c & 31);
      uint32_t h = ((uint32_t)w * 2654435761u) >> 21;  // multiplicative hash, 11 bits
      for (int probe = 0; probe < kWordTable; ++probe, h = (h + 1) & (kWordTable - 1)) {
        int32_t at = key[h];
        if (at == -1) {
          at = atomicCAS(&key[h], -1, w);
          if (at == -1) {
            atomicAdd(&used, 1);
            at = w;
          }
        }
        if (at == w) {
          if (!(mask[h] & bit)) atomicOr(&mask[h], bit);
          break;
        }
      }
    }
    __syncthreads();
    const int nw = used;
    __syncthreads();
    if (nw > kWordCap) {
      if (threadIdx.x == 0) {
        *refused = 1;
        nwords[g] = 0;
        ncols[g] = 0;
      }
      continue;
    }
    if (threadIdx.x == 0) used = 0;
    __syncthreads();
    int mine = 0;
    for (int t = threadIdx.x; t < kWordTable; t += kBlock)
      if (key[t] != -1) {
        item[atomicAdd(&used, 1)] =
            ((unsigned long long)(uint32_t)key[t] << 32) | (unsigned long long)mask[t];
        mine += __popc(mask[t]);
      }
    if (mine) atomicAdd(&total, mine);
    int P2 = 1;
    while (P2 < nw) P2 <<= 1;
    __syncthreads();
    for (int t = nw + threadIdx.x; t < P2; t += kBlock) item[t] = ~0ull;
    __syncthreads();
    for (int k = 2; k <= P2; k <<= 1)
      for (int j = k >> 1; j > 0; j >>= 1) {
        for (int t = threadIdx.x; t < P2; t += kBlock) {
          const int u = t ^ j;
          if (u > t) {
            const unsigned long long a = item[t], b = item[u];
            if ((a > b) == ((t & k) == 0)) {
              item[t] = b;
              item[u] = a;
            }
          }
        }
        __syncthreads();
      }
    for (int t = threadIdx.x; t < nw; t += kBlock) {
      word_key[g * kWordCap + t] = (int32_t)(item[t] >> 32);
      word_mask[g * kWordCap + t] = (uint32_t)item[t];
    }
    if (threadIdx.x == 0) {
      nwords[g] = nw;
      ncols[g] = total;
      atomicMax(most, total);
      if (total > kDictCap) *refused = 1;
    }
    __syncthreads();
  }
}

// One block per group: the dictionary's columns, and the rows' 16-bit places in
// slice order (with the values of an array in CSR order, if any).  A warp
// transposes its slice 16 entries at a time through shared memory, so that both
// sides are coalesced.
constexpr int kTile = 16;
struct SliceTile {
  double v[32][kTile + 1];
  uint16_t c[32][kTile + 2];
};
__global__ void __launch_bounds__(kBlock)
    slice_fill_kernel(int64_t n, const int64_t *ptr, const int32_t *col, const double *val,
                      const int32_t *word_key, const uint32_t *word_mask, const int32_t *nwords,
                      const int64_t *dptr, const int64_t *sptr, const uint8_t *order,
                      int32_t *dict, uint16_t *idx, double *out) {
  extern __shared__ __align__(16) unsigned char fill_smem[];
  SliceTile *tiles = reinterpret_cast<SliceTile *>(fill_smem);
  int32_t *key = reinterpret_cast<int32_t *>(tiles + kWarpsPerBlock);
  uint32_t *mask = reinterpret_cast<uint32_t *>(key + kWordCap);
  int32_t *pre = reinterpret_cast<int32_t *>(mask + kWordCap);
  __shared__ int wsum[kWarpsPerBlock];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  SliceTile &T = tiles[wid];
  const int64_t groups = ceil_div(n, kBlock);
  for (int64_t g = blockIdx.x; g < groups; g += gridDim.x) {
    const int nw = nwords[g];
    const int64_t d0 = dptr[g];
    __syncthreads();
    for (int t = threadIdx.x; t < nw; t += kBlock) {
      key[t] = word_key[g * kWordCap + t];
      mask[t] = word_mask[g * kWordCap + t];
    }
    __syncthreads();
    // exclusive prefix of the words' column counts: 4 words a thread
    static_assert(kWordCap == 4 * kBlock, "the prefix gives each thread four words");
    int cnt[4], mine = 0;
    for (int q = 0; q < 4; ++q) {
      const int t = threadIdx.x * 4 + q;
      cnt[q] = t < nw ? __popc(mask[t]) : 0;
      mine += cnt[q];
    }
    int inc = mine;
    for (int o = 1; o < 32; o <<= 1) {
      const int v = __shfl_up_sync(0xffffffffu, inc, o);
      if (lane >= o) inc += v;
    }
    if (lane == 31) wsum[wid] = inc;
    __syncthreads();
    int at = inc - mine;
    for (int w = 0; w < wid; ++w) at += wsum[w];
    for (int q = 0; q < 4; ++q) {
      const int t = threadIdx.x * 4 + q;
      if (t < nw) {
        pre[t] = at;
        int o = at;
        for (uint32_t m = mask[t]; m; m &= m - 1) dict[d0 + o++] = key[t] * 32 + __ffs(m) - 1;
      }
      at += cnt[q];
    }
    __syncthreads();
    const int64_t slice = g * kWarpsPerBlock + wid, r0 = slice * 32;
    if (r0 < n) {
      const int rows = (int)(n - r0 < 32 ? n - r0 : 32);
      const int64_t base = sptr[slice];
      const int width = (int)((sptr[slice + 1] - base) / 32);
      const int64_t row = g * kBlock + (lane < rows ? order[r0 + lane] : 0);
      const int64_t mybeg = lane < rows ? ptr[row] : 0;
      const int mylen = lane < rows ? (int)(ptr[row + 1] - mybeg) : 0;
      for (int t0 = 0; t0 < width; t0 += kTile) {
        // two rows at a time, 16 consecutive entries of each
        const int half = lane / kTile, t = lane % kTile;
        for (int r = 0; r < 32; r += 2) {
          const int64_t b = __shfl_sync(0xffffffffu, mybeg, r + half);
          const int l = __shfl_sync(0xffffffffu, mylen, r + half);
          uint16_t place = 0;
          double v = 0.0;
          if (t0 + t < l) {
            const int64_t k = b + t0 + t;
            const int32_t c = col[k], w = c >> 5;
            int lo = 0, hi = nw - 1;  // the word is in the list
            while (lo < hi) {
              const int mid = (lo + hi) >> 1;
              if (key[mid] < w) lo = mid + 1; else hi = mid;
            }
            place = (uint16_t)(pre[lo] + __popc(mask[lo] & ((1u << (c & 31)) - 1u)));
            if (val) v = val[k];
          }
          T.c[r + half][t] = place;
          T.v[r + half][t] = v;
        }
        __syncwarp();
        for (int q = 0; q < kTile && t0 + q < width; ++q) {
          const int64_t k = base + (int64_t)(t0 + q) * 32 + lane;
          idx[k] = T.c[lane][q];
          if (out) out[k] = T.v[lane][q];
        }
        __syncwarp();
      }
    }
  }
}

// Moves an array between the orders, in OUT's type.  TO_SLICES: padding gets 0.
template <typename IN, typename OUT, bool TO_SLICES>
__global__ void __launch_bounds__(kBlock)
    slice_move_kernel(int64_t n, const int64_t *ptr, const int64_t *sptr, const uint8_t *order,
                      const IN *in, OUT *out) {
  __shared__ OUT tile_sh[kWarpsPerBlock][32][kTile + 1];
  OUT(*T)[kTile + 1] = tile_sh[threadIdx.x >> 5];
  const int lane = threadIdx.x & 31;
  const int64_t warp = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
  for (int64_t slice = warp; slice * 32 < n; slice += nwarps) {
    const int64_t r0 = slice * 32;
    const int rows = (int)(n - r0 < 32 ? n - r0 : 32);
    const int64_t base = sptr[slice];
    const int width = (int)((sptr[slice + 1] - base) / 32);
    const int64_t row = r0 / kBlock * kBlock + (lane < rows ? order[r0 + lane] : 0);
    const int64_t mybeg = lane < rows ? ptr[row] : 0;
    const int mylen = lane < rows ? (int)(ptr[row + 1] - mybeg) : 0;
    const int half = lane / kTile, t = lane % kTile;
    for (int t0 = 0; t0 < width; t0 += kTile) {
      if (!TO_SLICES) {
        for (int q = 0; q < kTile && t0 + q < width; ++q)
          T[lane][q] = (OUT)in[base + (int64_t)(t0 + q) * 32 + lane];
        __syncwarp();
      }
      for (int r = 0; r < 32; r += 2) {
        const int64_t b = __shfl_sync(0xffffffffu, mybeg, r + half);
        const int l = __shfl_sync(0xffffffffu, mylen, r + half);
        const bool in_row = t0 + t < l;
        if (TO_SLICES)
          T[r + half][t] = in_row ? (OUT)in[b + t0 + t] : OUT(0);
        else if (in_row)
          out[b + t0 + t] = T[r + half][t];
      }
      __syncwarp();
      if (TO_SLICES) {
        for (int q = 0; q < kTile && t0 + q < width; ++q)
          out[base + (int64_t)(t0 + q) * 32 + lane] = T[lane][q];
        __syncwarp();
      }
    }
  }
}

template <typename IN, typename OUT, bool TO_SLICES>
static sph_rt_status slice_move(sph_rt *s, int64_t n, const int64_t *ptr, const SlicedRowsData &d,
                                const IN *in, OUT *out) {
  slice_move_kernel<IN, OUT, TO_SLICES>
      <<<blocks_for(s, ceil_div(n, 32), kWarpsPerBlock, 6), kBlock, 0, s->stream>>>(n, ptr, d.ptr,
                                                                                   d.order, in, out);
  SPH_LAUNCHED(s);
  return SPH_RT_OK;
}

// Slices and dictionaries of the CSR rows (ptr, col); with `val`, those values in
// slice order too.  *ok = false: a group's columns exceed the caps.  Buffers come
// from `take`; *out and *out_val hold those taken so far whatever the outcome, and
// the caller releases them where the slices are not kept.
sph_rt_status sliced_build(sph_rt *s, int64_t n, const int64_t *ptr, const int32_t *col,
                           const double *val, void *(*take)(sph_rt *, void *, size_t), void *owner,
                           SlicedRowsData *out, double **out_val, bool *ok) {
  *ok = false;
  *out = SlicedRowsData{};
  if (out_val) *out_val = nullptr;
  cudaStream_t st = s->stream;
  const int64_t slices = ceil_div(n, 32), groups = ceil_div(n, kBlock);
  SlicedRowsData &D = *out;  // filled in as it is allocated
  struct Scratch {           // back to the free list on every return
    sph_rt *s;
    std::vector<void *> held;
    ~Scratch() {
      cudaStreamSynchronize(s->stream);
      for (void *p : held) dfree(s, p);
    }
    void *take(size_t bytes) {
      held.push_back(dalloc_bytes(s, bytes));
      return held.back();
    }
  } tmp{s, {}};
  int32_t *key = (int32_t *)tmp.take(sizeof(int32_t) * groups * kWordCap);
  uint32_t *mask = (uint32_t *)tmp.take(sizeof(uint32_t) * groups * kWordCap);
  int32_t *nw = (int32_t *)tmp.take(sizeof(int32_t) * groups);
  int64_t *nc = (int64_t *)tmp.take(sizeof(int64_t) * groups);
  int64_t *w32 = (int64_t *)tmp.take(sizeof(int64_t) * slices);
  int *flags = (int *)tmp.take(sizeof(int) * 2);  // largest dictionary, refused
  if (!key || !nw || !mask || !nc || !w32 || !flags) return SPH_RT_ENOMEM;
  SPH_CUDA(s, cudaMemsetAsync(flags, 0, 2 * sizeof(int), st));
  dict_words_kernel<<<blocks_for(s, groups, 1, 6), kBlock, 0, st>>>(n, ptr, col, key, mask, nw, nc,
                                                                    flags, flags + 1);
  SPH_LAUNCHED(s);
  int hf[2] = {0, 0};
  SPH_CUDA(s, cudaMemcpyAsync(hf, flags, sizeof hf, cudaMemcpyDeviceToHost, st));
  SPH_CUDA(s, cudaStreamSynchronize(st));
  if (hf[1]) return SPH_RT_OK;
  D.dict_max = hf[0];
  D.len = (int32_t *)take(s, owner, sizeof(int32_t) * n);
  D.ptr = (int64_t *)take(s, owner, sizeof(int64_t) * (slices + 1));
  D.dptr = (int64_t *)take(s, owner, sizeof(int64_t) * (groups + 1));
  D.order = (uint8_t *)take(s, owner, n);
  D.place = (uint8_t *)take(s, owner, n);
  if (!D.len || !D.ptr || !D.dptr || !D.order || !D.place) return SPH_RT_ENOMEM;
  static_assert(kBlock == 256, "a place within a group is a byte");
  slice_order_kernel<<<blocks_for(s, groups, 1, 8), kBlock, 0, st>>>(n, ptr, D.order, D.place,
                                                                    D.len, w32);
  SPH_LAUNCHED(s);
  sph_rt_status rc;
  if ((rc = exclusive_scan(s, w32, slices, D.ptr))) return rc;
  if ((rc = exclusive_scan(s, nc, groups, D.dptr))) return rc;
  int64_t total[2];
  SPH_CUDA(s, cudaMemcpyAsync(&total[0], D.ptr + slices, sizeof(int64_t), cudaMemcpyDeviceToHost, st));
  SPH_CUDA(s, cudaMemcpyAsync(&total[1], D.dptr + groups, sizeof(int64_t), cudaMemcpyDeviceToHost, st));
  SPH_CUDA(s, cudaStreamSynchronize(st));
  D.padded = total[0];
  D.idx = (uint16_t *)take(s, owner, sizeof(uint16_t) * (D.padded + 1));
  D.dict = (int32_t *)take(s, owner, sizeof(int32_t) * (total[1] + 1));
  double *v = val ? (double *)take(s, owner, sizeof(double) * (D.padded + 1)) : nullptr;
  if (out_val) *out_val = v;
  if (!D.idx || !D.dict || (val && !v)) return SPH_RT_ENOMEM;
  const int smem = (int)(sizeof(SliceTile) * kWarpsPerBlock + 12 * kWordCap);
  SPH_CUDA(s, cudaFuncSetAttribute(slice_fill_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                   smem));
  slice_fill_kernel<<<blocks_for(s, groups, 1, 3), kBlock, smem, st>>>(
      n, ptr, col, val, key, mask, nw, D.dptr, D.ptr, D.order, D.dict, D.idx,
      v);
  SPH_LAUNCHED(s);
  *ok = true;
  return SPH_RT_OK;
}

static void *take_handle(sph_rt *s, void *, size_t bytes) { return dalloc_bytes(s, bytes); }
static void release_slices(sph_rt *s, const SlicedRowsData &d, double *G, double *val,
                           float *val32) {
  void *bufs[] = {d.ptr, d.dptr, d.idx, d.len, d.dict, d.order, d.place, G, val, val32};
  for (void *p : bufs) dfree(s, p);
}

// The fine operator's slices, before the particle set's first assembly: geometry
// moved from mat_G, which is released with the CSR values.  Tried once per particle
// set: buffers of the kept AMG hierarchy and of the captured step graph refer to the
// layout, so a set never changes to slices later.  Without room for them, or with too
// large a dictionary, the CSR rows stay.
sph_rt_status sliced_operator(sph_rt *s) {
  if (s->sl_decided) return SPH_RT_OK;
  s->sl_decided = true;
  if (!sliced_wanted(s)) return SPH_RT_OK;
  bool ok = false;
  SlicedRowsData d;
  double *G = nullptr, *val = nullptr;
  float *val32 = nullptr;
  sph_rt_status rc = sliced_build(s, s->n_int, s->mat_ptr, s->mat_col, s->mat_G, take_handle,
                                  nullptr, &d, &G, &ok);
  if (rc == SPH_RT_OK && ok) {
    val = dalloc<double>(s, d.padded + 1);  // + 1: never of size 0
    if (s->cfg.precision == SPH_RT_MIXED) val32 = dalloc<float>(s, d.padded + 1);
    if (!val || (s->cfg.precision == SPH_RT_MIXED && !val32)) rc = SPH_RT_ENOMEM;
  }
  if (rc != SPH_RT_OK || !ok) {
    release_slices(s, d, G, val, val32);
    if (rc != SPH_RT_OK && rc != SPH_RT_ENOMEM) return rc;
    s->err.clear();
    return SPH_RT_OK;
  }
  s->sl = d;
  s->sl_G = G;
  s->sl_val = val;
  s->sl_val32 = val32;
  dfree(s, s->mat_G);
  dfree(s, s->mat_val);
  dfree(s, s->mat_val32);
  s->mat_G = s->mat_val = nullptr;
  s->mat_val32 = nullptr;
  return SPH_RT_OK;
}

// The current values in CSR order (a scratch buffer of nnz_mat doubles; the
// caller releases it), for the AMG set-up.
sph_rt_status sliced_to_csr(sph_rt *s, double **csr) {
  *csr = dalloc<double>(s, s->nnz_mat);
  if (!*csr) return SPH_RT_ENOMEM;
  return slice_move<double, double, false>(s, s->n_int, s->mat_ptr, s->sl, s->sl_val, *csr);
}

// Back to the CSR rows, whose values the next assembly writes.  Without room for them
// the slices stay.
sph_rt_status sliced_undo(sph_rt *s) {
  double *G = dalloc<double>(s, s->nnz_mat), *val = dalloc<double>(s, s->nnz_mat);
  float *val32 = s->sl_val32 ? dalloc<float>(s, s->nnz_mat) : nullptr;
  sph_rt_status rc = G && val && (val32 || !s->sl_val32) ? SPH_RT_OK : SPH_RT_ENOMEM;
  if (!rc) rc = slice_move<double, double, false>(s, s->n_int, s->mat_ptr, s->sl, s->sl_G, G);
  cudaStreamSynchronize(s->stream);
  if (rc) {
    release_slices(s, SlicedRowsData{}, G, val, val32);
    return rc;
  }
  release_slices(s, s->sl, s->sl_G, s->sl_val, s->sl_val32);
  s->sl = SlicedRowsData{};
  s->sl_G = s->sl_val = nullptr;
  s->sl_val32 = nullptr;
  s->mat_G = G;
  s->mat_val = val;
  s->mat_val32 = val32;
  return SPH_RT_OK;
}

// ---------------------------------------------------------------------------
// values of A P
// ---------------------------------------------------------------------------
// pos[k]: place within its row's A P entries of the aggregate of entry k (slice
// order; kNoPlace: unaggregated column), from the CSR-order map of relative
// places (-1: none).
static_assert((uint16_t)(-1) == kNoPlace, "a place of -1 is stored as kNoPlace");
sph_rt_status sliced_places(sph_rt *s, const int32_t *map, uint16_t *pos) {
  return slice_move<int32_t, uint16_t, true>(s, s->n_int, s->mat_ptr, s->sl, map, pos);
}

// A thread per row adds its entries, in list order, to the row's A P entries (the
// diagonal first, into entry 0, the row's own aggregate).  The sums are kept in shared
// memory, entry q of thread t at [q][t] (no bank conflicts).
// Replaces a gather over 4-byte source lists with one thread per A P entry:
// 1.0 -> 0.36 ms a step in FP32 at 128^3 (2.18e8 entries), 0.10 ms in FP64 at 64^3.
// WINDOWS: rows of more A P entries than kApSmemMax holds walk their own entries once per
// `window` of them, of the half that leaves room for two blocks an SM: 7.0e7 FP64 entries
// of rows of 223 0.66 ms (summed in the A P array itself 1.07; windows of a third 0.71, of
// the whole 0.74).  One window is the faster form wherever it fits, even with one block an
// SM (244 entries a row, < 100 in A P: 0.79 ms against 1.06 in windows).
template <typename T, bool WINDOWS>
__global__ void __launch_bounds__(kBlock)
    ap_values_kernel(int64_t n, SlicedRowsData A, const uint16_t *pos, const T *val,
                     const T *diag, const int32_t *agg, SlicedRowsData ap, int window, T *ap_val) {
  extern __shared__ __align__(16) unsigned char ap_smem[];
  T *acc = reinterpret_cast<T *>(ap_smem) + threadIdx.x;
  const int64_t groups = ceil_div(n, kBlock);
  for (int64_t g = blockIdx.x; g < groups; g += gridDim.x) {
    const int64_t at = g * kBlock + threadIdx.x;  // place in the operator's slices
    if (at >= n) continue;
    const int64_t i = g * kBlock + A.order[at];   // its row
    const int q0 = ap.place[i];                   // the row's place in A P's slices
    const int m = ap.len[g * kBlock + q0], l = A.len[at];
    const int64_t o0 = ap.ptr[g * kWarpsPerBlock + q0 / 32] + q0 % 32;
    const int64_t k0 = A.ptr[at >> 5] + (threadIdx.x & 31);
    for (int w0 = 0; w0 < m; w0 += WINDOWS ? window : m) {
      const int mw = WINDOWS && m - w0 > window ? window : m - w0;
      for (int q = 0; q < mw; ++q) acc[q * kBlock] = T(0);
      if (w0 == 0 && agg[i] >= 0) acc[0] = diag[i];
      constexpr int U = 8;
      for (int t = 0; t < l; t += U) {
        int p[U];
        T v[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
          const bool in = t + u < l;
          p[u] = in ? (int)__ldg(pos + k0 + (int64_t)(t + u) * 32) : kNoPlace;
          v[u] = in ? __ldg(val + k0 + (int64_t)(t + u) * 32) : T(0);
        }
#pragma unroll
        for (int u = 0; u < U; ++u)
          if (WINDOWS ? (unsigned)(p[u] - w0) < (unsigned)mw : p[u] != kNoPlace)
            acc[(p[u] - w0) * kBlock] += v[u];
      }
      for (int q = 0; q < mw; ++q) ap_val[o0 + (int64_t)(w0 + q) * 32] = acc[q * kBlock];
    }
  }
}

template <typename T>
sph_rt_status sliced_ap_values(sph_rt *s, const uint16_t *pos, const int32_t *agg,
                               const SlicedRowsData &ap, int ap_most, const T *val, const T *diag,
                               T *ap_val) {
  constexpr int entry = kBlock * (int)sizeof(T);  // of one A P entry of a block's rows
  const int grid = blocks_for(s, ceil_div(s->n_int, kBlock), 1, 8);
  if (ap_most * entry <= kApSmemMax) {
    SPH_CUDA(s, cudaFuncSetAttribute(ap_values_kernel<T, false>,
                                     cudaFuncAttributeMaxDynamicSharedMemorySize, kApSmemMax));
    ap_values_kernel<T, false><<<grid, kBlock, ap_most * entry, s->stream>>>(
        s->n_int, s->sl, pos, val, diag, agg, ap, ap_most, ap_val);
  } else {
    const int64_t passes = ceil_div(ap_most, kApSmemMax / 2 / entry);
    const int window = (int)ceil_div(ap_most, passes);
    SPH_CUDA(s, cudaFuncSetAttribute(ap_values_kernel<T, true>,
                                     cudaFuncAttributeMaxDynamicSharedMemorySize, kApSmemMax / 2));
    ap_values_kernel<T, true><<<grid, kBlock, window * entry, s->stream>>>(
        s->n_int, s->sl, pos, val, diag, agg, ap, window, ap_val);
  }
  SPH_LAUNCHED(s);
  return SPH_RT_OK;
}
template sph_rt_status sliced_ap_values<double>(sph_rt *, const uint16_t *, const int32_t *,
                                                const SlicedRowsData &, int, const double *,
                                                const double *, double *);
template sph_rt_status sliced_ap_values<float>(sph_rt *, const uint16_t *, const int32_t *,
                                               const SlicedRowsData &, int, const float *,
                                               const float *, float *);

}  // namespace sphrt
