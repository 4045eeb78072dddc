// sliced.cuh -- building and using sliced operators (sliced.cu).
#pragma once

#include <cstring>

#include "common.cuh"

namespace sphrt {

// Levels at or below this many stored entries (~7 MB in FP64, L2-resident)
// may run in the cluster-resident tail of the V-cycle (which must hold at least
// two levels); the larger levels post-smooth through A P.
constexpr int64_t kTailMaxNnz = 600000;
constexpr int kSliceMinGroups = 2;
constexpr int kNoPlace = 0xffff;            // sliced A P: column without an aggregate
constexpr int kApSmemMax = 200 * 1024;      // of a block that sums A P entries

sph_rt_status sliced_operator(sph_rt *s);
sph_rt_status sliced_to_csr(sph_rt *s, double **csr);
sph_rt_status sliced_undo(sph_rt *s);
sph_rt_status sliced_build(sph_rt *s, int64_t n, const int64_t *ptr, const int32_t *col,
                           const double *val, void *(*take)(sph_rt *, void *, size_t), void *owner,
                           SlicedRowsData *out, double **out_val, bool *ok);
sph_rt_status sliced_places(sph_rt *s, const int32_t *map, uint16_t *pos);
template <typename T>
sph_rt_status sliced_ap_values(sph_rt *s, const uint16_t *pos, const int32_t *agg,
                               const SlicedRowsData &ap, int ap_most, const T *val, const T *diag,
                               T *ap_val);

template <typename T>
inline SlicedView<T> sliced_view(const SlicedRowsData &d, int64_t n, int64_t nnz, const T *val,
                                 const T *diag, const T *invdiag) {
  SlicedView<T> A;
  memset(&A, 0, sizeof A);
  A.n = n;
  A.ptr = d.ptr;
  A.idx = d.idx;
  A.val = val;
  A.len = d.len;
  A.order = d.order;
  A.dptr = d.dptr;
  A.dict = d.dict;
  A.diag = diag;
  A.invdiag = invdiag;
  A.nnz = nnz;
  A.dict_max = d.dict_max;
  return A;
}
// the fine operator in slices, FP64 or the mixed form's FP32 copy
template <typename T>
inline SlicedView<T> fine_sliced(const sph_rt *s);
template <>
inline SlicedView<double> fine_sliced<double>(const sph_rt *s) {
  return sliced_view<double>(s->sl, s->n_int, s->nnz_mat, s->sl_val, s->diag, s->invdiag);
}
template <>
inline SlicedView<float> fine_sliced<float>(const sph_rt *s) {
  return sliced_view<float>(s->sl, s->n_int, s->nnz_mat, s->sl_val32, s->diag32, s->invdiag32);
}

// Grid of a sweep over slices: a block per group, at most one wave.
inline int sliced_grid(const sph_rt *s, int64_t n, int blocks_per_sm) {
  const int64_t g = ceil_div(n > 0 ? n : 1, kBlock), cap = (int64_t)s->num_sms * blocks_per_sm;
  return (int)(g < cap ? g : cap);
}

}  // namespace sphrt

// Launch KERNEL<Rows, ...> over the fine operator, sliced or in CSR row tiles:
// CALL uses `Rows` (the row-source type), `rows` (its value), `grid` and `smem`.
#define SPH_FINE_ROWS(s_, MT_, A_, VB_, CALL)                                        \
  do {                                                                               \
    if ((s_)->sl.ptr) {                                                              \
      using Rows = SlicedRows<MT_>;                                                  \
      const Rows rows{fine_sliced<MT_>(s_)};                                         \
      const int grid = sliced_grid(s_, (s_)->n_int, Rows::kMinBlocks);               \
      const size_t smem = (size_t)(s_)->sl.dict_max * (VB_);                         \
      CALL;                                                                          \
    } else {                                                                         \
      const size_t smem = 0;                                                         \
      SPH_DISPATCH_SHAPE((A_).W, (A_).U, ({                                          \
                           using Rows = CsrRows<W, U, MT_>;                          \
                           const Rows rows{A_};                                      \
                           const int grid = row_grid((s_)->num_sms, (A_).n, W, U);   \
                           CALL;                                                     \
                         }));                                                        \
    }                                                                                \
  } while (0)
