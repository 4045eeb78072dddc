// common.cuh -- shared device helpers and the internal handle of libsphrt.
//
// Index spaces.  Particles are sorted once by (ghost flag, Morton code of the
// cell, caller index), so "slots" [0, n_int) are the interior particles in
// Morton order and [n_int, n) the ghosts.  Unknowns of the radiation system
// are the interior slots, so an unknown's index IS its slot and the solver
// needs no index maps.
//
// Operator scaling.  The library stores B = V A, V = diag(m/rho), where A is
// the paper's row operator of Eq. diffusion-solve.  B_ij = V_i V_j F_ij (D_i +
// D_j) is bitwise symmetric (V_i V_j commutes, F_ij is the symmetric two-h
// average) and B is an M-matrix, so the Krylov solver is CG and the AMG
// hierarchy is built from symmetric Galerkin products.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>
#include <stdio.h>

#include <cstring>

#include <map>
#include <string>
#include <unordered_map>
#include <vector>

#include "../../include/sph_rt.h"

namespace sphrt {

constexpr int kBlock = 256;          // threads per block of the 1-D kernels
constexpr int kWarpsPerBlock = kBlock / 32;
constexpr int kMaxRedBlocks = 2048;  // upper bound on blocks of a reducing kernel
// Resident blocks per SM the SpMV-class sweeps are compiled for, i.e. their
// register cap (65536 / (kBlock * blocks)): 5 blocks (48 registers) with U = 4
// loads in flight per lane, 4 blocks (64 registers) with U = 8.  Their grids
// never exceed this many blocks per SM (row_grid), so one wave covers all rows.
__host__ __device__ constexpr int sweep_min_blocks(int U) { return U >= 8 ? 4 : 5; }
// The coarse levels' sweeps (a few thousand to a few tens of thousands of
// L2-resident rows: latency-bound, not throughput-bound) also load their row
// operands before the row sums, which takes them to 64 registers.
constexpr int kCoarseMinBlocks = 4;

// --------------------------------------------------------------------------
// Scalars of one Krylov solve and of the outer loop, kept on the device so
// that the iteration runs without host round trips between kernels.
// --------------------------------------------------------------------------
struct Scalars {
  double rho;      // (r, z)
  double alpha;    // rho / (p, q)
  double beta;     // rho_new / rho
  double pq;       // (p, B p)
  double rnorm2;   // ||r / V||^2 (unscaled residual)
  double bnorm2;   // ||b||^2 (unscaled right-hand side)
  double thresh2;  // tol^2 ||b||^2
  double red[8];   // results of generic reductions
  int done;        // Krylov converged (or aborted)
  int iters;       // Krylov iterations taken
  int breakdown;   // non-positive curvature / NaN seen
  int bad_input;   // a step input (source or ghost value) was not finite
  int gate_timeout;  // a timing gate gave up waiting for the host (timing only)
  unsigned int counter;  // arrival counter of the last-block reductions
  // outer (nonlinear-elimination) loop of Alg. 1, advanced by the material solve (outer_check)
  int outer_iters;       // completed outer iterations
  int outer_status;      // 0 running, 1 converged, 2 Krylov failure, 3 max_outer reached
  int outer_trips;       // loop trips (termination guard of the device-driven loop)
  int krylov_total;      // Krylov iterations over the converged outer iterations
  int krylov_trips;      // Krylov loop trips over all outer iterations (launch count)
  int krylov_solve_trips;  // Krylov loop trips of the current solve (termination guard)
  int newton_max;        // largest material Newton iteration count
  int krylov_per_outer[64];
  double last_change_e, last_change_E;
  double energy_before_e, energy_before_E;  // interior totals at the start of the step
  // CG with the V-cycle's product (fine_post_smooth = 0)
  int pfirst;      // the next update starts the directions: p = z, q = B z
  int ru;          // mixed form: the next launch replaces r by the FP64 residual
  double rmax2;    // mixed form: largest ||r / V||^2 since the last replacement
  int yvalid;      // mixed form: the last solve ended on a verified residual whose B x
                   // (kept in the handle's w) is that of the next solve's start
  // time step choice of the last converged step (config.dt_target > 0)
  double dtc_ebar, dtc_Ebar, dtc_eta_e, dtc_eta_E, dtc_next;
  // start of the first solve of a step: x = sum_j guess_w[j] E^{n-1-j}, j <= guess_order
  // (E^{n-1} = E^l; guess_order 0: x = E^l)
  double guess_w[4];
  int guess_order;
};

// Lagrange extrapolation in time of order p (0..3): the weights w[0..p] with
// sum_j w[j] E(t_{n-1-j}) the value at t_n of the polynomial of degree p through
// E^{n-1}, ..., E^{n-1-p}.  dt is t_n - t_{n-1}; d[j] = t_{n-1-j} - t_{n-2-j}
// are the previous steps' sizes.  p = 1: w = (1 + dt/d0, -dt/d0).
__host__ __device__ inline void extrap_weights(int p, double dt, const double *d, double *w) {
  double tau[4];  // node times relative to t_{n-1}
  tau[0] = 0.0;
  for (int j = 1; j <= p; ++j) tau[j] = tau[j - 1] - d[j - 1];
  for (int j = 0; j <= p; ++j) {
    double num = 1.0, den = 1.0;
    for (int m = 0; m <= p; ++m) {
      if (m == j) continue;
      num *= dt - tau[m];
      den *= tau[j] - tau[m];
    }
    w[j] = num / den;
  }
}

// --------------------------------------------------------------------------
// Warp and block reductions (fixed order: deterministic).
// --------------------------------------------------------------------------
__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
  return v;
}
__device__ __forceinline__ double warp_max(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v = fmax(v, __shfl_down_sync(0xffffffffu, v, o));
  return v;
}
template <int W>
__device__ __forceinline__ double group_sum(double v) {
#pragma unroll
  for (int o = W / 2; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o, W);
  return v;
}

// Reduction of NV values over a block of kBlock threads, valid in thread 0: sums, or
// maxima (of non-negative quantities) where is_max[k].  Every thread calls it, twice in
// a kernel only with a barrier between.
//
// An FP64 operation costs a warp 16 cycles of its SM whatever its active lanes, so a
// shuffle tree in each of the 8 warps is 8 x 5 of them per value.  Here the warps
// shuffle once (twice with several values: shared memory is what the sliced rows'
// dictionaries leave) and ONE warp per value adds what they left, in a fixed order:
// 8 + 3 + 5 operations per value (16 + 1 + 5).  With the ticket below: newton at 1,024
// particles 11.2 -> 9.3 us, step_end 11.1 -> 7.1, spmv_pq 6.1 -> 5.3; update at 2.5e5
// rows 12.4 -> 10.9.
template <int NV>
__device__ __forceinline__ void block_reduce(double (&v)[NV], const bool (&is_max)[NV]) {
  static_assert(NV <= kWarpsPerBlock, "one warp per value");
  constexpr int R = NV == 1 ? 1 : 2;                 // shuffles before shared memory
  constexpr int N = kBlock >> R;                     // values left, of each
  __shared__ double sh[NV][N];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
#pragma unroll
  for (int k = 0; k < NV; ++k) {
#pragma unroll
    for (int o = 16; o > (16 >> R); o >>= 1) {
      const double u = __shfl_xor_sync(0xffffffffu, v[k], o);
      v[k] = is_max[k] ? fmax(v[k], u) : v[k] + u;
    }
    if (lane < (32 >> R)) sh[k][wid * (32 >> R) + lane] = v[k];
  }
  __syncthreads();
  if (wid < NV) {
    const double *p = sh[wid] + lane;
    bool mx = false;
#pragma unroll
    for (int k = 0; k < NV; ++k)
      if (wid == k) mx = is_max[k];
    double x = p[0], y = p[32];
#pragma unroll
    for (int w = 64; w < N; w += 64) {
      x = mx ? fmax(x, p[w]) : x + p[w];
      y = mx ? fmax(y, p[w + 32]) : y + p[w + 32];
    }
    x = mx ? warp_max(fmax(x, y)) : warp_sum(x + y);
    if (NV == 1)
      v[0] = x;
    else if (lane == 0)
      sh[wid][0] = x;
  }
  if (NV > 1) {
    __syncthreads();
#pragma unroll
    for (int k = 0; k < NV; ++k) v[k] = sh[k][0];
  }
}

template <int NV>
__device__ __forceinline__ void block_sums(double (&v)[NV]) {
  const bool mx[NV] = {};
  block_reduce<NV>(v, mx);
}

// Last-block reduction: every block stores its NV partial values, the block
// that arrives last combines all partials in block order (so the result does
// not depend on scheduling) and returns true in all its threads; `out` then
// holds the NV totals in thread 0 (sums, or maxima where is_max[k]).
//
// The ticket is taken with acquire-release order: it publishes the partials of
// thread 0 and, in the last block, makes all of them visible behind the barrier.  (A
// __threadfence before it and one per thread after it are sequentially consistent
// fences, of ~1 us each on the critical path of every reduction.)
template <int NV>
__device__ bool last_block_combine(const double (&part)[NV], double *partials, unsigned *counter,
                                   double (&out)[NV], const bool (&is_max)[NV]) {
  __shared__ bool am_last;
  if (threadIdx.x == 0) {
    for (int k = 0; k < NV; ++k) partials[(size_t)k * gridDim.x + blockIdx.x] = part[k];
    unsigned ticket;
    asm volatile("atom.acq_rel.gpu.global.add.u32 %0, [%1], 1;"
                 : "=r"(ticket)
                 : "l"(__cvta_generic_to_global(counter))
                 : "memory");
    am_last = (ticket == gridDim.x - 1);
  }
  __syncthreads();
  if (!am_last) return false;
  // each thread folds a strided subset in order, then the block's reduction
  for (int k = 0; k < NV; ++k) out[k] = 0.0;  // partial maxima are of non-negative quantities
  for (int b = threadIdx.x; b < (int)gridDim.x; b += blockDim.x)
    for (int k = 0; k < NV; ++k) {
      const double v = ((volatile double *)partials)[(size_t)k * gridDim.x + b];
      out[k] = is_max[k] ? fmax(out[k], v) : out[k] + v;
    }
  block_reduce<NV>(out, is_max);
  if (threadIdx.x == 0) *counter = 0u;
  return true;
}

__host__ __device__ inline int64_t ceil_div(int64_t a, int64_t b) { return (a + b - 1) / b; }

// Off-diagonal part of one CSR row times a gathered vector, computed by the W
// lanes of a row group (this lane's partial sum; reduce over the group after).
// Each pass first issues U independent column/value loads per lane and then U
// independent gathers, so a row of up to W*U entries costs one dependent
// memory round trip instead of one per W entries.  Out-of-range slots load
// nothing and add nothing.
// Explicit fused multiply-add: the kernels that must agree bit for bit (the
// launched V-cycle and its cluster-resident tail) spell out every fusion
// instead of leaving the choice to the compiler's contraction.
__device__ __forceinline__ double fmadd(double a, double b, double c) { return fma(a, b, c); }
__device__ __forceinline__ float fmadd(float a, float b, float c) { return fmaf(a, b, c); }

// FP32 <-> FP64 conversions on the integer pipe, with the results of the
// conversion instructions (round to nearest even when narrowing).  On GB300 the
// instructions run on the FP64 pipe, which issues one warp instruction in ~16
// cycles per SM; the ~6-9 integer instructions take a third of that.  Zeros,
// subnormals, infinities, NaN and narrowed values outside FP32's normal range take
// the instruction.
__device__ __forceinline__ double widen(float v) {
  const uint32_t u = __float_as_uint(v), e = (u >> 23) & 0xffu;
  if (e - 1u < 254u)  // normal: rebias the exponent by 1023 - 127, shift the fraction
    return __hiloint2double((int)((u & 0x80000000u) | (((u & 0x7fffffffu) >> 3) + 0x38000000u)),
                            (int)(u << 29));
  return (double)v;
}
__device__ __forceinline__ double widen(double v) { return v; }
// narrow_ok: 2^-126 <= |v| < 2^127, where narrow_fast is exact.
__device__ __forceinline__ bool narrow_ok(double v) {
  return (((uint32_t)__double2hiint(v) >> 20) & 0x7ffu) - 897u < 253u;
}
__device__ __forceinline__ float narrow_fast(double v) {
  // round the fraction to 23 bits, ties to even (a carry into the exponent is the
  // right result), then rebias
  const unsigned long long x = (unsigned long long)__double_as_longlong(v);
  const unsigned long long r = x + 0x0fffffffull + ((x >> 29) & 1ull);
  return __uint_as_float(((uint32_t)(x >> 32) & 0x80000000u) | ((uint32_t)(r >> 29) - 0xc0000000u));
}
template <typename T>
__device__ __forceinline__ T narrow(double v);
template <>
__device__ __forceinline__ double narrow<double>(double v) { return v; }
template <>
__device__ __forceinline__ float narrow<float>(double v) {
  return narrow_ok(v) ? narrow_fast(v) : (float)v;
}

// Quotients with few FP64 operations (the division in FP64 costs about ten, and the
// FP64 pipe bounds the per-particle kernels): a reciprocal of the divisor and one
// residual correction q + (x - q d) y (Markstein 1990).  Before its last rounding the
// result is off by ~2^-88 of itself (~2^-104 with div_by's reciprocal): the rounded
// quotient, but for about one in 2^35, which rounds to its neighbour.
// An infinite or overflowing product, of which the residual would make a NaN, takes the
// division.
__device__ __forceinline__ double corrected_quotient(double x, double d, double y) {
  const double q = x * y;
  return fma(fma(-q, d, x), y, q);
}
// div_by: y = 1/d is known (a constant of the launch).
__device__ __forceinline__ double div_by(double x, double d, double y) {
  return ((uint32_t)__double2hiint(x * y) & 0x7ff00000u) != 0x7ff00000u ? corrected_quotient(x, d, y)
                                                                       : x / d;
}
// recip: an FP32 seed (~2^-22) and one Newton step y (2 - d y), to ~2^-44; the
// divisor's magnitude must be within 2^-100 .. 2^100 (recip_ok).
__device__ __forceinline__ bool recip_ok(double d) {
  return (((uint32_t)__double2hiint(d) >> 20) & 0x7ffu) - (1023u - 100u) < 200u;
}
__device__ __forceinline__ double recip(double d) {
  const double y = widen(__fdividef(1.0f, narrow_fast(d)));
  return fma(y, fma(-d, y, 1.0), y);
}
__device__ __forceinline__ double quotient(double x, double d) {
  // |x| < 2^900: no product with a reciprocal of up to 2^100 overflows
  const bool fast = recip_ok(d) && ((uint32_t)__double2hiint(x) & 0x7ff00000u) < (1923u << 20);
  return fast ? corrected_quotient(x, d, recip(d)) : x / d;
}
// One update e1 = e - u / J of the material Newton solves; true once |u / J| <= tol |e1|.
// FP64 operations bound them, so the quotient is a product with a reciprocal of ~2^-44:
// the next iteration removes its error, and the last one's stays below 2^-56 |e1| where
// |u / J| <= 2^-12 |e1|.  exact (uniform; a looser tol, or the last iteration allowed)
// adds the residual correction of the quotients above.  The test reads bit patterns.
__device__ __forceinline__ bool newton_update(double u, double J, double e, double tol, bool exact,
                                              double &e1) {
  double de;
  if (recip_ok(J)) {
    const double y = recip(J);
    de = u * y;
    if (exact) de = fma(fma(-de, J, u), y, de);
  } else {
    de = u / J;
  }
  e1 = e - de;
  const long long lim = __double_as_longlong(tol * fabs(e1));
  return __double_as_longlong(fabs(de)) <= lim && lim <= 0x7ff0000000000000ll;
}
// Larger of two non-negative values by their bit patterns (integer pipe); a NaN
// in v is passed over, as by fmax.
__device__ __forceinline__ double max_bits(double m, double v) {
  const long long a = __double_as_longlong(m), b = __double_as_longlong(v);
  return __longlong_as_double(b > a && b <= 0x7ff0000000000000ll ? b : a);
}
__device__ __forceinline__ double warp_max_bits(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v = max_bits(v, __shfl_down_sync(0xffffffffu, v, o));
  return v;
}

template <int W, int U, typename MT, typename VT>
__device__ __forceinline__ VT row_dot(int64_t beg, int64_t end, const int32_t *__restrict__ col,
                                      const MT *__restrict__ val, const VT *__restrict__ x,
                                      int sub) {
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
      if (c[u] >= 0) s = fmadd((VT)v[u], __ldg(x + c[u]), s);
  }
  return s;
}

// Row loops of W-lane row groups must be WARP-UNIFORM: row_reduce's full-mask
// shuffles need every lane of the warp, so all the groups of a warp make the
// same number of passes.  Loop over the warp's base row (the row of its first
// group) and give each group its offset; a group past the end of the range is
// inactive (an empty row) but still takes part in the shuffles.
//   for (int64_t wb = r0 + warp_first_group<W>(grp); wb < r1; wb += ngrp) {
//     const int64_t i = wb + group_in_warp<W>(grp);
//     const bool active = i < r1;  ...
template <int W>
__device__ __forceinline__ int64_t group_in_warp(int64_t grp) {
  return grp % (32 / W);
}
template <int W>
__device__ __forceinline__ int64_t warp_first_group(int64_t grp) {
  return grp - group_in_warp<W>(grp);
}

// Sum over the W lanes of a row group (W divides 32; groups are aligned).
template <int W, typename T>
__device__ __forceinline__ T row_reduce(T v) {
#pragma unroll
  for (int o = W / 2; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o, W);
  return v;
}

// ---------------------------------------------------------------------------
// Row tiles: the layout of the SpMV-class sweeps.
//
// On this part an FP64 warp instruction occupies the narrow FP64 pipe for all
// 32 lanes whether or not a lane is active, so lanes left idle by a sweep cost
// as much as busy ones.  A warp therefore works on tiles of 32 consecutive rows
// in W rounds; in round t its G = 32/W row groups (W lanes each) take rows
// t G + g.  Per round the warp issues exactly as many FMA instructions as its
// longest row needs (not a multiple of the load batch); after the W rounds a
// transposed shuffle reduction leaves the sum of row (l mod W) G + l/W in lane
// l with W - 1 adds per lane instead of log2(W) adds per lane and row; and the
// row epilogue (diagonal term, vector updates, reductions) runs on all 32
// lanes instead of one lane per group, with its loads and stores coalesced.
//
// The arithmetic of a row is that of row_dot + row_reduce exactly: each lane
// sums its entries beg + sub + j W in increasing j, and the reduction adds the
// lane partials in the same tree (lanes W/2 apart first), so every row sum is
// bitwise that of the one-row-per-group form.
// ---------------------------------------------------------------------------

// Offset, within its tile, of the row whose sum and epilogue lane `lane` holds.
template <int W>
__device__ __forceinline__ int tile_own_row(int lane) {
  return (lane % W) * (32 / W) + lane / W;
}

// Contiguous rows [r0, r1) of this warp: the rows are cut into units of G =
// 32/W (one round of a tile) and the units are spread as evenly as possible
// over all warps of the grid.  Warp-uniform.
template <int W>
__device__ __forceinline__ void warp_rows(int64_t n, int64_t &r0, int64_t &r1) {
  constexpr int G = 32 / W;
  const int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
  const int64_t w = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int64_t units = ceil_div(n, G), q = units / nwarps, rem = units % nwarps;
  const int64_t u0 = w * q + (w < rem ? w : rem);
  const int64_t u1 = u0 + q + (w < rem ? 1 : 0);
  r0 = u0 * G < n ? u0 * G : n;
  r1 = u1 * G < n ? u1 * G : n;
}

// Off-diagonal sum of one row by its W-lane group with a warp-uniform trip
// count: nmax = the largest per-lane entry count over the warp, so the warp
// issues nmax FMA instructions.  Full passes keep U column/value loads and U
// gathers in flight per lane; the last, partial pass loads its slots at once
// and then runs its FMAs in a loop of exactly (nmax mod U) trips, shifting the
// loaded slots down.  Slots past a lane's row end load nothing and contribute
// fma(0, 0, s) = s.
// x(c) is the gathered vector's entry c.
template <typename VT>
struct GatherVec {
  const VT *__restrict__ x;
  __device__ __forceinline__ VT operator()(int32_t c) const { return __ldg(x + c); }
};
template <int W, int U, typename MT, typename VT, typename X>
__device__ __forceinline__ VT row_dot_n(int64_t beg, int64_t end, const int32_t *__restrict__ col,
                                        const MT *__restrict__ val, const X &x, int sub,
                                        int nmax) {
  VT s = VT(0);
  int64_t k = beg + sub;
  int j = 0;
  for (; j + U <= nmax; j += U, k += (int64_t)W * U) {
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
      if (c[u] >= 0) s = fmadd((VT)v[u], x(c[u]), s);
  }
  const int rem = nmax - j;  // warp-uniform, < U
  if (rem > 0) {
    VT a[U], g[U];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int64_t kk = k + (int64_t)u * W;
      const int32_t c = kk < end ? __ldg(col + kk) : -1;
      a[u] = c >= 0 ? (VT)__ldg(val + kk) : VT(0);
      g[u] = c >= 0 ? x(c) : VT(0);
    }
#pragma unroll 1
    for (int u = 0; u < rem; ++u) {
      s = fmadd(a[0], g[0], s);
#pragma unroll
      for (int q = 0; q + 1 < U; ++q) {
        a[q] = a[q + 1];
        g[q] = g[q + 1];
      }
    }
  }
  return s;
}

// Partial of a tile round that holds three sums (the gradient's components,
// or the assembly's off-diagonal, ghost-weight and ghost right-hand-side sums);
// added and shuffled component by component.
struct Sum3 {
  double a, b, c;
};
__device__ __forceinline__ Sum3 operator+(const Sum3 &x, const Sum3 &y) {
  return {x.a + y.a, x.b + y.b, x.c + y.c};
}
template <int W>
__device__ __forceinline__ double tile_shfl(double v, int o) {
  return __shfl_xor_sync(0xffffffffu, v, o, W);
}
template <int W>
__device__ __forceinline__ float tile_shfl(float v, int o) {
  return __shfl_xor_sync(0xffffffffu, v, o, W);
}
template <int W>
__device__ __forceinline__ Sum3 tile_shfl(const Sum3 &v, int o) {
  return {tile_shfl<W>(v.a, o), tile_shfl<W>(v.b, o), tile_shfl<W>(v.c, o)};
}

// One step of the transposed reduction at lane distance o: `lo` and `hi` are
// this lane's partials of two rounds that differ in bit o (lo: bit clear).
// The lane with bit o of its group index clear keeps round `lo` and adds its
// partner's partial of it; the partner keeps `hi`.  Both sides add the same
// two numbers, the lower lane's first, as row_reduce does.
template <int W, typename R>
__device__ __forceinline__ R tile_combine(const R &lo, const R &hi, int o, int sub) {
  const bool up = (sub & o) != 0;
  const R keep = up ? hi : lo, send = up ? lo : hi;
  const R recv = tile_shfl<W>(send, o);
  return up ? recv + keep : keep + recv;
}

// The reduction tree over the W rounds of a tile, evaluated depth first: the
// rounds are visited in bit-reversed order and each pair is combined as soon
// as both are done, so at most log2(W) + 1 partials are live at a time.
// Rounds t0 + j O (j = 0, 1, ...) are the subtree below bit O.  round(t)
// returns this lane's partial of round t; it is called by every lane of the
// warp, and only for rounds that hold rows (t G < rows, warp-uniform).  The
// result: lane sub of a group holds round sub, i.e. row sub G + g of the tile.
template <int W, int O, typename R, typename F>
__device__ __forceinline__ R tile_tree(int t0, int rows, int sub, const F &round) {
  if constexpr (O == W) {
    return t0 * (32 / W) < rows ? round(t0) : R{};
  } else {
    const R lo = tile_tree<W, 2 * O, R>(t0, rows, sub, round);
    const R hi = tile_tree<W, 2 * O, R>(t0 + O, rows, sub, round);
    return tile_combine<W, R>(lo, hi, O, sub);
  }
}

// Warp-uniform trip count of round t: the largest number of entries a lane
// of the warp has in its row [rb, re) (entries rb + sub + j W).
template <int W>
__device__ __forceinline__ int tile_nmax(int64_t rb, int64_t re, int sub) {
  const int cnt = (int)((re - rb - sub + W - 1) / W);  // >= 0
  return __reduce_max_sync(0xffffffffu, cnt);
}

// Row sums of the tile of `rows` (<= 32) rows starting at `base`: lane l gets
// the off-diagonal sum of row base + tile_own_row<W>(l) (0 past `rows`).  Every
// lane of the warp must call it with the same base and rows.
template <int W, int U, typename MT, typename VT, typename X>
__device__ __forceinline__ VT tile_row_sums_of(int64_t base, int rows,
                                               const int64_t *__restrict__ ptr,
                                               const int32_t *__restrict__ col,
                                               const MT *__restrict__ val, const X &x) {
  const int lane = threadIdx.x & 31, sub = lane % W;
  const int own = tile_own_row<W>(lane);
  int64_t b = 0, e = 0;  // row extents, one coalesced load per lane
  if (own < rows) {
    b = __ldg(ptr + base + own);
    e = __ldg(ptr + base + own + 1);
  }
  return tile_tree<W, 1, VT>(0, rows, sub, [&](int t) -> VT {
    // round t's row of group g has its extents in lane g W + t
    const int64_t rb = __shfl_sync(0xffffffffu, b, t, W);
    const int64_t re = __shfl_sync(0xffffffffu, e, t, W);
    return row_dot_n<W, U, MT, VT>(rb, re, col, val, x, sub, tile_nmax<W>(rb, re, sub));
  });
}
template <int W, int U, typename MT, typename VT>
__device__ __forceinline__ VT tile_row_sums(int64_t base, int rows, const int64_t *__restrict__ ptr,
                                            const int32_t *__restrict__ col,
                                            const MT *__restrict__ val, const VT *__restrict__ x) {
  return tile_row_sums_of<W, U, MT, VT>(base, rows, ptr, col, val, GatherVec<VT>{x});
}

// Chebyshev iteration coefficients on [lo, hi] (Saad, Iterative Methods,
// Alg. 12.1): the first step scales by 1/theta, step k >= 1 uses
// d = c1[k] d + c2[k] D^{-1} res.  Computed once per interval (host, or one
// thread) rather than per thread: an FP64 division costs tens of FP64-pipe
// operations, and the FP64 pipe is narrow on this part.
constexpr int kChebMaxDeg = 48;
struct ChebCoef {
  int degree;        // number of steps (the requested degree, clamped to [1, kChebMaxDeg])
  double inv_theta;  // 1 / theta, theta = (hi + lo) / 2
  double c1[kChebMaxDeg], c2[kChebMaxDeg];
};
// A collapsed interval means D^{-1} A = I (no off-diagonal coupling): the
// first (Jacobi) step is then exact and the recurrence is undefined, so the
// later steps get c1 = c2 = 0 (d = 0, z unchanged).  The number of steps never
// depends on the data, so a captured launch sequence stays valid.
__host__ __device__ inline void cheb_coefficients(int degree, double lo, double hi,
                                                  ChebCoef *cf) {
  const double theta = 0.5 * (hi + lo), delta = 0.5 * (hi - lo);
  const bool collapsed = !(delta > 1e-12 * theta);
  if (degree > kChebMaxDeg) degree = kChebMaxDeg;
  if (degree < 1) degree = 1;
  cf->degree = degree;
  cf->inv_theta = 1.0 / theta;
  const double sigma1 = collapsed ? 1.0 : theta / delta;
  double rho0 = 1.0 / sigma1;
  cf->c1[0] = 0.0;
  cf->c2[0] = cf->inv_theta;
  for (int k = 1; k < degree; ++k) {
    if (collapsed) {
      cf->c1[k] = 0.0;
      cf->c2[k] = 0.0;
      continue;
    }
    const double rho1 = 1.0 / (2.0 * sigma1 - rho0);
    cf->c1[k] = rho1 * rho0;
    cf->c2[k] = 2.0 * rho1 / delta;
    rho0 = rho1;
  }
}

// Fusions at the two ends of an AMG preconditioner application on the finest
// level (launches saved per CG iteration).
// FineInit: the zero-guess smoother start of the finest level
// (cheb_init_zero_kernel's arithmetic) fused into the CG update, in the
// V-cycle's precision IT; r_lo receives the narrowed residual when the V-cycle
// runs in FP32 (else nullptr).  d == nullptr: no fusion.
template <typename IT>
struct FineInit {
  IT *r_lo;
  const IT *invdiag;
  const ChebCoef *cf;
  IT *d, *z;
};
// DotFuse: the preconditioned inner product rho = (r, z) and beta -- for the
// flexible variant (r, z) - (r, z_old) with z widened from the FP32 V-cycle
// into z64, whose old contents are z_old -- fused into the last V-cycle sweep.
struct DotFuse {
  int first;  // first CG inner product (no beta)
  int flex;   // flexible (mixed) variant
  const double *r;
  double *z64;
  Scalars *sc;
  double *partials;
};

// Krylov loop of the step's graph: the last kernel of an iteration (kind 1; of the
// prologue: kind 2) sets the WHILE node's condition instead of a kernel of its own.
// kind 0: none (host-driven loop).
struct LoopCond {
  cudaGraphConditionalHandle h;
  int kind, max_trips;
};
// By one thread of the grid, after sc->done is final for the iteration: go on while
// not converged, at most max_trips trips.
__device__ __forceinline__ void loop_cond_set(const LoopCond &c, Scalars *sc) {
  if (c.kind == 0) return;
  int t = 0;
  if (c.kind == 1) {
    sc->krylov_trips += 1;
    t = sc->krylov_solve_trips + 1;
  }
  sc->krylov_solve_trips = t;
  cudaGraphSetConditional(c.h, sc->done || t >= c.max_trips ? 0u : 1u);
}
// a kernel that returns at once because the solve is done still sets it
__device__ __forceinline__ void loop_cond_skip(const LoopCond &c, Scalars *sc) {
  if (blockIdx.x == 0 && threadIdx.x == 0) loop_cond_set(c, sc);
}

// What the material solve's last block does beside the reductions.
//   kOuterNone   nothing
//   kOuterInit   the initial solve of a step: resets the outer loop's state
//   kOuterTail   the solve of an outer iteration: the Krylov check, the statistics and
//                the outer convergence test (outer_check), and the loop condition
enum OuterMode { kOuterNone = 0, kOuterInit = 1, kOuterTail = 2 };
struct OuterTail {
  int mode, max_outer, in_graph;
  double tol_e, tol_E;
  cudaGraphConditionalHandle h;
};

// Vectors of the CG with the V-cycle's product (fine_post_smooth = 0), in the
// hierarchy's precision T: residual r, preconditioned residual z, w = B z,
// direction p and q = B p, the finest level's smoother start zpre, and the
// finest level's 1 / diagonal in T.  The iterate x and b stay FP64.
template <typename T>
struct FcgSet {
  T *r, *z, *w, *p, *q, *zpre;
  const T *invdiag;
};
struct FcgVecs {
  FcgSet<double> f64;
  FcgSet<float> f32;
  const ChebCoef *cf;  // the finest level's smoother coefficients (zpre = cf->inv_theta D^{-1} r)
};

// Chebyshev coefficient slots of a handle (device array): slot 0 belongs to
// the fine-level Chebyshev preconditioner, slot 1 + l to AMG level l (its
// smoother, or the coarse solve on the last level).
constexpr int kChebSlots = 1 + 32;

// Row-group shape of the SpMV-class kernels: W lanes per row, U loads in flight
// per lane.  A lane sums its entries (beg + sub + j W, j = 0, 1, ...) in
// increasing j whatever U is, so results depend on W only.  W follows from the
// mean row length (deterministic); U may be picked by the autotuner.
struct RowShape {
  int W, U;
};
// W = 4 lanes per row: loads stay sector-coalesced (4 x 8 B = one 32 B sector
// per row per instruction) while the FP64 reduction costs W - 1 = 3 adds per
// lane and tile (tile_row_sums) -- on GB300 the FP64 pipe, not HBM, limits a
// wide-warp CSR sweep.  Very long rows (coarse AMG levels) use 8 lanes.
__host__ inline int lanes_for_mean(double mean) { return mean <= 160 ? 4 : 8; }
// U = 4: with row tiles the sweeps are FP64-pipe-bound before they are
// latency-bound, and U = 4 keeps them at 48 registers (5 resident blocks per SM
// instead of 4 at U = 8); on the 64^3 and 128^3 operators it is 2-3 % faster.
__host__ inline RowShape shape_for_mean(double mean) {
  return {lanes_for_mean(mean), 4};
}
// Grid of a row-tile sweep (W lanes per row, kBlock threads per block): one
// wave of sweep_min_blocks(U) resident blocks per SM at most (the sweeps are
// compiled with that register cap); warp_rows splits the rows over its warps.
__host__ inline int row_grid_blocks(int num_sms, int64_t n, int W, int blocks_per_sm) {
  int64_t g = ceil_div(n > 0 ? n : 1, kBlock / W);
  int64_t cap = (int64_t)num_sms * blocks_per_sm;
  return (int)(g < cap ? g : cap);
}
__host__ inline int row_grid(int num_sms, int64_t n, int W, int U) {
  return row_grid_blocks(num_sms, n, W, sweep_min_blocks(U));
}

// Launch CALL with constexpr W and U set to the supported row-group shape:
// W in {4, 8}; U in {4, 8}.
#define SPH_DISPATCH_SHAPE(W_, U_, CALL)            \
  do {                                              \
    if ((W_) <= 4) {                                \
      if ((U_) <= 4) {                              \
        constexpr int W = 4, U = 4;                 \
        CALL;                                       \
      } else {                                      \
        constexpr int W = 4, U = 8;                 \
        CALL;                                       \
      }                                             \
    } else {                                        \
      if ((U_) <= 4) {                              \
        constexpr int W = 8, U = 4;                 \
        CALL;                                       \
      } else {                                      \
        constexpr int W = 8, U = 8;                 \
        CALL;                                       \
      }                                             \
    }                                               \
  } while (0)

// A CSR operator as seen by the SpMV-shaped kernels: off-diagonal entries in
// (ptr, col, val) and the diagonal apart.  (W, U) = row-group shape.
template <typename T>
struct CsrView {
  int64_t n = 0;
  const int64_t *ptr = nullptr;
  const int32_t *col = nullptr;
  const T *val = nullptr;
  const T *diag = nullptr;
  const T *invdiag = nullptr;
  int64_t nnz = 0;
  int W = 32;
  int U = 4;
};

// ---------------------------------------------------------------------------
// Sliced operators: the layout of the finest level's sweeps on large particle
// sets (sliced.cu builds it from the CSR rows; sliced_wanted says when).
//
// Rows are cut into groups of kBlock (one thread block's), sorted by length
// within the group (order: the row of each place) and cut into slices of 32
// (one warp's).  Entry t of the row of lane l of slice s stands at ptr[s] + 32 t
// + l, so a warp's loads are whole lines and a thread sums one row in list order,
// with no reduction across lanes; the sorting (by eighths of the length, so that
// most neighbouring rows stay together) keeps a warp's rows of nearly one length
// (unsorted, the longest of 32 rows is 13 % over the mean at 64^3, and an FP64
// instruction costs all 32 lanes).  Columns are 16-bit places in the group's
// dictionary, the sorted list of its distinct columns (neighbours of Morton-
// consecutive particles are few: ~7 per row for a group of 256 rows of ~104
// entries): a group stages x at its dictionary's columns in shared memory, one
// coalesced pass, and gathers from there.
//
// What it buys over the CSR row tiles: 2 instead of 4 bytes of column per entry
// (6 instead of 8 bytes in FP32, 10 instead of 12 in FP64), one line per warp
// load instead of 8 sectors, and gathers that do not go through the L1 tags,
// which bound the FP32 sweeps.  V-cycle residual at 128^3 in FP32, in the
// jobs: 0.410 -> 0.264 ms (5.16 TB/s of its 6 bytes an entry and 24 a row, 0.76 of the
// copy bandwidth); FP64 sweeps stay FP64-bound (one multiply-add per entry):
// 0.21 -> 0.18 ms at 97 x 96 x 91.
// ---------------------------------------------------------------------------
template <typename T>
struct SlicedView {
  int64_t n = 0;
  const int64_t *ptr = nullptr;    // [slices + 1] first entry of each slice (multiples of 32)
  const uint16_t *idx = nullptr;   // place in the group's dictionary
  const T *val = nullptr;
  const int32_t *len = nullptr;    // [n] entries of the row of each place
  const uint8_t *order = nullptr;  // [n] row within the group of each place
  const int64_t *dptr = nullptr;   // [groups + 1]
  const int32_t *dict = nullptr;   // columns, ascending within a group
  const T *diag = nullptr;
  const T *invdiag = nullptr;
  int64_t nnz = 0;     // entries without the padding
  int dict_max = 0;    // largest dictionary
};

// Row sources of the finest level's sweeps: each(x, pre, f) calls f(i, s, o) for
// every row i with s its off-diagonal sum over x and o = pre(i) its operands;
// every thread of the block takes part.  Sliced rows load the operands before the
// sums, so that their latency passes behind the staging of x; the row tiles after
// them (fewer registers, more warps).
template <int W_, int U_, typename MT>
struct CsrRows {
  static constexpr int W = W_, U = U_, kMinBlocks = sweep_min_blocks(U_);
  CsrView<MT> A;
  template <typename VT, typename P, typename F>
  __device__ __forceinline__ void each(const VT *x, const P &pre, const F &f) const {
    const int own = tile_own_row<W>(threadIdx.x & 31);
    int64_t r0, r1;
    warp_rows<W>(A.n, r0, r1);
    for (int64_t base = r0; base < r1; base += 32) {
      const int rows = (int)(r1 - base < 32 ? r1 - base : 32);
      const VT s = tile_row_sums<W, U, MT, VT>(base, rows, A.ptr, A.col, A.val, x);
      if (own < rows) f(base + own, s, pre(base + own));
    }
  }
};

constexpr int kSliceU = 8;  // entries in flight per thread
// operands of a row
template <typename T>
struct Ops1 { T a; };
template <typename T>
struct Ops2 { T a, b; };
template <typename T>
struct Ops3 { T a, b, c; };
template <typename T>
struct Ops4 { T a, b, c, d; };
template <typename T>
struct Ops7 { T a, b, c, d, e, f, g; };
template <typename MT>
struct SlicedRows {
  // FP32 sweeps are bound by HBM and load latency (more warps), FP64 ones by the
  // FP64 pipe (registers for the operands)
  static constexpr int kMinBlocks = sizeof(MT) == sizeof(float) ? 5 : 4;
  SlicedView<MT> A;
  // dictionary places and values of one batch, then their products in order
  template <typename VT>
  __device__ __forceinline__ VT row_sum(int64_t slice, int len, const VT *xs) const {
    const int64_t k0 = A.ptr[slice] + (threadIdx.x & 31);
    const int width = __reduce_max_sync(0xffffffffu, len);
    VT s = VT(0);
    int c[kSliceU];
    MT v[kSliceU];
    auto load = [&](int t) {
#pragma unroll
      for (int u = 0; u < kSliceU; ++u) {
        const int64_t k = k0 + (int64_t)(t + u) * 32;
        const bool in = t + u < len;
        c[u] = in ? (int)__ldg(A.idx + k) : 0;
        v[u] = in ? __ldg(A.val + k) : MT(0);
      }
    };
    int t = 0;
    for (; t + kSliceU <= width; t += kSliceU) {
      load(t);
#pragma unroll
      for (int u = 0; u < kSliceU; ++u) s = fmadd((VT)v[u], xs[c[u]], s);
    }
    if (t < width) {  // as many products as the longest row has left
      load(t);
#pragma unroll
      for (int u = 0; u < kSliceU - 1; ++u)
        if (t + u < width) s = fmadd((VT)v[u], xs[c[u]], s);
    }
    return s;
  }
  template <typename VT, typename P, typename F>
  __device__ __forceinline__ void each(const VT *x, const P &pre, const F &f) const {
    extern __shared__ __align__(16) unsigned char slice_smem[];
    VT *xs = reinterpret_cast<VT *>(slice_smem);
    __shared__ VT sums[kBlock];  // the rows' sums in row order, for the epilogue
    const int64_t groups = (A.n + kBlock - 1) / kBlock;
    for (int64_t g = blockIdx.x; g < groups; g += gridDim.x) {
      const int64_t d0 = A.dptr[g];
      const int nd = (int)(A.dptr[g + 1] - d0);
      const int64_t i = g * kBlock + threadIdx.x;
      const auto ops = pre(i < A.n ? i : A.n - 1);
      for (int t = threadIdx.x; t < nd; t += kBlock) xs[t] = __ldg(x + __ldg(A.dict + d0 + t));
      __syncthreads();
      const int64_t slice = i >> 5;
      if (slice * 32 < A.n) {  // warp-uniform
        const VT s = row_sum<VT>(slice, i < A.n ? A.len[i] : 0, xs);
        if (i < A.n) sums[A.order[i]] = s;
      }
      __syncthreads();  // also: xs may be staged again
      if (i < A.n) f(i, sums[threadIdx.x], ops);
    }
  }
};

}  // namespace sphrt

// --------------------------------------------------------------------------
// Internal handle.
// --------------------------------------------------------------------------
struct SphLevel;  // AMG level (amg.cu)

// Buffers of a sliced operator's structure (see SlicedView).
struct SlicedRowsData {
  int64_t *ptr = nullptr, *dptr = nullptr;
  uint16_t *idx = nullptr;
  int32_t *len = nullptr, *dict = nullptr;
  uint8_t *order = nullptr, *place = nullptr;  // row of each place, place of each row
  int64_t padded = 0;  // entries with the padding
  int dict_max = 0;
};

struct sph_rt {
  sph_rt_config cfg;
  std::string err;
  int64_t launches = 0;
  cudaStream_t stream = nullptr;
  bool own_stream = false;
  bool cuda_ready = false;
  int num_sms = 152;
  std::vector<void *> allocs;  // device allocations of the current particle set
  std::unordered_map<void *, size_t> alloc_size;
  std::multimap<size_t, void *> pool;  // released buffers kept for reuse
  // sph_rt_test_hook: allocations until one fails (-1: none), A P's slices refused
  int64_t test_fail_after = -1;
  bool test_refuse_ap = false;

  // sizes
  bool have_particles = false;
  bool have_operator = false;
  int64_t n = 0, n_int = 0;
  int64_t nnz_nbr = 0, nnz_mat = 0, nnz_gh = 0;
  int dim = 3;

  // permutation
  int64_t *slot2caller = nullptr;  // [n]
  int64_t *caller2slot = nullptr;  // [n]

  // particle data, slot order
  double *px = nullptr, *py = nullptr, *pz = nullptr;
  double *mass = nullptr, *rho = nullptr, *h = nullptr, *sigma0 = nullptr;
  double *V = nullptr, *invV = nullptr;
  int32_t *kind = nullptr;      // [n]
  int32_t *copysrc = nullptr;   // [n] slot of the copied interior particle, else -1
  double *e = nullptr, *E = nullptr;  // state [n] (ghost entries hold ghost values)

  // neighbour lists (interior rows)
  int64_t *nbr_ptr = nullptr;  // [n_int + 1]
  int32_t *nbr_col = nullptr;  // slot of the neighbour
  double *nbr_F = nullptr;     // F_ij = W'(r)/r, two-h average
  int32_t *gcol = nullptr;     // slot whose E neighbour k carries (copy ghosts: the copied one)
  double *gvx = nullptr, *gvy = nullptr, *gvz = nullptr;  // V_j F_ij x_ij (limiter only)

  // operator B = V A (interior rows; unknown index == slot)
  int64_t *mat_ptr = nullptr;
  int32_t *mat_col = nullptr;
  double *mat_G = nullptr;     // V_i V_j F_ij
  double *mat_val = nullptr;   // B_ij of the current step
  float *mat_val32 = nullptr;  // FP32 copy for the mixed form (written by the assembly)
  float *diag32 = nullptr, *invdiag32 = nullptr;
  double *diag = nullptr, *invdiag = nullptr;
  // the same operator in slices (sl.ptr == nullptr: not built, the CSR values above
  // are in use; otherwise mat_G, mat_val and mat_val32 are not)
  SlicedRowsData sl;
  double *sl_G = nullptr, *sl_val = nullptr;
  float *sl_val32 = nullptr;
  bool sl_decided = false;  // the layout of this particle set is chosen (sliced_operator)
  int64_t *gh_ptr = nullptr;   // Dirichlet-ghost couplings
  int32_t *gh_slot = nullptr;
  double *gh_W = nullptr;      // V_j F_ij
  int32_t *gh_row = nullptr;   // row of each coupling
  double *gb = nullptr;        // unscaled Dirichlet coupling sum_j w_ij E_j

  // material data of the step, slot order [n]
  double *T = nullptr, *sigma = nullptr, *f = nullptr, *R = nullptr, *lambda = nullptr,
         *D = nullptr;

  // step vectors (interior)
  double *e_old = nullptr, *E_old = nullptr, *e_l = nullptr, *E_l = nullptr;
  double *Qe = nullptr, *QE = nullptr;  // slot order [n]
  double *b = nullptr, *x = nullptr, *r = nullptr, *z = nullptr, *p = nullptr, *q = nullptr,
         *w = nullptr;
  double *z_old = nullptr;  // previous preconditioned residual (flexible CG)
  double *tmp_n = nullptr;   // [n] staging for caller-order transfers
  double *tmp_n2 = nullptr;  // [n] staging / Chebyshev scratch
  double *tmp_n3 = nullptr;
  double *e_bak = nullptr, *E_bak = nullptr;  // [n] state at the start of the step
  double *stage_ge = nullptr, *stage_gE = nullptr;  // [n] ghost values staged from the host

  // reductions
  sphrt::Scalars *sc = nullptr;  // device
  sphrt::Scalars *sc_host = nullptr;  // pinned mirror
  double *partials = nullptr;    // [8 * kMaxRedBlocks]

  // AMG hierarchy and Chebyshev data
  std::vector<SphLevel *> levels;
  bool amg_ready = false;
  int coarse_smem_optin = 0;                 // shared-memory opt-in done (bit per value type)
  int tail_level = 0;    // first AMG level of the cluster-resident V-cycle tail (0 = none)
  int tail_cluster = 0;  // thread blocks in the tail's cluster
  double *gersh = nullptr;                   // device scalar written by the assembly
  double *amg_gersh = nullptr;               // per-level Gershgorin bounds
  sphrt::ChebCoef *cheb_slots = nullptr;     // device [kChebSlots] (see kChebSlots)

  // device-driven outer loop: one CUDA graph with conditional WHILE nodes
  cudaGraph_t graph = nullptr;
  cudaGraphExec_t graph_exec = nullptr;
  std::vector<uint64_t> graph_sig;  // launch parameters the graph was captured with
  cudaStream_t cap_stream = nullptr;
  sphrt::LoopCond loop_cond{0, 0, 0};  // of the part being captured
  int64_t graph_l_init = 0, graph_l_outer = 0, graph_l_inner = 0;  // kernels per part
  int64_t graph_builds = 0, graph_launches = 0;

  // row-group shape of the fine SpMV-class kernels (autotuned or from the mean row length)
  sphrt::RowShape fine_shape{16, 6};
  // extrapolated Krylov start (config.krylov_start = p > 0).  Between steps E_old
  // holds E^{n-2} (the last step's start) and E_hist[j] E^{n-3-j}; during a step
  // E_hist[j] holds E^{n-2-j}.  hist counts the consecutive converged steps of
  // this particle set (capped at 3), dt_hist[j] the sizes of the last ones.
  double *E_hist[3] = {nullptr, nullptr, nullptr};
  int hist = 0;
  double dt_hist[3] = {0.0, 0.0, 0.0};
  bool fine_shape_set = false;
  int64_t fine_shape_n = 0, fine_shape_nnz = 0;  // sizes the shape was tuned on
  // solver autotuner (config.autotune): done once per handle; its trials
  bool solver_tuned = false;
  std::vector<sph_rt_tune_trial> tune_trials;

  // kernel timing
  std::vector<cudaEvent_t> ev_pool;
  std::vector<double> ev_bytes;   // bytes of each event pair
  std::vector<int> ev_kind;       // kernel kind of each event pair (sphrt::TimedKind)
  int *ev_flags = nullptr;        // device: work flag of each event pair
  // timing gate: with kernel_timing the stream is held by gate_kernel until a
  // whole chunk of the solve is queued, so that the timed kernels run back to
  // back and an event pair measures the kernel, not the host's launch latency
  volatile int *gate_host = nullptr;  // mapped pinned word written by the host
  int *gate_dev = nullptr;            // its device address
  int gate_epoch = 0;
  int ev_used = 0;
  int64_t spmv_launches = 0;
  double spmv_ms = 0.0, spmv_bytes = 0.0;
  int64_t kind_launches[5] = {0, 0, 0, 0, 0};  // per sphrt::TimedKind
  double kind_ms[5] = {0, 0, 0, 0, 0}, kind_bytes[5] = {0, 0, 0, 0, 0};
};

// Helpers shared by the translation units (defined in sph_rt.cu).
namespace sphrt {
sph_rt_status set_error(sph_rt *s, sph_rt_status st, const std::string &msg);
bool cuda_ok(sph_rt *s, cudaError_t e, const char *what);
void *dalloc_bytes(sph_rt *s, size_t bytes);  // tracked cudaMalloc; nullptr on failure
template <typename T>
inline T *dalloc(sph_rt *s, size_t count) {
  return static_cast<T *>(dalloc_bytes(s, sizeof(T) * (count > 0 ? count : 1)));
}
void free_all(sph_rt *s);
void dfree(sph_rt *s, void *p);  // back to the free list (stream-ordered users must sync first)
// CUDA-event bracketing of fine-operator SpMV-class launches (config.kernel_timing).
// timing_begin returns the work flag of the launch (nullptr when timing is off):
// the kernel writes 1 there if it does work and 0 if it returns at once because
// the solve has converged; only launches that worked are counted.
// kinds of timed fine-operator launches (SPH_RT_KERNEL_* in sph_rt.h)
enum TimedKind { kTimedSpmvPQ = 0, kTimedResid = 1, kTimedCheb = 2, kTimedPost = 3,
                 kTimedTrueResid = 4 };
constexpr int kTimedKinds = 5;
int *timing_begin(sph_rt *s);
void timing_end(sph_rt *s, double bytes, int kind);
void timing_flush(sph_rt *s);
__device__ __forceinline__ void mark_work(int *wflag, int worked) {
  if (wflag && blockIdx.x == 0 && threadIdx.x == 0) *wflag = worked;
}
}  // namespace sphrt

// Host-side phase trace to stderr, enabled by the environment variable
// SPH_RT_TRACE=1 (diagnostics only; off by default).
namespace sphrt {
bool trace_enabled();
}
#define SPH_TRACE(...)                                \
  do {                                                \
    if (sphrt::trace_enabled()) {                     \
      fprintf(stderr, "[sphrt] " __VA_ARGS__);        \
      fputc('\n', stderr);                            \
      fflush(stderr);                                 \
    }                                                 \
  } while (0)

#define SPH_CUDA(s, call)                                          \
  do {                                                             \
    cudaError_t e_ = (call);                                       \
    if (e_ != cudaSuccess) {                                       \
      sphrt::cuda_ok((s), e_, #call);                              \
      return SPH_RT_EDEVICE;                                       \
    }                                                              \
  } while (0)

#define SPH_LAUNCHED(s)                                            \
  do {                                                             \
    (s)->launches++;                                               \
    cudaError_t e_ = cudaGetLastError();                           \
    if (e_ != cudaSuccess) {                                       \
      sphrt::cuda_ok((s), e_, "kernel launch");                    \
      return SPH_RT_EDEVICE;                                       \
    }                                                              \
  } while (0)

namespace sphrt {

// Programmatic dependent launch.  A kernel launched with pdl_launch may be
// launched while the previous kernel on the stream drains (its last blocks
// finishing, its writes being flushed); every such kernel calls pdl_wait() as
// its first statement, which returns once the previous kernel has completed
// and its writes are visible (at once for a kernel launched the ordinary way).
// Since every kernel of the chain waits before it does anything, each one still
// completes after all earlier ones.  (Allowing the next launch early, right
// after the wait, measured no faster and is not done.)
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

// Launch `kernel` on the handle's stream, with programmatic dependent launch
// when the configuration asks for it.  The caller checks with SPH_LAUNCHED.
template <typename... KP, typename... A>
inline void pdl_launch(const sph_rt *s, void (*kernel)(KP...), dim3 grid, dim3 block, size_t smem,
                       A... args) {
  cudaLaunchConfig_t lc;
  memset(&lc, 0, sizeof lc);
  lc.gridDim = grid;
  lc.blockDim = block;
  lc.dynamicSmemBytes = smem;
  lc.stream = s->stream;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  lc.attrs = attr;
  lc.numAttrs = s->cfg.pdl ? 1 : 0;
  cudaLaunchKernelEx(&lc, kernel, args...);
}

}  // namespace sphrt
