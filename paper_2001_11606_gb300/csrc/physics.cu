// physics.cu -- per-particle and per-row kernels of one time step
// (rows a3, a4, a7, a8, a9 of the hot path).
//
//  a3  material data, frozen for the step (Sec. 3.2):
//        T = e/c_v, sigma = sigma0 T^p, Fleck factor f = 1/(1 + c sigma dt 4aT^3/(rho c_v))
//        (Sec. 2.2), SPH gradient grad E_i = sum_j V_j (E_j - E_i) F_ij x_ij (Sec. 2.3),
//        R = |grad E|/(sigma_t E), flux limiter lambda(R) (Sec. 2.1), D = c lambda / sigma_t,
//        sigma_t = sigma_a + sigma_s (constant scattering opacity sigma_s).
//  a4  operator of Eq. diffusion-solve scaled by V:  B_ij = V_i V_j F_ij (D_i + D_j) for
//        j != i, B_ii = V_i (1/dt + c sigma_i f_i) + sum over all neighbours of
//        V_i w_ij, w_ij = -V_j (D_i + D_j) F_ij >= 0; Dirichlet neighbours move to
//        the right-hand side as gb_i = sum_j w_ij E_j.
//  a7  right-hand side (Sec. 3.2, operators S and N):
//        b_i = E_i^{n-1}/dt + c sigma_i a T_i^4 - (1 - f_i) c sigma_i E_i + Q_E,i + gb_i.
//  a8  material solve M^{-1} (Eq. material-energy-update), one thread per particle.
//  a9  outer convergence (Eq. mat-rad-convergence) and energy totals (Sec. 2.5).
#include <cuda_runtime.h>

#include "common.cuh"
#include "sliced.cuh"

namespace sphrt {

struct Phys {
  double a, c, cv, p, T_floor, larsen_k, dt;
  double sigma_s;  // scattering opacity: sigma_t = sigma_a + sigma_s (R and D, Sec. 2.1)
  double inv_cv, inv_dt;  // 1/cv, 1/dt (the Newton loop multiplies instead of dividing)
  double tol_inner;
  int limiter, max_inner;
};

__device__ __forceinline__ double opacity(double sigma0, double Ts, double p) {
  if (p == 0.0) return sigma0;
  if (p == -3.0) return quotient(sigma0, Ts * Ts * Ts);
  return sigma0 * pow(Ts, p);
}

__device__ __forceinline__ double limiter_lambda(int limiter, double k, double R) {
  if (limiter == SPH_RT_LIMITER_LEVERMORE) return quotient(2.0 + R, 6.0 + 3.0 * R + R * R);
  if (limiter == SPH_RT_LIMITER_LARSEN) {
    if (k == 2.0) return quotient(1.0, sqrt(9.0 + R * R));
    return 1.0 / pow(pow(3.0, k) + pow(R, k), 1.0 / k);
  }
  return 1.0 / 3.0;
}

// a3, point part: every non-copy slot (interior and Dirichlet ghosts).
__global__ void props_point_kernel(Phys ph, int64_t n, const int32_t *kind, const double *rho,
                                   const double *sigma0, const double *e, double *T,
                                   double *sigma, double *f, double *R, double *lambda,
                                   double *D) {
  // R = 0 here; interior rows with a limiter are overwritten by the gradient kernel
  const double lam = limiter_lambda(ph.limiter, ph.larsen_k, 0.0);
  const double cl = ph.c * lam, c4 = ph.c * ph.dt * 4.0 * ph.a;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x) {
    if (kind[i] == SPH_RT_COPY) continue;
    const double Ti = div_by(e[i], ph.cv, ph.inv_cv);
    const double Ts = Ti > ph.T_floor ? Ti : ph.T_floor;
    const double sig = opacity(sigma0[i], Ts, ph.p);
    // 1 / (1 + c sigma dt 4 a T^3 / (rho c_v)) over one denominator
    const double rc = rho[i] * ph.cv;
    T[i] = Ti;
    sigma[i] = sig;
    f[i] = quotient(rc, rc + (c4 * sig) * (Ti * Ti * Ti));
    R[i] = 0.0;
    lambda[i] = lam;
    D[i] = quotient(cl, sig + ph.sigma_s);
  }
}

// a3, gradient part: one group of W lanes per interior row.
template <int W>
__global__ void props_grad_kernel(Phys ph, int64_t n_int, const int64_t *nbr_ptr,
                                  const int32_t *nbr_col, const double *nbr_F, const double *px,
                                  const double *py, const double *pz, const double *V,
                                  const int32_t *kind, const int32_t *copysrc, const double *E,
                                  const double *sigma, double *R, double *lambda, double *D) {
  const int sub = threadIdx.x % W;
  const int64_t grp = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) / W;
  const int64_t ngrp = ((int64_t)gridDim.x * blockDim.x) / W;
  for (int64_t wb = warp_first_group<W>(grp); wb < n_int; wb += ngrp) {
    const int64_t i = wb + group_in_warp<W>(grp);
    const bool active = i < n_int;
    const int64_t ia = active ? i : 0;
    double xi = px[ia], yi = py[ia], zi = pz[ia], Ei = E[ia];
    double gx = 0.0, gy = 0.0, gz = 0.0;
    const int64_t kbeg = active ? nbr_ptr[i] : 0, kend = active ? nbr_ptr[i + 1] : 0;
    for (int64_t k = kbeg + sub; k < kend; k += W) {
      int32_t j = nbr_col[k];
      int32_t js = kind[j] == SPH_RT_COPY ? copysrc[j] : j;
      double s = V[j] * (E[js] - Ei) * nbr_F[k];
      gx += s * (xi - px[j]);
      gy += s * (yi - py[j]);
      gz += s * (zi - pz[j]);
    }
    gx = group_sum<W>(gx);
    gy = group_sum<W>(gy);
    gz = group_sum<W>(gz);
    if (active && sub == 0) {
      double gn = sqrt(gx * gx + gy * gy + gz * gz);
      double Es = Ei > 1e-300 ? Ei : 1e-300;
      const double sig_t = sigma[i] + ph.sigma_s;
      double Ri = gn / (sig_t * Es);
      double lam = limiter_lambda(ph.limiter, ph.larsen_k, Ri);
      R[i] = Ri;
      lambda[i] = lam;
      D[i] = ph.c * lam / sig_t;
    }
  }
}

// Gradient sums of one row by its W-lane group (a row-tile round): entries
// beg + sub + j W, j < nmax (nmax warp-uniform; see row_dot_n), each adding
// (E_j - E_i) g_ij to the three components.  Slots past the row's end add
// fma(0, 0, g) = g.  D3: three dimensions (below, the z weights are zero and are
// neither stored nor read: 3 of 4 FP64 operations and 20 of 28 bytes a pair).
template <int W, int U, bool D3>
__device__ __forceinline__ Sum3 grad_row_n(int64_t beg, int64_t end, const int32_t *__restrict__ gcol,
                                           const double *__restrict__ gvx,
                                           const double *__restrict__ gvy,
                                           const double *__restrict__ gvz,
                                           const double *__restrict__ E, double Ei, int sub,
                                           int nmax) {
  double gx = 0.0, gy = 0.0, gz = 0.0;
  int64_t k = beg + sub;
  int j = 0;
  for (; j + U <= nmax; j += U, k += (int64_t)W * U) {
    int32_t c[U];
    double ax[U], ay[U], az[U];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int64_t kk = k + (int64_t)u * W;
      const bool ok = kk < end;
      c[u] = ok ? __ldg(gcol + kk) : -1;
      ax[u] = ok ? __ldg(gvx + kk) : 0.0;
      ay[u] = ok ? __ldg(gvy + kk) : 0.0;
      az[u] = D3 && ok ? __ldg(gvz + kk) : 0.0;
    }
#pragma unroll
    for (int u = 0; u < U; ++u) {
      if (c[u] < 0) continue;
      const double dE = __ldg(E + c[u]) - Ei;
      gx = fmadd(dE, ax[u], gx);
      gy = fmadd(dE, ay[u], gy);
      if (D3) gz = fmadd(dE, az[u], gz);
    }
  }
  const int rem = nmax - j;  // warp-uniform, < U
  if (rem > 0) {
    double dE[U], ax[U], ay[U], az[U];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int64_t kk = k + (int64_t)u * W;
      const bool ok = kk < end;
      const int32_t c = ok ? __ldg(gcol + kk) : -1;
      ax[u] = ok ? __ldg(gvx + kk) : 0.0;
      ay[u] = ok ? __ldg(gvy + kk) : 0.0;
      az[u] = D3 && ok ? __ldg(gvz + kk) : 0.0;
      dE[u] = c >= 0 ? __ldg(E + c) - Ei : 0.0;
    }
#pragma unroll 1
    for (int u = 0; u < rem; ++u) {
      gx = fmadd(dE[0], ax[0], gx);
      gy = fmadd(dE[0], ay[0], gy);
      if (D3) gz = fmadd(dE[0], az[0], gz);
#pragma unroll
      for (int q = 0; q + 1 < U; ++q) {
        dE[q] = dE[q + 1];
        ax[q] = ax[q + 1];
        ay[q] = ay[q + 1];
        az[q] = az[q + 1];
      }
    }
  }
  return {gx, gy, gz};
}

// a3, gradient part with precomputed pair geometry g_ij = V_j F_ij x_ij and
// the slot whose E a neighbour carries (its own, or the copied particle's):
// grad E_i = sum_j (E_j - E_i) g_ij.  Row tiles (common.cuh): 32 rows per warp,
// the row epilogue (|grad E|, R, the limiter, D) on all 32 lanes.
// Resident blocks per SM the row-tile gradient and assembly kernels are
// compiled for (80 registers: their rounds carry three sums and, at the end of
// a row, up to U slots of pair data).
constexpr int kPairMinBlocks = 3;

template <int W, int U, bool D3>
__global__ void __launch_bounds__(kBlock, kPairMinBlocks)
    props_grad_pre_kernel(Phys ph, int64_t n_int, const int64_t *nbr_ptr, const int32_t *gcol,
                          const double *gvx, const double *gvy, const double *gvz,
                          const double *E, const double *sigma, double *R, double *lambda,
                          double *D) {
  const int lane = threadIdx.x & 31, sub = lane % W, own = tile_own_row<W>(lane);
  int64_t r0, r1;
  warp_rows<W>(n_int, r0, r1);
  for (int64_t base = r0; base < r1; base += 32) {
    const int rows = (int)(r1 - base < 32 ? r1 - base : 32);
    const int64_t i = base + own;
    const bool active = own < rows;
    int64_t b = 0, e = 0;
    double Eo = 0.0;
    if (active) {
      b = nbr_ptr[i];
      e = nbr_ptr[i + 1];
      Eo = E[i];
    }
    const Sum3 g = tile_tree<W, 1, Sum3>(0, rows, sub, [&](int t) -> Sum3 {
      const int64_t rb = __shfl_sync(0xffffffffu, b, t, W);
      const int64_t re = __shfl_sync(0xffffffffu, e, t, W);
      const double Ei = __shfl_sync(0xffffffffu, Eo, t, W);
      return grad_row_n<W, U, D3>(rb, re, gcol, gvx, gvy, gvz, E, Ei, sub,
                              tile_nmax<W>(rb, re, sub));
    });
    if (active) {
      const double gx = g.a, gy = g.b, gz = g.c;
      double gn = sqrt(gx * gx + gy * gy + gz * gz);
      double Es = Eo > 1e-300 ? Eo : 1e-300;
      const double sig_t = sigma[i] + ph.sigma_s;
      double Ri = quotient(gn, sig_t * Es);
      double lam = limiter_lambda(ph.limiter, ph.larsen_k, Ri);
      R[i] = Ri;
      lambda[i] = lam;
      D[i] = quotient(ph.c * lam, sig_t);
    }
  }
}

// pair geometry for the gradient (once per particle set); gvz == nullptr below
// three dimensions.  A warp per row, so that the list reads and the writes are
// coalesced: a thread per row took 26.7 ms for 1.44e8 pairs (1.3e6 rows), this
// takes 2.8 ms.
__global__ void grad_geom_kernel(int64_t n_int, const int64_t *nbr_ptr, const int32_t *nbr_col,
                                 const double *nbr_F, const double *px, const double *py,
                                 const double *pz, const double *V, const int32_t *kind,
                                 const int32_t *copysrc, int32_t *gcol, double *gvx, double *gvy,
                                 double *gvz) {
  const int lane = threadIdx.x & 31;
  const int64_t warp = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
  for (int64_t i = warp; i < n_int; i += nwarps) {
    const double xi = px[i], yi = py[i], zi = pz[i];
    const int64_t e = nbr_ptr[i + 1];
    for (int64_t k = nbr_ptr[i] + lane; k < e; k += 32) {
      const int32_t j = nbr_col[k];
      gcol[k] = kind[j] == SPH_RT_COPY ? copysrc[j] : j;
      const double vf = V[j] * nbr_F[k];
      gvx[k] = vf * (xi - px[j]);
      gvy[k] = vf * (yi - py[j]);
      if (gvz) gvz[k] = vf * (zi - pz[j]);
    }
  }
}

// Ghosts, after the gradient: copy ghosts take every property of the particle they
// copy, Dirichlet ghosts their values at t^n (caller order; null: kept).
__global__ void ghost_kernel(int64_t n_int, int64_t n, const int32_t *kind,
                             const int32_t *copysrc, const int64_t *slot2caller,
                             const double *ge_c, const double *gE_c, double *T, double *sigma,
                             double *f, double *R, double *lambda, double *D, double *e,
                             double *E) {
  for (int64_t i = n_int + (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x) {
    const int32_t s = copysrc[i];
    if (s >= 0) {
      T[i] = T[s];
      sigma[i] = sigma[s];
      f[i] = f[s];
      R[i] = R[s];
      lambda[i] = lambda[s];
      D[i] = D[s];
    } else if (kind[i] == SPH_RT_DIRICHLET && (ge_c || gE_c)) {
      const int64_t c = slot2caller[i];
      if (ge_c) e[i] = ge_c[c];
      if (gE_c) E[i] = gE_c[c];
    }
  }
}

// Off-diagonal values of one row of B by its W-lane group (a row-tile round):
// B_ij = G_ij (D_i + D_j) written for entries beg + sub + j W, j < nmax
// (nmax warp-uniform), and this lane's sum of them.  Slots past the row's end
// store nothing and add +0.
// F32: also write the FP32 copy of the mixed form.
template <int W, int U, bool F32>
__device__ __forceinline__ double assemble_row_n(int64_t beg, int64_t end,
                                                 const int32_t *__restrict__ mat_col,
                                                 const double *__restrict__ mat_G,
                                                 const double *__restrict__ D, double Di,
                                                 double *__restrict__ mat_val,
                                                 float *__restrict__ mat_val32, int sub,
                                                 int nmax) {
  double offsum = 0.0;
  int64_t k = beg + sub;
  int j = 0;
  for (; j + U <= nmax; j += U, k += (int64_t)W * U) {
    int32_t c[U];
    double g[U];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int64_t kk = k + (int64_t)u * W;
      c[u] = kk < end ? __ldg(mat_col + kk) : -1;
      g[u] = kk < end ? __ldg(mat_G + kk) : 0.0;
    }
#pragma unroll
    for (int u = 0; u < U; ++u) {
      if (c[u] < 0) continue;
      const double v = g[u] * (Di + __ldg(D + c[u]));
      mat_val[k + (int64_t)u * W] = v;
      if (F32) mat_val32[k + (int64_t)u * W] = (float)v;
      offsum += v;
    }
  }
  const int rem = nmax - j;  // warp-uniform, < U
  if (rem > 0) {
    double g[U], dj[U];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int64_t kk = k + (int64_t)u * W;
      const int32_t c = kk < end ? __ldg(mat_col + kk) : -1;
      g[u] = c >= 0 ? __ldg(mat_G + kk) : 0.0;
      dj[u] = c >= 0 ? __ldg(D + c) : 0.0;
    }
#pragma unroll 1
    for (int u = 0; u < rem; ++u, k += W) {
      if (k < end) {
        const double v = g[0] * (Di + dj[0]);
        mat_val[k] = v;
        if (F32) mat_val32[k] = (float)v;
        offsum += v;
      }
#pragma unroll
      for (int q = 0; q + 1 < U; ++q) {
        g[q] = g[q + 1];
        dj[q] = dj[q + 1];
      }
    }
  }
  return offsum;
}

// a4: values of B for the step.  Row tiles (common.cuh): in each round a
// W-lane group writes one row's off-diagonal values and sums them, then adds
// up its Dirichlet-ghost couplings (few rows have any); the diagonal, its
// inverse, the ghost right-hand side and the Gershgorin ratio are computed on
// all 32 lanes.
template <int W, int U, bool F32>
__global__ void __launch_bounds__(kBlock, kPairMinBlocks)
    assemble_kernel(Phys ph, int64_t n_int, const int64_t *mat_ptr, const int32_t *mat_col,
                    const double *mat_G, double *mat_val, const int64_t *gh_ptr,
                    const int32_t *gh_slot, const double *gh_W, const double *V,
                    const double *sigma, const double *f, const double *D, const double *E,
                    double *diag, double *invdiag, double *gb, double *partials,
                    unsigned *counter, double *gersh_out, float *mat_val32, float *diag32,
                    float *invdiag32) {
  // gersh_out = max_i sum_{j != i} |B_ij| / B_ii: the eigenvalues of D^{-1} B
  // lie in [1 - gersh, 1 + gersh] (Gershgorin; B is symmetric, so real).
  const int lane = threadIdx.x & 31, sub = lane % W, own = tile_own_row<W>(lane);
  int64_t r0, r1;
  warp_rows<W>(n_int, r0, r1);
  double gmax = 0.0;
  for (int64_t base = r0; base < r1; base += 32) {
    const int rows = (int)(r1 - base < 32 ? r1 - base : 32);
    const int64_t i = base + own;
    const bool active = own < rows;
    int64_t b = 0, e = 0, hb = 0, he = 0;
    double Do = 0.0;
    if (active) {
      b = mat_ptr[i];
      e = mat_ptr[i + 1];
      hb = gh_ptr[i];
      he = gh_ptr[i + 1];
      Do = D[i];
    }
    const Sum3 acc = tile_tree<W, 1, Sum3>(0, rows, sub, [&](int t) -> Sum3 {
      const int64_t rb = __shfl_sync(0xffffffffu, b, t, W);
      const int64_t re = __shfl_sync(0xffffffffu, e, t, W);
      const int64_t gb0 = __shfl_sync(0xffffffffu, hb, t, W);
      const int64_t ge0 = __shfl_sync(0xffffffffu, he, t, W);
      const double Di = __shfl_sync(0xffffffffu, Do, t, W);
      const double offsum = assemble_row_n<W, U, F32>(rb, re, mat_col, mat_G, D, Di, mat_val,
                                                      mat_val32, sub, tile_nmax<W>(rb, re, sub));
      double wsum = 0.0, gbs = 0.0;
      const int ng = tile_nmax<W>(gb0, ge0, sub);
      for (int jj = 0; jj < ng; ++jj) {
        const int64_t k = gb0 + sub + (int64_t)jj * W;
        if (k < ge0) {
          const int32_t j = gh_slot[k];
          const double wk = -gh_W[k] * (Di + D[j]);
          wsum += wk;
          gbs += wk * E[j];
        }
      }
      return {offsum, wsum, gbs};
    });
    if (active) {
      const double offsum = acc.a, wsum = acc.b, gbs = acc.c;
      double d = V[i] * (1.0 / ph.dt + ph.c * sigma[i] * f[i] + wsum) - offsum;
      diag[i] = d;
      invdiag[i] = 1.0 / d;
      if (F32) {
        diag32[i] = (float)d;
        invdiag32[i] = (float)(1.0 / d);
      }
      gb[i] = gbs;
      gmax = fmax(gmax, -offsum / d);  // off-diagonals are <= 0
    }
  }
  double part[1] = {gmax}, out[1];
  const bool mx[1] = {true};
  block_reduce(part, mx);
  if (last_block_combine<1>(part, partials, counter, out, mx) && threadIdx.x == 0)
    *gersh_out = out[0];
}

// a4 on a sliced operator: a thread per row, D at the row group's dictionary in
// shared memory (see SlicedView).  Reads 10 bytes (place, G) and writes 8 (12 with
// the FP32 copy) per entry, but the FP64 pipe bounds it (three operations an entry,
// 80 % busy): the FP32 copy is narrowed with integer instructions, and the values
// of a batch are formed without a branch between them, so that their chains
// overlap.  2.18e8 entries: 2.10 -> 1.61 ms with the FP32 copy.
template <bool F32>
__global__ void __launch_bounds__(kBlock, 4)
    assemble_sliced_kernel(Phys ph, SlicedView<double> A, double *__restrict__ val,
                           float *__restrict__ val32, const int64_t *gh_ptr,
                           const int32_t *gh_slot, const double *gh_W, const double *V,
                           const double *sigma, const double *f, const double *D, const double *E,
                           double *diag, double *invdiag, double *gb, double *partials,
                           unsigned *counter, double *gersh_out, float *diag32,
                           float *invdiag32) {
  extern __shared__ __align__(16) unsigned char asm_smem[];
  double *Ds = reinterpret_cast<double *>(asm_smem);
  __shared__ double sums[3][kBlock];
  const int64_t groups = (A.n + kBlock - 1) / kBlock;
  double gmax = 0.0;
  for (int64_t g = blockIdx.x; g < groups; g += gridDim.x) {
    const int64_t d0 = A.dptr[g];
    const int nd = (int)(A.dptr[g + 1] - d0);
    for (int t = threadIdx.x; t < nd; t += kBlock) Ds[t] = D[A.dict[d0 + t]];
    __syncthreads();
    const int64_t i = g * kBlock + threadIdx.x;  // place in the slices, then row
    const unsigned lanes = __ballot_sync(0xffffffffu, i < A.n);  // of the last slice: its rows
    if (i < A.n) {
      const int len = A.len[i], row = A.order[i];
      const int64_t k0 = A.ptr[i >> 5] + (threadIdx.x & 31);
      const double Di = D[g * kBlock + row];
      double offsum = 0.0;
      const int width = __reduce_max_sync(lanes, len);  // rows of one warp
      for (int t = 0; t < width; t += kSliceU) {
        int c[kSliceU];
        double v[kSliceU];
        const int64_t k1 = k0 + (int64_t)t * 32;
#pragma unroll
        for (int u = 0; u < kSliceU; ++u) {
          const bool in = t + u < len;
          c[u] = in ? (int)__ldg(A.idx + k1 + u * 32) : 0;
          v[u] = in ? __ldg(A.val + k1 + u * 32) : 0.0;
        }
        // no branch among the values: their chains overlap (past a row's end G = 0)
#pragma unroll
        for (int u = 0; u < kSliceU; ++u) {
          v[u] *= Di + Ds[c[u]];
          offsum += v[u];
        }
        bool plain = true;
#pragma unroll
        for (int u = 0; u < kSliceU; ++u)
          if (t + u < len) {
            val[k1 + u * 32] = v[u];
            if (F32) {
              val32[k1 + u * 32] = narrow_fast(v[u]);
              plain = plain && narrow_ok(v[u]);
            }
          }
        if (F32 && !plain)  // rare: zeros and values outside FP32's normal range
          for (int u = 0; u < kSliceU && t + u < len; ++u)
            val32[k1 + u * 32] = (float)val[k1 + u * 32];
      }
      // Dirichlet couplings, in place order too: the rows that have any are the
      // short ones, which the sorting puts side by side
      double wsum = 0.0, gbs = 0.0;
      const int64_t h0 = gh_ptr[g * kBlock + row], h1 = gh_ptr[g * kBlock + row + 1];
      for (int64_t k = h0; k < h1; k += 8) {
        int32_t j[8];
        double w[8], Dj[8], Ej[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) j[u] = k + u < h1 ? gh_slot[k + u] : -1;
#pragma unroll
        for (int u = 0; u < 8; ++u) {
          w[u] = j[u] >= 0 ? gh_W[k + u] : 0.0;
          Dj[u] = j[u] >= 0 ? D[j[u]] : 0.0;
          Ej[u] = j[u] >= 0 ? E[j[u]] : 0.0;
        }
#pragma unroll
        for (int u = 0; u < 8; ++u)
          if (j[u] >= 0) {
            const double wk = -w[u] * (Di + Dj[u]);
            wsum += wk;
            gbs += wk * Ej[u];
          }
      }
      sums[0][row] = offsum;
      sums[1][row] = wsum;
      sums[2][row] = gbs;
    }
    __syncthreads();  // also: Ds may be staged again
    if (i >= A.n) continue;
    const double offsum = sums[0][threadIdx.x], wsum = sums[1][threadIdx.x];
    const double d = V[i] * (ph.inv_dt + ph.c * sigma[i] * f[i] + wsum) - offsum;
    const double inv = 1.0 / d;
    diag[i] = d;
    invdiag[i] = inv;
    if (F32) {
      diag32[i] = (float)d;
      invdiag32[i] = (float)inv;
    }
    gb[i] = sums[2][threadIdx.x];
    gmax = fmax(gmax, -offsum * inv);  // off-diagonals are <= 0
  }
  double part[1] = {gmax}, out[1];
  const bool mx[1] = {true};
  block_reduce(part, mx);
  if (last_block_combine<1>(part, partials, counter, out, mx) && threadIdx.x == 0)
    *gersh_out = out[0];
}

// a7: right-hand side of the diffusion solve (B-scaled), the warm start x = E^l,
// ||b||^2 of the unscaled rows, and reset of the Krylov scalars.
__global__ void rhs_kernel(Phys ph, int64_t n_int, const double *V, const double *sigma,
                           const double *f, const double *E_old, const double *e_l,
                           const double *E_l, const double *QE, const double *gb, double *b,
                           double *x, double tol, Scalars *sc, double *partials,
                           const double *H0, const double *H1, const double *H2) {
  // the first outer iteration's solve may start from the extrapolation in time
  // through E^l = E^{n-1} and H0, H1, H2 = E^{n-2}, E^{n-3}, E^{n-4}
  const int ord = sc->outer_iters == 0 ? sc->guess_order : 0;
  const double w0 = sc->guess_w[0], w1 = sc->guess_w[1], w2 = sc->guess_w[2],
               w3 = sc->guess_w[3];
  double acc = 0.0;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n_int;
       i += (int64_t)gridDim.x * blockDim.x) {
    double Tl = div_by(e_l[i], ph.cv, ph.inv_cv), T2 = Tl * Tl;
    double B = ph.a * (T2 * T2);
    double cs = ph.c * sigma[i];
    double bi = div_by(E_old[i], ph.dt, ph.inv_dt) + cs * B - (1.0 - f[i]) * cs * E_l[i] + QE[i] + gb[i];
    b[i] = V[i] * bi;
    double xi = E_l[i];
    if (ord >= 1) {
      xi = w0 * xi + w1 * H0[i];
      if (ord >= 2) xi += w2 * H1[i];
      if (ord >= 3) xi += w3 * H2[i];
    }
    x[i] = xi;
    acc += bi * bi;
  }
  double part[1] = {acc}, out[1];
  block_sums(part);
  const bool mx[1] = {false};
  if (last_block_combine<1>(part, partials, &sc->counter, out, mx) && threadIdx.x == 0) {
    sc->bnorm2 = out[0];
    sc->thresh2 = tol * tol * out[0];
    sc->done = 0;
    sc->iters = 0;
    sc->breakdown = 0;
  }
}

// outer-loop state at the start of a step; newton_max starts from the initial
// material solve of Alg. 1 (its iteration count is in red[2])
__device__ void outer_init(Scalars *sc) {
  sc->outer_iters = 0;
  sc->outer_status = 0;
  sc->outer_trips = 0;
  sc->krylov_total = 0;
  sc->krylov_trips = 0;
  sc->krylov_solve_trips = 0;
  sc->newton_max = (int)sc->red[2];
  sc->yvalid = 0;  // a new step has a new operator
  sc->last_change_e = 0.0;
  sc->last_change_E = 0.0;
  for (int k = 0; k < 64; ++k) sc->krylov_per_outer[k] = 0;
}

// After the material solve of an outer iteration: the Krylov check, the
// bookkeeping of the step statistics and the outer convergence test
// max_i |x^{l+1} - x^l| / |x^{l+1}| < tol for e and E (changes in red[0..1],
// Newton iterations in red[2]).  In the graph it also sets the loop condition.
// (As kernels of their own, this, the copy of the iterate and outer_init took 2-4 us
// each of a step that is 430 us at 1,024 particles.)
__device__ void outer_check(Scalars *sc, const OuterTail &t) {
  int status = 0;
  sc->outer_trips += 1;
  const bool kconv = !sc->breakdown && !(sc->rnorm2 > sc->thresh2);
  if (!kconv) {
    status = 2;
  } else {
    const int o = sc->outer_iters;
    if (o < 64) sc->krylov_per_outer[o] = sc->iters;
    sc->krylov_total += sc->iters;
    sc->outer_iters = o + 1;
    const double ce = sc->red[0], cE = sc->red[1];
    sc->newton_max = max(sc->newton_max, (int)sc->red[2]);
    sc->last_change_e = ce;
    sc->last_change_E = cE;
    if (ce < t.tol_e && cE < t.tol_E)
      status = 1;
    else if (sc->outer_iters >= t.max_outer)
      status = 3;
  }
  if (status == 0 && sc->outer_trips > t.max_outer) status = 3;
  sc->outer_status = status;
  if (t.in_graph) cudaGraphSetConditional(t.h, status == 0 ? 1u : 0u);
}

// a8 + a9: material solve with the new radiation energy and the outer
// convergence measures.  P_i = c sigma_i E_i + Q_e,i (Eq. material-energy-solve);
// Newton from e_start.  red[0] = max |e_new - e_start|/|e_new|,
// red[1] = max |E_new - E_prev|/|E_new|, red[2] = max Newton iterations,
// red[3] = number of particles that hit the iteration limit.
//
// FP64-bound: ~14 operations an iteration (newton_update in common.cuh), tests and
// maxima on bit patterns, and integer reductions.  2.1e6 particles: 0.335 -> 0.214 ms,
// 2.5e5 (heating wave): 0.068 -> 0.028.
__global__ void __launch_bounds__(kBlock)
    newton_kernel(Phys ph, int64_t n_int, const double *rho, const double *sigma,
                  const double *e_old, const double *Qe, const double *E_new, double *E_prev,
                  const double *e_start, double *e_new, Scalars *sc, double *partials,
                  const OuterTail tail) {
  double ce = 0.0, cE = 0.0;
  int itmax = 0, fails = 0;
  const double tiny = 1e-300;
  const bool loose = ph.tol_inner > 0x1p-12;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n_int;
       i += (int64_t)gridDim.x * blockDim.x) {
    const double cs = ph.c * sigma[i];
    const double En = E_new[i];
    const double P = fma(cs, En, Qe[i]);
    // per-particle constants of u(e) = rho/dt (e - e_old) + c sigma a T^4 - P and
    // J = rho/dt + 4 c sigma a T^3 / cv
    const double rdt = rho[i] * ph.inv_dt;
    const double csa = cs * ph.a;
    const double k4 = 4.0 * csa * ph.inv_cv;
    const double eo = e_old[i], e0 = e_start[i];
    double ei = e0;
    int it = 0;
    bool ok = false;
    while (it < ph.max_inner) {
      const double T = ei * ph.inv_cv;
      const double T3 = T * T * T;
      const double u = fma(rdt, ei - eo, fma(csa * T3, T, -P));
      const double J = fma(k4, T3, rdt);
      ++it;
      ok = newton_update(u, J, ei, ph.tol_inner, loose || it == ph.max_inner, ei);
      if (ok) break;
    }
    e_new[i] = ei;
    ce = max_bits(ce, quotient(fabs(ei - e0), max_bits(tiny, fabs(ei))));
    cE = max_bits(cE, quotient(fabs(En - E_prev[i]), max_bits(tiny, fabs(En))));
    if (tail.mode == kOuterTail) E_prev[i] = En;  // the new iterate becomes the current one
    itmax = max(itmax, it);
    fails += !ok;
  }
  __shared__ double sh[2][kWarpsPerBlock];
  __shared__ int shi[2][kWarpsPerBlock];
  ce = warp_max_bits(ce);
  cE = warp_max_bits(cE);
  itmax = __reduce_max_sync(0xffffffffu, itmax);
  fails = __reduce_add_sync(0xffffffffu, fails);
  const int wid = threadIdx.x >> 5;
  if ((threadIdx.x & 31) == 0) {
    sh[0][wid] = ce;
    sh[1][wid] = cE;
    shi[0][wid] = itmax;
    shi[1][wid] = fails;
  }
  __syncthreads();
  if (threadIdx.x == 0)
    for (int w = 1; w < kWarpsPerBlock; ++w) {
      ce = max_bits(ce, sh[0][w]);
      cE = max_bits(cE, sh[1][w]);
      itmax = max(itmax, shi[0][w]);
      fails += shi[1][w];
    }
  double part[4] = {ce, cE, (double)itmax, (double)fails}, out[4];
  const bool mx[4] = {true, true, true, false};
  if (last_block_combine<4>(part, partials, &sc->counter, out, mx) && threadIdx.x == 0) {
    sc->red[0] = out[0];
    sc->red[1] = out[1];
    sc->red[2] = out[2];
    sc->red[3] = out[3];
    if (tail.mode == kOuterInit) outer_init(sc);
    if (tail.mode == kOuterTail) outer_check(sc, tail);
  }
}

// Start of a step, in one pass over the slots: the snapshot of the state, the
// sources gathered to slot order (null: 0), the check that the step's inputs are
// finite (sources of interior particles, values of Dirichlet ghosts; caller order)
// and the energy before the step.  Latency at small sizes (5.2 us at 1,024 particles),
// HBM at large ones (10.4 us at 2.5e5), in place of nine launches and copies of 2-4 us
// each.
__global__ void step_begin_kernel(int64_t n_int, int64_t n, const int64_t *slot2caller,
                                  const int32_t *kind, const double *Qe_c, const double *QE_c,
                                  const double *ge, const double *gE, const double *mass,
                                  const double *V, const double *e, const double *E,
                                  double *e_bak, double *E_bak, double *Qe, double *QE,
                                  Scalars *sc, double *partials) {
  double a = 0.0, b = 0.0;
  int bad = 0;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x) {
    const double ei = e[i], Ei = E[i];
    e_bak[i] = ei;
    E_bak[i] = Ei;
    const int64_t c = slot2caller[i];
    if (i < n_int) {
      const double qe = Qe_c ? Qe_c[c] : 0.0, qE = QE_c ? QE_c[c] : 0.0;
      Qe[i] = qe;
      QE[i] = qE;
      if (!isfinite(qe) || !isfinite(qE)) bad = 1;
      a += mass[i] * ei;
      b += V[i] * Ei;
    } else if (kind[i] == SPH_RT_DIRICHLET) {
      if ((ge && !isfinite(ge[c])) || (gE && !isfinite(gE[c]))) bad = 1;
    }
  }
  double part[3] = {a, b, bad ? 1.0 : 0.0}, out[3];
  const bool mx[3] = {false, false, true};
  block_reduce(part, mx);
  if (last_block_combine<3>(part, partials, &sc->counter, out, mx) && threadIdx.x == 0) {
    sc->energy_before_e = out[0];
    sc->energy_before_E = out[1];
    sc->bad_input = out[2] != 0.0;
  }
}

// Before the initial material solve: the history of the extrapolated Krylov start
// moves down one place (H2 <- H1 <- H0 <- E_old, as far as `depth` reaches), and
// e_old, E_old and E^{n,0} take the state.
__global__ void step_start_kernel(int64_t n_int, int depth, const double *e, const double *E,
                                  double *e_old, double *E_old, double *E_l, double *H0,
                                  double *H1, double *H2, Scalars *sc, int order, double w0,
                                  double w1, double w2, double w3) {
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    sc->guess_order = order;
    sc->guess_w[0] = w0;
    sc->guess_w[1] = w1;
    sc->guess_w[2] = w2;
    sc->guess_w[3] = w3;
  }
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n_int;
       i += (int64_t)gridDim.x * blockDim.x) {
    if (depth >= 3) H2[i] = H1[i];
    if (depth >= 2) H1[i] = H0[i];
    if (depth >= 1) H0[i] = E_old[i];
    const double Ei = E[i];
    e_old[i] = e[i];
    E_old[i] = Ei;
    E_l[i] = Ei;
  }
}

// Totals over interior particles: red[4] = sum m e, red[5] = sum V E.
__global__ void totals_kernel(int64_t n_int, const double *mass, const double *V, const double *e,
                              const double *E, Scalars *sc, double *partials) {
  double a = 0.0, b = 0.0;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n_int;
       i += (int64_t)gridDim.x * blockDim.x) {
    a += mass[i] * e[i];
    b += V[i] * E[i];
  }
  double part[2] = {a, b}, out[2];
  block_sums(part);
  const bool mx[2] = {false, false};
  if (last_block_combine<2>(part, partials, &sc->counter, out, mx) && threadIdx.x == 0) {
    sc->red[4] = out[0];
    sc->red[5] = out[1];
  }
}

// End of a step, in one pass.  A converged step with valid inputs commits its
// interior state (copy ghosts take their particle's); any other step restores the
// snapshot taken at its start (ghost entries included), so a failed step leaves the
// state unchanged.  Of a committed step also the energies (meaningless otherwise):
//   red[4], red[5]  totals sum m e, sum V E
//   red[6]          added by the sources, dt sum V (Q_e + Q_E)
//   red[7]          added through the boundary, dt sum_i V_i sum_{Dirichlet j} w_ij
//                   (E_j - E_i), over the couplings as one flat list: few rows have
//                   any, those have tens, and a thread per row spent its time on the
//                   longest (0.22 ms at 128^3 with 5.7e6 couplings, 0.076 flat)
// One launch, 7.1 us at 1,024 particles and 12 us at 2.5e5, in place of four.
__global__ void step_end_kernel(Phys ph, int64_t n_int, int64_t n, int64_t nnz_gh,
                                const int32_t *copysrc, const double *e_new,
                                const double *E_new, const double *e_bak, const double *E_bak,
                                const double *mass, const double *V, const double *Qe,
                                const double *QE, const int32_t *gh_row, const int32_t *gh_slot,
                                const double *gh_W, const double *D, double *e, double *E,
                                Scalars *sc, double *partials) {
  const bool commit = sc->outer_status == 1 && !sc->bad_input;
  double te = 0.0, tE = 0.0, a = 0.0, b = 0.0;
  const int64_t t0 = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const int64_t step = (int64_t)gridDim.x * blockDim.x;
  for (int64_t i = t0; i < n; i += step) {
    if (i < n_int) {
      const double ei = commit ? e_new[i] : e_bak[i], Ei = commit ? E_new[i] : E_bak[i];
      e[i] = ei;
      E[i] = Ei;
      const double Vi = V[i];
      te += mass[i] * ei;
      tE += Vi * Ei;
      a += Vi * (Qe[i] + QE[i]);
    } else {
      const int32_t c = copysrc[i];
      if (c >= 0) {
        e[i] = commit ? e_new[c] : e_bak[c];
        E[i] = commit ? E_new[c] : E_bak[c];
      } else if (!commit) {
        e[i] = e_bak[i];
        E[i] = E_bak[i];
      }
    }
  }
  if (commit)
    for (int64_t k = t0; k < nnz_gh; k += step) {
      const int32_t i = gh_row[k], j = gh_slot[k];  // j: a ghost, not written above
      b -= (V[i] * gh_W[k]) * (D[i] + D[j]) * (E[j] - E_new[i]);
    }
  double part[4] = {te, tE, a, b}, out[4];
  block_sums(part);
  const bool mx[4] = {false, false, false, false};
  if (last_block_combine<4>(part, partials, &sc->counter, out, mx) && threadIdx.x == 0) {
    sc->red[4] = out[0];
    sc->red[5] = out[1];
    sc->red[6] = ph.dt * out[2];
    sc->red[7] = ph.dt * out[3];
  }
}

// caller-order source -> slot order (interior part); NULL source gives zeros
__global__ void gather_interior_kernel(const double *in_c, const int64_t *slot2caller,
                                       int64_t n_int, double *out) {
  for (int64_t s = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; s < n_int;
       s += (int64_t)gridDim.x * blockDim.x)
    out[s] = in_c ? in_c[slot2caller[s]] : 0.0;
}

__global__ void scatter_caller_kernel(const double *in_s, const int64_t *slot2caller, int64_t n,
                                      double *out_c) {
  for (int64_t s = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; s < n;
       s += (int64_t)gridDim.x * blockDim.x)
    out_c[slot2caller[s]] = in_s[s];
}

// ---------------------------------------------------------------------------
// Host launchers
// ---------------------------------------------------------------------------
static int grid_items(const sph_rt *s, int64_t n, int per_block) {
  int64_t g = ceil_div(n > 0 ? n : 1, per_block);
  int64_t cap = (int64_t)s->num_sms * 8;
  if (cap > kMaxRedBlocks) cap = kMaxRedBlocks;
  return (int)(g < cap ? g : cap);
}

// Streaming reductions: half the blocks of grid_items, so that a thread has two or
// more rows to sum before the FP64 shuffle reduction of its block.
static int grid_reduce(const sph_rt *s, int64_t n) {
  const int64_t g = ceil_div(n > 0 ? n : 1, kBlock), cap = (int64_t)s->num_sms * 4;
  return (int)(g < cap ? g : cap);
}

Phys make_phys(const sph_rt *s, double dt) {
  Phys ph;
  ph.a = s->cfg.a;
  ph.c = s->cfg.c;
  ph.cv = s->cfg.cv;
  ph.inv_cv = 1.0 / s->cfg.cv;
  ph.inv_dt = 1.0 / dt;
  ph.p = s->cfg.opacity_exp;
  ph.T_floor = s->cfg.T_floor;
  ph.larsen_k = s->cfg.larsen_k;
  ph.sigma_s = s->cfg.sigma_s;
  ph.dt = dt;
  ph.tol_inner = s->cfg.tol_inner_e;
  ph.limiter = s->cfg.limiter;
  ph.max_inner = s->cfg.max_inner_e;
  return ph;
}

// rows per group of the warp-per-row kernels, from the mean row length
int row_width(int64_t nnz, int64_t rows) {
  double mean = rows > 0 ? (double)nnz / (double)rows : 0.0;
  if (mean > 48) return 32;
  if (mean > 12) return 16;
  return 8;
}

#define SPH_ROWS_LAUNCH(KERNEL, W, grid, s, ...)                              \
  do {                                                                        \
    if ((W) == 32) KERNEL<32><<<grid, kBlock, 0, (s)->stream>>>(__VA_ARGS__); \
    else if ((W) == 16) KERNEL<16><<<grid, kBlock, 0, (s)->stream>>>(__VA_ARGS__); \
    else KERNEL<8><<<grid, kBlock, 0, (s)->stream>>>(__VA_ARGS__);            \
    SPH_LAUNCHED(s);                                                          \
  } while (0)

sph_rt_status launch_properties(sph_rt *s, double dt, const double *ge_c, const double *gE_c) {
  Phys ph = make_phys(s, dt);
  int g = grid_items(s, s->n, kBlock);
  props_point_kernel<<<g, kBlock, 0, s->stream>>>(ph, s->n, s->kind, s->rho, s->sigma0, s->e,
                                                   s->T, s->sigma, s->f, s->R, s->lambda, s->D);
  SPH_LAUNCHED(s);
  if (s->cfg.limiter != SPH_RT_LIMITER_NONE) {
    // pair geometry once per particle set, if it fits a modest share of memory
    const bool d3 = s->dim == 3;
    const double geom_bytes = 28.0 * (double)s->nnz_nbr;
    if (!s->gvx && geom_bytes < 24e9) {
      s->gcol = dalloc<int32_t>(s, s->nnz_nbr);
      s->gvx = dalloc<double>(s, s->nnz_nbr);
      s->gvy = dalloc<double>(s, s->nnz_nbr);
      s->gvz = d3 ? dalloc<double>(s, s->nnz_nbr) : nullptr;
      if (!s->gcol || !s->gvx || !s->gvy || (d3 && !s->gvz)) return SPH_RT_ENOMEM;
      grad_geom_kernel<<<grid_items(s, s->n_int, kWarpsPerBlock), kBlock, 0, s->stream>>>(
          s->n_int, s->nbr_ptr, s->nbr_col, s->nbr_F, s->px, s->py, s->pz, s->V, s->kind,
          s->copysrc, s->gcol, s->gvx, s->gvy, s->gvz);
      SPH_LAUNCHED(s);
    }
    if (s->gvx) {
      RowShape sh = shape_for_mean(s->n_int ? (double)s->nnz_nbr / (double)s->n_int : 0.0);
      int gr = row_grid_blocks(s->num_sms, s->n_int, sh.W, kPairMinBlocks);
      if (d3)
        SPH_DISPATCH_SHAPE(sh.W, sh.U,
                           (props_grad_pre_kernel<W, U, true><<<gr, kBlock, 0, s->stream>>>(
                               ph, s->n_int, s->nbr_ptr, s->gcol, s->gvx, s->gvy, s->gvz, s->E,
                               s->sigma, s->R, s->lambda, s->D)));
      else
        SPH_DISPATCH_SHAPE(sh.W, sh.U,
                           (props_grad_pre_kernel<W, U, false><<<gr, kBlock, 0, s->stream>>>(
                               ph, s->n_int, s->nbr_ptr, s->gcol, s->gvx, s->gvy, nullptr, s->E,
                               s->sigma, s->R, s->lambda, s->D)));
      SPH_LAUNCHED(s);
    } else {
      int W = row_width(s->nnz_nbr, s->n_int);
      int gr = grid_items(s, s->n_int, kBlock / W);
      SPH_ROWS_LAUNCH(props_grad_kernel, W, gr, s, ph, s->n_int, s->nbr_ptr, s->nbr_col,
                      s->nbr_F, s->px, s->py, s->pz, s->V, s->kind, s->copysrc, s->E, s->sigma,
                      s->R, s->lambda, s->D);
    }
  }
  if (s->n > s->n_int) {
    ghost_kernel<<<grid_items(s, s->n - s->n_int, kBlock), kBlock, 0, s->stream>>>(
        s->n_int, s->n, s->kind, s->copysrc, s->slot2caller, ge_c, gE_c, s->T, s->sigma, s->f,
        s->R, s->lambda, s->D, s->e, s->E);
    SPH_LAUNCHED(s);
  }
  return SPH_RT_OK;
}

sph_rt_status launch_assembly(sph_rt *s, double dt, double *gersh_out) {
  Phys ph = make_phys(s, dt);
  if (s->sl.ptr) {
    const SlicedView<double> A =
        sliced_view<double>(s->sl, s->n_int, s->nnz_mat, s->sl_G, nullptr, nullptr);
    const int grid = sliced_grid(s, s->n_int, 4);
    const size_t smem = sizeof(double) * (size_t)s->sl.dict_max;
    if (s->sl_val32)
      assemble_sliced_kernel<true><<<grid, kBlock, smem, s->stream>>>(
          ph, A, s->sl_val, s->sl_val32, s->gh_ptr, s->gh_slot, s->gh_W, s->V, s->sigma, s->f,
          s->D, s->E, s->diag, s->invdiag, s->gb, s->partials, &s->sc->counter, gersh_out,
          s->diag32, s->invdiag32);
    else
      assemble_sliced_kernel<false><<<grid, kBlock, smem, s->stream>>>(
          ph, A, s->sl_val, nullptr, s->gh_ptr, s->gh_slot, s->gh_W, s->V, s->sigma, s->f, s->D,
          s->E, s->diag, s->invdiag, s->gb, s->partials, &s->sc->counter, gersh_out, nullptr,
          nullptr);
    SPH_LAUNCHED(s);
    return SPH_RT_OK;
  }
  RowShape sh = shape_for_mean(s->n_int ? (double)s->nnz_mat / (double)s->n_int : 0.0);
  int gr = row_grid_blocks(s->num_sms, s->n_int, sh.W, kPairMinBlocks);
  // the mixed form gets its FP32 copy of the fine operator in the same pass
  if (s->mat_val32)
    SPH_DISPATCH_SHAPE(sh.W, sh.U,
                       (assemble_kernel<W, U, true><<<gr, kBlock, 0, s->stream>>>(
                           ph, s->n_int, s->mat_ptr, s->mat_col, s->mat_G, s->mat_val, s->gh_ptr,
                           s->gh_slot, s->gh_W, s->V, s->sigma, s->f, s->D, s->E, s->diag,
                           s->invdiag, s->gb, s->partials, &s->sc->counter, gersh_out,
                           s->mat_val32, s->diag32, s->invdiag32)));
  else
    SPH_DISPATCH_SHAPE(sh.W, sh.U,
                       (assemble_kernel<W, U, false><<<gr, kBlock, 0, s->stream>>>(
                           ph, s->n_int, s->mat_ptr, s->mat_col, s->mat_G, s->mat_val, s->gh_ptr,
                           s->gh_slot, s->gh_W, s->V, s->sigma, s->f, s->D, s->E, s->diag,
                           s->invdiag, s->gb, s->partials, &s->sc->counter, gersh_out,
                           nullptr, nullptr, nullptr)));
  SPH_LAUNCHED(s);
  return SPH_RT_OK;
}

sph_rt_status launch_rhs(sph_rt *s, double dt) {
  Phys ph = make_phys(s, dt);
  int g = grid_items(s, s->n_int, kBlock);
  rhs_kernel<<<g, kBlock, 0, s->stream>>>(ph, s->n_int, s->V, s->sigma, s->f, s->E_old, s->e_l,
                                           s->E_l, s->QE, s->gb, s->b, s->x, s->cfg.tol_krylov,
                                           s->sc, s->partials, s->E_hist[0], s->E_hist[1],
                                           s->E_hist[2]);
  SPH_LAUNCHED(s);
  return SPH_RT_OK;
}

// order and weights of the extrapolated start of the step's first solve (order 0: E^l)
sph_rt_status launch_step_start(sph_rt *s, int depth, int order, const double *w) {
  step_start_kernel<<<grid_items(s, s->n_int, kBlock), kBlock, 0, s->stream>>>(
      s->n_int, depth, s->e, s->E, s->e_old, s->E_old, s->E_l, s->E_hist[0], s->E_hist[1],
      s->E_hist[2], s->sc, order, w[0], w[1], w[2], w[3]);
  SPH_LAUNCHED(s);
  return SPH_RT_OK;
}

sph_rt_status launch_newton(sph_rt *s, double dt, const double *E_new, double *E_prev,
                            const double *e_start, double *e_out, const OuterTail &tail) {
  Phys ph = make_phys(s, dt);
  int g = grid_items(s, s->n_int, kBlock);
  newton_kernel<<<g, kBlock, 0, s->stream>>>(ph, s->n_int, s->rho, s->sigma, s->e_old, s->Qe,
                                              E_new, E_prev, e_start, e_out, s->sc, s->partials, tail);
  SPH_LAUNCHED(s);
  return SPH_RT_OK;
}

sph_rt_status launch_step_begin(sph_rt *s, const double *Qe, const double *QE, const double *ge,
                                const double *gE) {
  step_begin_kernel<<<grid_reduce(s, s->n), kBlock, 0, s->stream>>>(
      s->n_int, s->n, s->slot2caller, s->kind, Qe, QE, ge, gE, s->mass, s->V, s->e, s->E,
      s->e_bak, s->E_bak, s->Qe, s->QE, s->sc, s->partials);
  SPH_LAUNCHED(s);
  return SPH_RT_OK;
}

sph_rt_status launch_step_end(sph_rt *s, double dt, const double *e_new, const double *E_new) {
  step_end_kernel<<<grid_reduce(s, s->n), kBlock, 0, s->stream>>>(
      make_phys(s, dt), s->n_int, s->n, s->nnz_gh, s->copysrc, e_new, E_new, s->e_bak, s->E_bak,
      s->mass, s->V, s->Qe, s->QE, s->gh_row, s->gh_slot, s->gh_W, s->D, s->e, s->E, s->sc,
      s->partials);
  SPH_LAUNCHED(s);
  return SPH_RT_OK;
}

// ---------------------------------------------------------------------------
// Time step choice (Sec. 3.3, Eq. energy-fractional), after a converged step:
//   xbar = sum_i x_i^n V_i / sum_i V_i                       (volume average)
//   eta_x = max_i |x_i^n - x_i^{n-1}| / (x_i^n + target xbar + floor)
//   dt_x = dt (target / eta_x)^(1/2)
//   dt_next = min(dt_e, dt_E, growth dt, dt_max), at least dt_min
// for x = e and x = E over the interior particles.  x^{n-1} is the snapshot
// taken at the start of the step.
// ---------------------------------------------------------------------------
__global__ void dtc_sums_kernel(int64_t n_int, const double *V, const double *e, const double *E,
                                Scalars *sc, double *partials) {
  double a = 0.0, b = 0.0, v = 0.0;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n_int;
       i += (int64_t)gridDim.x * blockDim.x) {
    const double Vi = V[i];
    a += e[i] * Vi;
    b += E[i] * Vi;
    v += Vi;
  }
  double part[3] = {a, b, v}, out[3];
  block_sums(part);
  const bool mx[3] = {false, false, false};
  if (last_block_combine<3>(part, partials, &sc->counter, out, mx) && threadIdx.x == 0) {
    sc->dtc_ebar = out[0] / out[2];
    sc->dtc_Ebar = out[1] / out[2];
  }
}

struct DtControl {
  double dt, target, growth, dt_min, dt_max, floor;
};

__global__ void dtc_eta_kernel(int64_t n_int, const double *e, const double *E,
                               const double *e_old, const double *E_old, DtControl c, Scalars *sc,
                               double *partials) {
  const double de = c.target * sc->dtc_ebar + c.floor, dE = c.target * sc->dtc_Ebar + c.floor;
  double me = 0.0, mE = 0.0;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n_int;
       i += (int64_t)gridDim.x * blockDim.x) {
    const double en = e[i], En = E[i];
    me = fmax(me, fabs(en - e_old[i]) / (en + de));
    mE = fmax(mE, fabs(En - E_old[i]) / (En + dE));
  }
  double part[2] = {me, mE}, out[2];
  const bool mx[2] = {true, true};
  block_reduce(part, mx);
  if (last_block_combine<2>(part, partials, &sc->counter, out, mx) && threadIdx.x == 0) {
    double next = fmin(c.growth * c.dt, c.dt_max);
    if (out[0] > 0.0) next = fmin(next, c.dt * sqrt(c.target / out[0]));
    if (out[1] > 0.0) next = fmin(next, c.dt * sqrt(c.target / out[1]));
    sc->dtc_eta_e = out[0];
    sc->dtc_eta_E = out[1];
    sc->dtc_next = fmax(next, c.dt_min);
  }
}

sph_rt_status launch_dt_control(sph_rt *s, double dt) {
  const int g = grid_reduce(s, s->n_int);
  dtc_sums_kernel<<<g, kBlock, 0, s->stream>>>(s->n_int, s->V, s->e, s->E, s->sc, s->partials);
  SPH_LAUNCHED(s);
  const DtControl c = {dt, s->cfg.dt_target, s->cfg.dt_growth, s->cfg.dt_min, s->cfg.dt_max,
                       s->cfg.dt_eta_floor};
  dtc_eta_kernel<<<g, kBlock, 0, s->stream>>>(s->n_int, s->e, s->E, s->e_bak, s->E_bak, c, s->sc,
                                              s->partials);
  SPH_LAUNCHED(s);
  return SPH_RT_OK;
}

sph_rt_status launch_totals(sph_rt *s, const double *e, const double *E) {
  int g = grid_reduce(s, s->n_int);
  totals_kernel<<<g, kBlock, 0, s->stream>>>(s->n_int, s->mass, s->V, e, E, s->sc, s->partials);
  SPH_LAUNCHED(s);
  return SPH_RT_OK;
}

sph_rt_status launch_gather_interior(sph_rt *s, const double *in_c, double *out) {
  int g = grid_items(s, s->n_int, kBlock);
  gather_interior_kernel<<<g, kBlock, 0, s->stream>>>(in_c, s->slot2caller, s->n_int, out);
  SPH_LAUNCHED(s);
  return SPH_RT_OK;
}

sph_rt_status launch_scatter_caller(sph_rt *s, const double *in_s, int64_t count, double *out_c) {
  int g = grid_items(s, count, kBlock);
  scatter_caller_kernel<<<g, kBlock, 0, s->stream>>>(in_s, s->slot2caller, count, out_c);
  SPH_LAUNCHED(s);
  return SPH_RT_OK;
}

}  // namespace sphrt
