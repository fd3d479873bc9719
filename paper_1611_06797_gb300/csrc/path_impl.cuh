// Launchers of the hot path for one real type T.  Included once per precision by
// kernels_f64.cu / kernels_f32.cu, which explicitly instantiate Path<T>.
#pragma once
#include <algorithm>
#include <type_traits>

#include "kernels.cuh"
#include "once_device.h"
#include "plane_block.h"
#include "sized.h"
#include "sym.cuh"

namespace ltmp2 {

// f(integral_constant<int, n>) for the grid size n; false when no kernel is compiled for it
template <typename F> static bool with_size(int n, F &&f) {
  switch (n) {
#define LTMP2_CASE(NN)                      \
  case NN:                                  \
    f(std::integral_constant<int, NN>{});   \
    return true;
    LTMP2_FOR_EACH_N(LTMP2_CASE)
#undef LTMP2_CASE
    default:
      return false;
  }
}

// Plane kernels: 0 = k_planes (full-plane passes), 1 = k_planes2 (compacted passes),
// 2 = k_planes3 (product in registers, compact intermediate), 3 = k_planes4 (as 2, each
// warp on its own occupied planes without block barriers).
// ib = occupied planes per block (kernel 3: per warp step); 0 picks the default of each kernel.
// FP64 has one plane kernel, 2 in fixed point: the others are accepted and run it.  In FP32 kernel 2
// takes pairs of columns.
template <typename T> static size_t plane_smem(const Plan &p, int kernel, int ib);
template <typename T> static int plane_ib_default(const Plan &p, int kernel) {
  const int n = p.n;
  const size_t plane = (size_t)n * (n + 1) * sizeof(cpx<T>);
  const int nxa = p.mxhi_aux - p.mxlo_aux + 1;
  int ib;
  if (kernel == 3) {
    // as many planes per warp step as fill the 32 lanes of the x pass, at least 2 (two
    // planes per warp step were fastest in FP32 on the 24^3 and 36^3 workloads: 20.6 and
    // 790 ms per plane pass against 23.5 and 905 with one), within ~100 KB
    ib = (32 + n - 1) / n;
    if (ib < 2) ib = 2;
    const size_t per = (size_t)kPlaneWarps * plane_stride(n, nxa) * sizeof(cpx<T>);
    while (ib > 1 && plane + ib * per > 100 * 1024) --ib;
  } else if (kernel == 0) {
    ib = (int)((96 * 1024) / plane) - 1;   // about 96 KB of shared memory
    if (ib > 8) ib = 8;
  } else if (kernel == 2 && std::is_same<T, double>::value) {
    // fixed point: blocks of two warps whose lanes the n ib lines of the x pass fill, or of three
    // where they fill those better by 15 % (two warps keep more blocks resident).  One Laplace point's
    // plane pass: 20^3 with 3 of 4 planes 9.9 against 11.8 ms, 18^3 4.2 against 4.9, 27^3 with 2 of 4
    // 19.8 against 21.9, 32^3 18.5 against 20.2; 24^3 with 4 (three warps) 9.8 against 11.5 with 2
    const int two = 64 / n, three = 96 / n;
    ib = two > 0 && 1.15 * two * n / 64.0 >= three * n / 96.0 ? two : three;
    while (ib > 1 && plane + (sizeof(int) * p.n_daux + 64) + (size_t)ib * plane_stride(n, nxa) * sizeof(cpx<T>) > 100 * 1024) --ib;
  } else if (kernel == 2) {
    // blocks of 64 threads: the fewest steps of 64 lines per occupied (x pass and y pass), weighed against
    // the shared memory above what six blocks per SM (the registers' limit) have
    ib = 1;
    double best = 1e9;
    for (int k = 1; k <= 8; ++k) {
      const double steps = (double)((k * n + 63) / 64 + (k * nxa + 63) / 64) / k;
      const double score = steps * std::max(1.0, (double)plane_smem<T>(p, 2, k) / 36864.0);
      if (score < 0.99 * best) {
        best = score;
        ib = k;
      }
    }
  } else {
    const size_t per = plane + (size_t)p.n_daux * sizeof(cpx<T>);
    ib = (int)((100 * 1024 - plane - 3 * sizeof(int) * (n + 1) - 64) / per);
    if (ib > 384 / n) ib = 384 / n;
  }
  if (ib > p.n_occ) ib = p.n_occ;
  if (ib < 1) ib = 1;
  return ib;
}

template <typename T> static size_t plane_smem(const Plan &p, int kernel, int ib) {
  const int n = p.n;
  const size_t plane = (size_t)n * (n + 1) * sizeof(cpx<T>);
  const int nxa = p.mxhi_aux - p.mxlo_aux + 1;
  if (kernel == 0) return plane * (1 + ib);
  const size_t q = (size_t)plane_stride(n, nxa);
  if (kernel == 2) return 16 * ((size_t)n * (n + 1) + (size_t)ib * q) + sizeof(int) * p.n_daux;
  if (kernel == 3) return plane + (size_t)kPlaneWarps * ib * q * sizeof(cpx<T>) + sizeof(int) * p.n_daux;
  return plane * (1 + ib) + (size_t)ib * p.n_daux * sizeof(cpx<T>) + 3 * sizeof(int) * nxa;
}

// launch the plane kernel for the ncols columns of the current slab (z1 -> tbuf)
template <typename T> static cudaError_t launch_planes(const Plan &p, int ncols, int kernel, int ib, cudaStream_t st) {
  constexpr bool kFp64 = std::is_same<T, double>::value;
  if (kFp64) kernel = 2;
  if (ib <= 0) ib = plane_ib_default<T>(p, kernel);
  if (kFp64) ib = plane_block_f64(p.n, ib).ib;
  if (kernel == 2)
    while (ib > 1 && plane_smem<T>(p, kernel, ib) > 200 * 1024) --ib;
  const size_t smem = plane_smem<T>(p, kernel, ib);
  int threads = kernel == 3 ? 32 * kPlaneWarps : kFp64 ? plane_block_f64(p.n, ib).threads : ib * p.n;
  if (threads < 64 || (kernel == 2 && !kFp64)) threads = 64;
  if (threads > 1024 || smem > 200 * 1024) return cudaErrorInvalidValue;
  if (!with_size(p.n, [&](auto n) { Sized<T, decltype(n)::value>::planes(p, ncols, kernel, ib, threads, smem, st); }))
    return cudaErrorInvalidValue;
  return cudaGetLastError();
}

template <typename T> bool Path<T>::plane_feasible(const Plan &p, int kernel, int ib) {
  if (kernel < 0 || kernel > 3 || ib < 0) return false;
  if (ib == 0) ib = plane_ib_default<T>(p, kernel);
  const int threads = kernel == 3 ? 32 * kPlaneWarps : ib * p.n;
  size_t smem = plane_smem<T>(p, kernel, ib);
  // FP32 pairs: as many planes as fit unpaired are accepted, and a launch takes as many pairs as fit
  if (kernel == 2 && std::is_same<T, float>::value) smem = smem / 2 + 2 * p.n_daux;
  return threads <= 1024 && smem <= 200 * 1024;
}

template <typename T>
cudaError_t Path<T>::plane_pass(const Plan &p, int ncols, int kernel, int ib, cudaStream_t st) {
  return launch_planes<T>(p, ncols, kernel, ib, st);
}

struct ScopedStage {
  StageTimer *tm;
  int st;
  ScopedStage(StageTimer *t, int s) : tm(t), st(s) { if (tm) tm->begin(st); }
  ~ScopedStage() { if (tm) tm->end(st); }
};

template <typename T> cudaError_t Path<T>::init_device() {
  static OncePerDevice once;
  int dev = 0;
  const cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  // twiddle tables and dynamic shared memory limits of the FFT kernels
  return once.run(dev, [] {
    cudaError_t r = cudaSuccess;
    for (int n : kFftSizes)
      if (r == cudaSuccess) with_size(n, [&](auto c) { r = Sized<T, decltype(c)::value>::init(); });
    return r;
  });
}

template <typename T>
cudaError_t Path<T>::setup_occupied(const Plan &p, const void *c_occ_dev, cudaStream_t st) {
  const int n = p.n;
  const size_t n3 = (size_t)n * n * n;
  cudaError_t e = cudaMemsetAsync(p.cgrid, 0, sizeof(cpx<T>) * n3 * p.n_occ, st);
  if (e != cudaSuccess) return e;
  const cpx<T> *c = (const cpx<T> *)c_occ_dev;
  k_scatter_grid<T><<<dim3((p.n_pw + 255) / 256, p.n_occ), 256, 0, st>>>(p, p.n_occ, c, (cpx<T> *)p.cgrid);
  e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  // p.z1 is the scratch (max_cols >= n_occ always holds)
  if (!with_size(n, [&](auto c) {
        Sized<T, decltype(c)::value>::zinv(p, p.n_occ, c_occ_dev, p.z1, st);
        Sized<T, decltype(c)::value>::planes_store(p, p.z1, st);
      }))
    return cudaErrorInvalidValue;
  if constexpr (std::is_same<T, double>::value) k_unorm3<<<1, 256, 0, st>>>(p);
  return cudaGetLastError();
}

template <typename T> cudaError_t Path<T>::transpose_virtuals(const Plan &p, void *out, cudaStream_t st) {
  const dim3 grid((p.n_pw + 31) / 32, (p.n_v + 31) / 32), block(32, 8);
  const size_t n = (size_t)p.n_v * p.n_pw;
  for (int k = 0; k < (p.nk > 0 ? p.nk : 1); ++k) {
    if (p.real_basis) k_transpose<T><<<grid, block, 0, st>>>(p.n_v, p.n_pw, (const T *)p.cv, (T *)out);
    else k_transpose<cpx<T>><<<grid, block, 0, st>>>(p.n_v, p.n_pw, (const cpx<T> *)p.cv + k * n, (cpx<T> *)out + k * n);
    const cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

template <typename T> cudaError_t Path<T>::overlap_setup(const Plan &p, cudaStream_t st) {
  // r_a transposed into pt ([n_pw][n_v]); pt is free on this route (no Green's function)
  k_transpose<T><<<dim3((p.n_pw + 31) / 32, (p.n_v + 31) / 32), dim3(32, 8), 0, st>>>(p.n_v, p.n_pw, (const T *)p.cv,
                                                                                      (T *)p.pt);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  for (int gp0 = 0; gp0 < p.n_prim; gp0 += p.max_prim) {
    const int np = p.n_prim - gp0 < p.max_prim ? p.n_prim - gp0 : p.max_prim;
    const int ncols = np * p.n_occ;
    // rho^T[(G', j)][a] = sum_q (U e^{-iG'r} phi_j)[q] r_a[q]: U is unitary and r_a = U phi_a
    // is real, so this is <a| e^{-iG'r} |j> (Eq. SCHovrlp), step (i) of Sec. III A
    k_gather_s_real<T><<<dim3((p.n_pw + 255) / 256, ncols), 256, 0, st>>>(p, gp0, np, (cpx<T> *)p.st, true);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    dim3 grid((p.n_v + 63) / 64, (ncols + 63) / 64);
    k_rgemm<T, cpx<T>, true><<<grid, 256, 0, st>>>(ncols, p.n_v, p.n_pw, (const cpx<T> *)p.st, p.n_pw,
                                                    (const T *)p.pt, p.n_v, nullptr,
                                                    (cpx<T> *)p.rt + (size_t)gp0 * p.n_occ * p.n_v, p.n_v);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
  }
  return cudaSuccess;
}

template <typename T>
cudaError_t Path<T>::green(const Plan &p, double tau, cudaStream_t st, StageTimer *tm) {
  ScopedStage s(tm, kStageGreen);
  k_dscale<T><<<(p.n_orb + 255) / 256, 256, 0, st>>>(p.n_orb, p.n_occ, p.eps, p.mu, tau, (T *)p.dscale);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  // no Green's function on the paper's route, nor when W goes through the virtual space
  if (p.route == 1 || p.w_virtual) return cudaSuccess;
  if constexpr (std::is_same<T, float>::value) {
    if (p.tc && p.tc->green_on()) {
      // precision form, real basis: P_r on the tensor cores (3xTF32), then the split of P_r
      // into the transformed-state GEMM's operands
      if ((e = tc_green(*p.tc, (const float *)p.dscale + p.n_occ, p.pt, st)) != cudaSuccess) return e;
      return tc_pack_b(*p.tc, p.pt, st);
    }
  }
  const int M = p.n_pw, N = p.n_pw, K = p.nv_tau > 0 ? p.nv_tau : p.n_v;
  if (p.oz) {
    // on the tensor cores by exact slices, then the result's own slices for the W product
    const void *dv = (const T *)p.dscale + p.n_occ;
    if ((e = oz_green<T>(*p.oz, p.real_basis ? p.rvt : p.cvt, dv, 0, K, p.pt, st)) != cudaSuccess) return e;
    return oz_split_b<T>(*p.oz, p.pt, st);
  }
  dim3 grid((N + 63) / 64, (M + 63) / 64);
  if (p.real_basis) {
    // P_r[q][p] = sum_a r_a(q) e^{-(e_a-mu)tau} r_a(p), r_a the real coordinates of a
    k_rgemm<T, T, false><<<grid, 256, 0, st>>>(M, N, K, (const T *)p.cv, p.n_pw, (const T *)p.cv, p.n_pw,
                                               (const T *)p.dscale + p.n_occ, (T *)p.pt, p.n_pw);
  } else {
    // P^T[q][p] = sum_a conj(c_a(q)) e^{-(e_a-mu)tau} c_a(p)
    k_cgemm<T, false, true><<<grid, 256, 0, st>>>(M, N, K, (const cpx<T> *)p.cv, p.n_pw,
                                                  (const cpx<T> *)p.cv, p.n_pw,
                                                  (const T *)p.dscale + p.n_occ, (cpx<T> *)p.pt, p.n_pw);
  }
  return cudaGetLastError();
}

template <typename T>
cudaError_t Path<T>::slab_pre(const Plan &p, int gp0, int np, cudaStream_t st, StageTimer *tm) {
  const int n = p.n, no = p.n_occ;
  const bool sym = p.sym_nj > 0;   // the columns of the pass's orbitals, without the occupied factors
  const int ncols = sym ? np * p.sym_nj : np * p.slots_per_prim() * no;
  cudaError_t e;
  if (p.route != 1) {
    ScopedStage s(tm, kStageGatherZ);
    if (p.real_basis)
      k_gather_s_real<T><<<dim3((p.n_pw + 255) / 256, ncols), 256, 0, st>>>(p, gp0, np, (cpx<T> *)p.st, sym);
    else
      k_gather_s<T><<<dim3((p.n_pw + 255) / 256, ncols), 256, 0, st>>>(p, gp0, np, (cpx<T> *)p.st, sym);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
  }
  {
    ScopedStage s(tm, kStageWGemm);
    bool done = false;
    if (p.route == 1) {
      // W (real-basis coordinates, before the e^{(e_j-mu)tau} row factor) =
      // sum_a rho^T[(G', j)][a] e^{-(e_a-mu)tau} r_a: step (iii) with the stored overlap densities
      dim3 grid((p.n_pw + 63) / 64, (ncols + 63) / 64);
      const int nv = p.nv_tau > 0 ? p.nv_tau : p.n_v;
      k_rgemm<T, cpx<T>, true><<<grid, 256, 0, st>>>(ncols, p.n_pw, nv,
                                                      (const cpx<T> *)p.rt + (size_t)gp0 * no * p.n_v, p.n_v,
                                                      (const T *)p.cv, p.n_pw, (const T *)p.dscale + p.n_occ,
                                                      (cpx<T> *)p.wt, p.n_pw);
      if ((e = cudaGetLastError()) != cudaSuccess) return e;
      done = true;
    } else if (p.w_virtual) {
      // X^T = (U S)^T R_v'^T [ncols][nv] in the z1 buffer (free until the z transform; it
      // holds n n_dorb >= n_pw > nv values per column), then W^T = X^T D' R_v'
      const int nv = p.nv_tau;
      const T *dv = (const T *)p.dscale + p.n_occ;
      if (p.oz) {
        if ((e = oz_virtual<T>(*p.oz, p.st, ncols, dv, nv, p.z1, p.wt, st)) != cudaSuccess) return e;
      } else {
        dim3 gx((nv + 63) / 64, (ncols + 63) / 64);
        k_rgemm<T, cpx<T>, true><<<gx, 256, 0, st>>>(ncols, nv, p.n_pw, (const cpx<T> *)p.st, p.n_pw,
                                                      (const T *)p.rvt, p.n_v, nullptr, (cpx<T> *)p.z1, nv);
        if ((e = cudaGetLastError()) != cudaSuccess) return e;
        dim3 gw((p.n_pw + 63) / 64, (ncols + 63) / 64);
        k_rgemm<T, cpx<T>, true><<<gw, 256, 0, st>>>(ncols, p.n_pw, nv, (const cpx<T> *)p.z1, nv, (const T *)p.cv,
                                                      p.n_pw, dv, (cpx<T> *)p.wt, p.n_pw);
        if ((e = cudaGetLastError()) != cudaSuccess) return e;
      }
      done = true;
    }
    if constexpr (std::is_same<T, float>::value) {
      // the opt-in 3xTF32 Green's function leaves its operands to the 3xTF32 product
      if (!done && p.tc && p.tc->green_on()) {
        if ((e = tc_wgemm(*p.tc, p.st, ncols, p.wt, st)) != cudaSuccess) return e;
        done = true;
      }
    }
    if (p.oz && !done) {
      if ((e = oz_wgemm<T>(*p.oz, p.st, ncols, p.wt, st)) != cudaSuccess) return e;
      done = true;
    }
    if (!done) {
      dim3 grid((p.n_pw + 63) / 64, (ncols + 63) / 64);
      if (p.real_basis)
        k_rgemm<T, cpx<T>, true><<<grid, 256, 0, st>>>(ncols, p.n_pw, p.n_pw, (const cpx<T> *)p.st, p.n_pw,
                                                        (const T *)p.pt, p.n_pw, nullptr, (cpx<T> *)p.wt,
                                                        p.n_pw);
      else
        k_cgemm<T, true, false><<<grid, 256, 0, st>>>(ncols, p.n_pw, p.n_pw, (const cpx<T> *)p.st, p.n_pw,
                                                      (const cpx<T> *)p.pt, p.n_pw, nullptr,
                                                      (cpx<T> *)p.wt, p.n_pw);
      if ((e = cudaGetLastError()) != cudaSuccess) return e;
    }
  }
  // real basis: W^T back to plane-wave coefficients, into the (now free) S^T buffer
  const cpx<T> *w_pw = (const cpx<T> *)p.wt;
  if (p.real_basis) {
    ScopedStage s(tm, kStageGatherZ);
    k_from_real_basis<T><<<dim3((p.n_pw + 255) / 256, ncols), 256, 0, st>>>(
        p, (const cpx<T> *)p.wt, (cpx<T> *)p.st, p.route == 1 ? (const T *)p.dscale : nullptr);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    w_pw = (const cpx<T> *)p.st;
  }
  if constexpr (std::is_same<T, double>::value) {
    ScopedStage s(tm, kStageGatherZ);
    k_wnorm<<<ncols, 128, 0, st>>>(p, (const cpx<T> *)w_pw);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
  }
  {
    ScopedStage s(tm, kStageGatherZ);
    if (!with_size(n, [&](auto c) { Sized<T, decltype(c)::value>::zinv(p, ncols, w_pw, p.z1, st); }))
      return cudaErrorInvalidValue;
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
  }
  return cudaSuccess;
}

template <typename T>
cudaError_t Path<T>::slab(const Plan &p, int gp0, int np, double coef, cudaStream_t st, StageTimer *tm) {
  const int n = p.n, no = p.n_occ;
  const int nslots = np * p.slots_per_prim();
  const int ncols = nslots * no;
  cudaError_t e;
  if ((e = slab_pre(p, gp0, np, st, tm)) != cudaSuccess) return e;
  const bool lev = p.n_lev > 1;
  const size_t smem_col = (lev ? 2 : 1) * (size_t)p.n_aux * sizeof(cpx<T>);
  const int npairs = p.real_orb ? np * (no * (no + 1) / 2) : np * no * no;
  int col_threads = ((p.n_daux + 31) / 32) * 32;
  if (col_threads > 256) col_threads = 256;   // the column kernel's launch bound (FP64 N >= 36 uses ~255 registers)
  {
    ScopedStage s(tm, kStagePlane);
    if ((e = launch_planes<T>(p, ncols, p.plane_kernel, p.plane_ib, st)) != cudaSuccess) return e;
  }
  {
    ScopedStage s(tm, kStageColumn);
    if (!with_size(n, [&](auto c) {
          Sized<T, decltype(c)::value>::zcol(p, gp0, np, npairs, col_threads, smem_col, lev, st);
        }))
      return cudaErrorInvalidValue;
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
  }
  return slab_post(p, gp0, np, coef, st, tm);
}

template <typename T>
cudaError_t Path<T>::slab_post(const Plan &p, int gp0, int np, double coef, cudaStream_t st, StageTimer *tm) {
  const int no = p.n_occ;
  const bool lev = p.n_lev > 1;
  cudaError_t e;
  {
    ScopedStage s(tm, kStageDirect);
    int th = no < 128 ? ((no + 31) / 32) * 32 : 128;
    // FP32 (general orbitals, or the tensor-core product off): the shared-memory tiled kernel, which reads
    // each co-density once per 32 others: two Laplace points of one or two slabs of 48 / 64 / 96 / 128
    // occupied take 0.78 / 1.27 / 1.38 / 0.86 ms, 1.24 / 2.27 / 3.39 / 3.35 ms by warp-level sums (which pad
    // nothing: 0.23 against 0.09 ms with 8 occupied, 1.33 against 1.16 ms with 32).  FP64 is bound by the
    // FP64 pipe, and the warp-level sums take the real part alone where only that enters.
    bool done = false;
    if constexpr (std::is_same<T, float>::value) {
      if (!lev && p.tc && p.tc->direct_on()) {   // real orbitals: one tensor-core product per G'
        if ((e = tc_direct(*p.tc, p.mdiag, p.v_aux32, np, p.yd, st)) != cudaSuccess) return e;
        done = true;
      }
    }
    if (done) {
    } else if (lev) {
      k_direct_lev<T><<<dim3(np, no), th, 0, st>>>(p, np, (const cpx<T> *)p.mdiag, p.yd);
    } else if constexpr (std::is_same<T, float>::value) {
      const int t = (no + 31) / 32;
      k_direct_tiled<T><<<dim3(np, t, t), 256, 0, st>>>(p, np, (const cpx<T> *)p.mdiag, p.yd);
    } else {
      const int t = (no + 3) / 4;
      k_direct_w<T><<<np * (p.real_orb ? t * (t + 1) / 2 : t * t), 128, 0, st>>>(p, np, (const cpx<T> *)p.mdiag, p.yd);
    }
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
  }
  {
    ScopedStage s(tm, kStageAccum);
    k_accum<<<(no * no + 3) / 4, 128, 0, st>>>(p, gp0, np, coef, p.sx, p.yd);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    if (lev) {
      k_accum_lev<<<dim3((no * no + 31) / 32, p.n_lev - 1), 32, 0, st>>>(p, gp0, np, coef);
      if ((e = cudaGetLastError()) != cudaSuccess) return e;
    }
  }
  return cudaSuccess;
}

// pair slots of a pass over sym_nj orbitals from sym_j0
static int sym_pairs(const Plan &p) { return p.sym_nj * p.sym_j0 + p.sym_nj * (p.sym_nj + 1) / 2; }

// orbitals per pass and G' per part of it: columns as of a slab; whole orbitals j if they fit, else one j
// in several parts
static void sym_shape(const Plan &p, int &nj, int &np_max) {
  const int budget = p.max_prim * p.slots_per_prim() * p.n_occ;
  nj = std::max(1, std::min(std::min(budget / p.n_idx, p.n_occ), p.sym_nj_cap));
  np_max = std::max(1, std::min(p.n_idx, budget / nj));
}

// The matrices S_ij of the pass of orbitals p.sym_j0 .. + p.sym_nj, in parts of np_max G'
template <typename T>
static cudaError_t sym_pass(const Plan &p, int np_max, cudaStream_t st, StageTimer *tm, long long *launches) {
  const int n_idx = p.n_idx, threads = std::min(256, ((p.n_daux + 31) / 32) * 32);
  const size_t smem = (size_t)p.sym_planes * n_idx * sizeof(cpx<T>);
  cudaError_t e;
  for (int g0 = 0; g0 < n_idx; g0 += np_max) {
    const int np = std::min(np_max, n_idx - g0), ncols = np * p.sym_nj;
    if ((e = Path<T>::slab_pre(p, g0, np, st, tm)) != cudaSuccess) return e;
    {
      ScopedStage s(tm, kStagePlane);
      if ((e = launch_planes<T>(p, ncols, p.plane_kernel, p.plane_ib, st)) != cudaSuccess) return e;
    }
    {
      ScopedStage s(tm, kStageColumn);
      if (!with_size(p.n, [&](auto c) { Sized<T, decltype(c)::value>::zsym(p, g0, ncols, threads, smem, st); }))
        return cudaErrorInvalidValue;
      if ((e = cudaGetLastError()) != cudaSuccess) return e;
    }
    *launches += Path<T>::pre_launches(p) + 2;
  }
  return cudaSuccess;
}
// the rows of the pass's exchange sums
template <typename T> static cudaError_t launch_xsym(const Plan &p, cudaStream_t st) {
  k_xsym<T><<<dim3(sym_pairs(p), (p.n_idx + 31) / 32), 256, 0, st>>>(p, p.sym_rows);
  return cudaGetLastError();
}

template <typename T> cudaError_t Path<T>::sym_probe(const Plan &p0, cudaStream_t st, double *columns) {
  Plan p = p0;
  p.prim = p.sym_order;
  int np_max = 0;
  sym_shape(p, p.sym_nj, np_max);
  // the middle orbitals: a column has the items of an energy's mean column, or half an item more
  p.sym_j0 = (p.n_occ - p.sym_nj + 1) / 2;
  *columns = (double)p.n_idx * p.sym_nj;
  long long launches = 0;
  const cudaError_t e = sym_pass<T>(p, np_max, st, nullptr, &launches);
  return e == cudaSuccess ? launch_xsym<T>(p, st) : e;
}

template <typename T>
cudaError_t Path<T>::sym_tau(const Plan &p0, double coef, cudaStream_t st, StageTimer *tm, long long *launches) {
  Plan p = p0;
  p.prim = p.sym_order;   // the slots of a pass: every G' of the index set, in its order
  const int no = p.n_occ;
  int nj, np_max;
  sym_shape(p, nj, np_max);
  cudaError_t e;
  for (p.sym_j0 = 0; p.sym_j0 < no; p.sym_j0 += nj) {
    p.sym_nj = std::min(nj, no - p.sym_j0);
    if ((e = sym_pass<T>(p, np_max, st, tm, launches)) != cudaSuccess) return e;
    ScopedStage s(tm, kStageColumn);
    if ((e = launch_xsym<T>(p, st)) != cudaSuccess) return e;
    // real orbitals: the rows are the primary G', each standing for -G' too
    k_xsym_sum<T><<<sym_pairs(p), 128, 0, st>>>(p, p.sym_rows, (p.real_orb ? 2.0 : 1.0) * coef);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    *launches += 2;
  }
  {
    ScopedStage s(tm, kStageDirect);
    const int t = (no + 3) / 4;
    k_dsym<T><<<dim3(p.n_groups, t * (t + 1) / 2), 256, 0, st>>>(p, p, true, p.sym_part);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    k_dsym_sum<T><<<(no * no + 3) / 4, 128, 0, st>>>(p, p, true, p.sym_part, (p.real_orb ? -4.0 : -2.0) * coef, p.ed,
                                                     p.edl);
    *launches += 2;
  }
  return cudaGetLastError();
}

template <typename T>
cudaError_t Path<T>::sym_cross(const Plan &pa, const Plan &pb, double coef, double *part, double *acc, cudaStream_t st) {
  k_dsym<T><<<dim3(pa.n_groups, ((pa.n_occ + 3) / 4) * ((pb.n_occ + 3) / 4)), 256, 0, st>>>(pa, pb, false, part);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  k_dsym_sum<T><<<(pa.n_occ * pb.n_occ + 3) / 4, 128, 0, st>>>(pa, pb, false, part, (pa.real_orb ? -2.0 : -1.0) * coef, acc,
                                                               nullptr);
  return cudaGetLastError();
}

template <typename T> cudaError_t Path<T>::green_k(const Plan &p, double tau, cudaStream_t st, StageTimer *tm) {
  ScopedStage s(tm, kStageGreen);
  k_dscale_k<T><<<dim3((p.n_orb + 255) / 256, p.nk), 256, 0, st>>>(p, p.eps, p.mu, tau, (T *)p.dscale);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  if (p.oz) {
    if ((e = oz_green<T>(*p.oz, p.cvt, (const T *)p.dscale + p.no_k, p.n_orb, p.n_v, p.pt, st)) != cudaSuccess) return e;
    return oz_split_b<T>(*p.oz, p.pt, st);
  }
  const size_t pw2 = (size_t)p.n_pw * p.n_pw;
  dim3 grid((p.n_pw + 63) / 64, (p.n_pw + 63) / 64);
  for (int k = 0; k < p.nk; ++k) {
    // P^T_k[q][p] = sum_a conj(c_{a k}(q)) e^{-(e_{a k}-mu)tau} c_{a k}(p)
    const cpx<T> *cv = (const cpx<T> *)p.cv + (size_t)k * p.n_v * p.n_pw;
    k_cgemm<T, false, true><<<grid, 256, 0, st>>>(p.n_pw, p.n_pw, p.n_v, cv, p.n_pw, cv, p.n_pw,
                                                  (const T *)p.dscale + (size_t)k * p.n_orb + p.no_k,
                                                  (cpx<T> *)p.pt + k * pw2, p.n_pw);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
  }
  return cudaSuccess;
}

template <typename T>
cudaError_t Path<T>::slab_k(const Plan &p, int gp0, int np, double coef, cudaStream_t st, StageTimer *tm) {
  const int n = p.n, NO = p.n_occ;
  const int nslots = 2 * np;
  const int ncols = nslots * NO;          // nk blocks of nslots * n_o columns, one block per kt
  const int rows_k = nslots * p.no_k;
  cudaError_t e;
  {
    ScopedStage s(tm, kStageGatherZ);
    k_gather_k<T><<<dim3((p.n_pw + 255) / 256, ncols), 256, 0, st>>>(p, gp0, np, (cpx<T> *)p.st);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
  }
  {
    ScopedStage s(tm, kStageWGemm);
    const size_t pw2 = (size_t)p.n_pw * p.n_pw;
    dim3 grid((p.n_pw + 63) / 64, (rows_k + 63) / 64);
    if (p.oz && (e = oz_wgemm<T>(*p.oz, p.st, rows_k, p.wt, st)) != cudaSuccess) return e;
    for (int kt = 0; kt < p.nk && !p.oz; ++kt) {
      const size_t row0 = (size_t)kt * rows_k * p.n_pw;
      k_cgemm<T, true, false><<<grid, 256, 0, st>>>(rows_k, p.n_pw, p.n_pw, (const cpx<T> *)p.st + row0, p.n_pw,
                                                    (const cpx<T> *)p.pt + kt * pw2, p.n_pw, nullptr,
                                                    (cpx<T> *)p.wt + row0, p.n_pw);
      if ((e = cudaGetLastError()) != cudaSuccess) return e;
    }
  }
  if constexpr (std::is_same<T, double>::value) {
    ScopedStage s(tm, kStageGatherZ);
    k_wnorm<<<ncols, 128, 0, st>>>(p, (const cpx<T> *)p.wt);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
  }
  const size_t smem_col = (size_t)p.n_aux * sizeof(cpx<T>);
  const int npairs = np * NO * NO;
  int col_threads = ((p.n_daux + 31) / 32) * 32;
  if (col_threads > 256) col_threads = 256;
  {
    ScopedStage s(tm, kStageGatherZ);
    if (!with_size(n, [&](auto c) { Sized<T, decltype(c)::value>::zinv(p, ncols, p.wt, p.z1, st); }))
      return cudaErrorInvalidValue;
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
  }
  {
    ScopedStage s(tm, kStagePlane);
    if ((e = launch_planes<T>(p, ncols, p.plane_kernel, p.plane_ib, st)) != cudaSuccess) return e;
  }
  {
    ScopedStage s(tm, kStageColumn);
    with_size(n, [&](auto c) { Sized<T, decltype(c)::value>::zcol_k(p, gp0, np, npairs, col_threads, smem_col, st); });
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
  }
  {
    ScopedStage s(tm, kStageDirect);
    const int t = (NO + 3) / 4;
    k_direct_k<T><<<np * t * t, 128, 0, st>>>(p, np, gp0, (const cpx<T> *)p.mdiag, p.yd);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
  }
  {
    ScopedStage s(tm, kStageAccum);
    k_accum_k<<<(NO * NO + 3) / 4, 128, 0, st>>>(p, gp0, np, coef, p.sx, p.yd);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
  }
  return cudaSuccess;
}

template <typename T> size_t Path<T>::plane_smem_for(const Plan &p, int ib) { return plane_smem<T>(p, 2, ib); }

template <typename T> cudaError_t Path<T>::persist_attributes() {
  cudaError_t e = PersistPlanes<T>::init();
  if (e == cudaSuccess) e = PersistColumns<T>::init();
  return e;
}

// resident blocks of the persistent kernel: every SM filled to its occupancy
template <typename T> int Path<T>::persist_blocks(bool planes, size_t smem) {
  int dev = 0, sms = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
    return 0;
  return sms * (planes ? PersistPlanes<T>::blocks_per_sm(smem) : PersistColumns<T>::blocks_per_sm(smem));
}

template <typename T>
cudaError_t Path<T>::planes_persist(const Plan *d_plans, const BatchRound &r, int *counter, int blocks, size_t smem,
                                    cudaStream_t st) {
  cudaError_t e = cudaMemsetAsync(counter, 0, sizeof(int), st);
  if (e != cudaSuccess) return e;
  PersistPlanes<T>::launch(d_plans, r, counter, blocks, smem, st);
  return cudaGetLastError();
}

template <typename T>
cudaError_t Path<T>::zcol_persist(const Plan *d_plans, const BatchRound &r, int *counter, int blocks, size_t smem,
                                  cudaStream_t st) {
  cudaError_t e = cudaMemsetAsync(counter, 0, sizeof(int), st);
  if (e != cudaSuccess) return e;
  PersistColumns<T>::launch(d_plans, r, counter, blocks, smem, st);
  return cudaGetLastError();
}

template <typename T>
cudaError_t Path<T>::descriptors(const Plan &p, double *moments, double *overlap, cudaStream_t st) {
  k_orb_moments<T><<<p.n_occ, 256, 0, st>>>(p, moments);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  k_pair_overlap<T><<<dim3(p.n_occ, p.n_occ), 256, 0, st>>>(p, overlap);
  return cudaGetLastError();
}

template <typename T>
cudaError_t Path<T>::direct_cross(const Plan &pa, const Plan &pb, int gp0, int np, double coef, double *y,
                                  double *acc, cudaStream_t st) {
  const int th = pb.n_occ < 128 ? ((pb.n_occ + 31) / 32) * 32 : 128;
  k_direct_cross<T><<<dim3(np, pa.n_occ), th, 0, st>>>(pa, pb, np, (const cpx<T> *)pa.mdiag,
                                                       (const cpx<T> *)pb.mdiag, y);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  k_accum_cross<<<(pa.n_occ * pb.n_occ + 127) / 128, 128, 0, st>>>(pa, pb.n_occ, gp0, np, coef, y, acc);
  return cudaGetLastError();
}

template <typename T> cudaError_t Path<T>::sum(int n, const double *x, double *out, cudaStream_t st) {
  k_sum<<<1, 256, 0, st>>>(n, x, out);
  return cudaGetLastError();
}

template <typename T> cudaError_t Path<T>::zero_acc(const Plan &p, cudaStream_t st) {
  k_zero_acc<<<(p.n_occ * p.n_occ + 255) / 256, 256, 0, st>>>(p);
  return cudaGetLastError();
}

template <typename T> cudaError_t Path<T>::finish(const Plan &p, cudaStream_t st, StageTimer *tm) {
  ScopedStage s(tm, kStageAccum);
  k_finish<<<1, 256, 0, st>>>(p);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess || p.n_lev < 2) return e;
  k_finish_lev<<<1, 256, 0, st>>>(p);
  return cudaGetLastError();
}

}  // namespace ltmp2
