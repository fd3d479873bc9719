// Definitions of Sized<T, N> (sized.h); included by the translation units that instantiate it.
#pragma once
#include "kernels.cuh"
#include "sized.h"
#include "sym.cuh"

namespace ltmp2 {

template <typename T, int N> cudaError_t Sized<T, N>::init() {
  cudaError_t e = upload_twiddles_once();
  auto limit = [&](auto *k) {
    if (e == cudaSuccess) e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024);
  };
  if constexpr (std::is_same<T, float>::value) {
    limit(k_planes<T, N>);
    limit(k_planes2<T, N>);
    limit(k_planes4<T, N>);
  }
  limit(k_planes3<T, N>);
  limit(k_zcol<T, N, false>);
  limit(k_zcol<T, N, true>);
  limit(k_zcol_k<T, N>);
  limit(k_zsym<T, N>);
  return e;
}

template <typename T, int N> void Sized<T, N>::zinv(const Plan &p, int cols, const void *w, void *z1, cudaStream_t st) {
  k_w_zinv<T, N><<<dim3((p.n_dorb + 127) / 128, cols), 128, 0, st>>>(p, p.n_pw, (const cpx<T> *)w, (cpx<T> *)z1);
}

template <typename T, int N> void Sized<T, N>::planes_store(const Plan &p, const void *z1, cudaStream_t st) {
  const size_t smem = (size_t)N * (N + 1) * sizeof(cpx<T>);
  k_planes_store<T, N><<<dim3(N, p.n_occ), 128, smem, st>>>(p, (const cpx<T> *)z1, (cpx<T> *)p.u, p.ut, p.utr);
}

template <typename T, int N>
void Sized<T, N>::planes(const Plan &p, int cols, int kernel, int ib, int threads, size_t smem, cudaStream_t st) {
  const dim3 grid(N, cols);
  if constexpr (std::is_same<T, float>::value) {
    const cpx<T> *z1 = (const cpx<T> *)p.z1;
    cpx<T> *tbuf = (cpx<T> *)p.tbuf;
    if (kernel == 0) k_planes<T, N><<<grid, threads, smem, st>>>(p, ib, z1, tbuf);
    else if (kernel == 1) k_planes2<T, N><<<grid, threads, smem, st>>>(p, ib, z1, tbuf);
    else if (kernel == 3) k_planes4<T, N><<<grid, threads, smem, st>>>(p, ib, z1, tbuf);
  }
  if (kernel == 2) {
    const int cps = cols_per_slot(p), cols2 = std::is_same<T, double>::value ? cols : (cols / cps + 1) / 2 * cps;
    k_planes3<T, N><<<dim3(N, cols2), threads, smem, st>>>(p, ib, cols, p.z1, p.tbuf);
  }
}

template <typename T, int N>
void Sized<T, N>::zcol(const Plan &p, int gp0, int np, int npairs, int threads, size_t smem, bool lev, cudaStream_t st) {
  if (lev) k_zcol<T, N, true><<<npairs, threads, smem, st>>>(p, gp0, np, p.tbuf, (cpx<T> *)p.mdiag, p.sx);
  else k_zcol<T, N, false><<<npairs, threads, smem, st>>>(p, gp0, np, p.tbuf, (cpx<T> *)p.mdiag, p.sx);
}

template <typename T, int N>
void Sized<T, N>::zsym(const Plan &p, int gp0, int cols, int threads, size_t smem, cudaStream_t st) {
  k_zsym<T, N><<<dim3(p.sym_j0 + p.sym_nj, cols), threads, smem, st>>>(p, gp0);
}

template <typename T, int N>
void Sized<T, N>::zcol_k(const Plan &p, int gp0, int np, int npairs, int threads, size_t smem, cudaStream_t st) {
  k_zcol_k<T, N><<<npairs, threads, smem, st>>>(p, gp0, np, p.tbuf, (cpx<T> *)p.mdiag, p.sx);
}

}  // namespace ltmp2
