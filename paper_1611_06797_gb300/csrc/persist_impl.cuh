// Persistent kernels of the batching form (sized.h declares their launchers); the translation
// units define LTMP2_PERSIST_PLANES or LTMP2_PERSIST_COLUMNS and instantiate one of them.
#pragma once
#include "kernels.cuh"
#include "sized.h"

namespace ltmp2 {

// ---------------------------------------------------------------- batching form: persistent stages
// Thread blocks of kPersistThreads stay resident and take items from a device counter:
// plane items (system, column, z) and column items (system, pair) of every active system of
// the round, each run by the same body as the system's own kernel (dispatch on its grid).
#ifdef LTMP2_PERSIST_PLANES
template <typename T>
__global__ void __launch_bounds__(kPersistThreads) k_planes_persist(const Plan *__restrict__ plans, BatchRound r,
                                                                     int *__restrict__ counter) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ int s_item;
  // the round's tables in shared memory: indexed by the item's system, which a kernel
  // parameter array would have to copy to local memory for
  __shared__ BatchRound sr;
  if (threadIdx.x == 0) sr = r;
  const int total = r.first[r.nsys];
  for (;;) {
    __syncthreads();
    if (threadIdx.x == 0) s_item = atomicAdd(counter, 1);
    __syncthreads();
    const int item = s_item;
    if (item >= total) return;
    int e = 0;
    while (item >= sr.first[e + 1]) ++e;
    const Plan &p = plans[sr.sys[e]];
    const int local = item - sr.first[e];
    const int z = local % p.n, col = local / p.n;
    switch (p.n) {
#define LTMP2_CASE(NN)                                                                                        \
  case NN:                                                                                                    \
    planes3_any<T, NN>(p, sr.ib[e], z, col, (sr.first[e + 1] - sr.first[e]) / NN, p.z1, p.tbuf, smem_raw);   \
    break;
      LTMP2_FOR_EACH_N(LTMP2_CASE)
#undef LTMP2_CASE
      default:
        break;
    }
  }
}

template <typename T> cudaError_t PersistPlanes<T>::init() {
  const cudaError_t e = upload_twiddles_once();
  return e == cudaSuccess ? cudaFuncSetAttribute(k_planes_persist<T>, cudaFuncAttributeMaxDynamicSharedMemorySize, kPersistSmem) : e;
}
template <typename T> int PersistPlanes<T>::blocks_per_sm(size_t smem) {
  int per = 0;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, k_planes_persist<T>, kPersistThreads, smem) != cudaSuccess) return 0;
  return per > 0 ? per : 1;
}
template <typename T>
void PersistPlanes<T>::launch(const Plan *d_plans, const BatchRound &r, int *counter, int blocks, size_t smem, cudaStream_t st) {
  k_planes_persist<T><<<blocks, kPersistThreads, smem, st>>>(d_plans, r, counter);
}
#endif

#ifdef LTMP2_PERSIST_COLUMNS
template <typename T>
__global__ void __launch_bounds__(kPersistThreads) k_zcol_persist(const Plan *__restrict__ plans, BatchRound r,
                                                                   int *__restrict__ counter) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ int s_item;
  // the round's tables in shared memory: indexed by the item's system, which a kernel
  // parameter array would have to copy to local memory for
  __shared__ BatchRound sr;
  if (threadIdx.x == 0) sr = r;
  const int total = r.first[r.nsys];
  for (;;) {
    __syncthreads();
    if (threadIdx.x == 0) s_item = atomicAdd(counter, 1);
    __syncthreads();
    const int item = s_item;
    if (item >= total) return;
    int e = 0;
    while (item >= sr.first[e + 1]) ++e;
    const Plan &p = plans[sr.sys[e]];
    const int local = item - sr.first[e];
    switch (p.n) {
#define LTMP2_CASE(NN)                                                                                        \
  case NN:                                                                                                    \
    zcol_body<T, NN, false>(p, sr.gp0[e], sr.np[e], local, p.tbuf, (cpx<T> *)p.mdiag, p.sx,                   \
                            smem_raw);                                                                        \
    break;
      LTMP2_FOR_EACH_N(LTMP2_CASE)
#undef LTMP2_CASE
      default:
        break;
    }
  }
}

template <typename T> cudaError_t PersistColumns<T>::init() {
  const cudaError_t e = upload_twiddles_once();
  return e == cudaSuccess ? cudaFuncSetAttribute(k_zcol_persist<T>, cudaFuncAttributeMaxDynamicSharedMemorySize, kPersistSmem) : e;
}
template <typename T> int PersistColumns<T>::blocks_per_sm(size_t smem) {
  int per = 0;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, k_zcol_persist<T>, kPersistThreads, smem) != cudaSuccess) return 0;
  return per > 0 ? per : 1;
}
template <typename T>
void PersistColumns<T>::launch(const Plan *d_plans, const BatchRound &r, int *counter, int blocks, size_t smem, cudaStream_t st) {
  k_zcol_persist<T><<<blocks, kPersistThreads, smem, st>>>(d_plans, r, counter);
}
#endif

}  // namespace ltmp2
