// Launchers of the kernels that are compiled once per grid size N (line FFTs of N points in
// registers), and of the persistent kernels that hold every size.  Declared here, defined in
// sized_impl.cuh / persist_impl.cuh and instantiated in several translation units, which
// compile in parallel.
#pragma once
#include <cuda_runtime.h>

#include "plan.h"

namespace ltmp2 {

#define LTMP2_FOR_EACH_N(X) X(8) X(10) X(12) X(16) X(18) X(20) X(24) X(25) X(27) X(30) X(32) X(36) X(40)

template <typename T, int N> struct Sized {
  // this translation unit's twiddle tables and the kernels' shared-memory limits, once per device
  static cudaError_t init();
  // inverse z transform of `cols` rows of plane-wave coefficients, z1 of a slab
  static void zinv(const Plan &p, int cols, const void *w, void *z1, cudaStream_t st);
  static void planes_store(const Plan &p, const void *z1, cudaStream_t st);
  static void planes(const Plan &p, int cols, int kernel, int ib, int threads, size_t smem, cudaStream_t st);
  static void zcol(const Plan &p, int gp0, int np, int npairs, int threads, size_t smem, bool lev, cudaStream_t st);
  static void zsym(const Plan &p, int gp0, int cols, int threads, size_t smem, cudaStream_t st);
  static void zcol_k(const Plan &p, int gp0, int np, int npairs, int threads, size_t smem, cudaStream_t st);
};

// persistent kernels of the batching form: twiddle tables and shared-memory limit, blocks per SM, launch.
// The limit is the same for every batch: several threads may create batches of different sizes.
template <typename T> struct PersistPlanes {
  static cudaError_t init();
  static int blocks_per_sm(size_t smem);
  static void launch(const Plan *d_plans, const BatchRound &r, int *counter, int blocks, size_t smem, cudaStream_t st);
};
template <typename T> struct PersistColumns {
  static cudaError_t init();
  static int blocks_per_sm(size_t smem);
  static void launch(const Plan *d_plans, const BatchRound &r, int *counter, int blocks, size_t smem, cudaStream_t st);
};

}  // namespace ltmp2
