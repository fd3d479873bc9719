// Host side of the exact-slice tensor-core products (gemm_f64tc.cuh): slice buffers and tensor
// maps of a context, the Green's function, the per-tau slices of it, the transformed states of a
// slab, and ltmp2_dgemm_nt (the same product on caller matrices).
#include <cuda.h>
#include <cuda_runtime.h>

#include <algorithm>

#include "../../include/ltmp2.h"
#include "fft.cuh"
#include "gemm_f64tc.cuh"
#include "once_device.h"
#include "plan.h"

namespace ltmp2 {

int tc_make_map_slices(CUtensorMap *m, void *base, int planes, int rows, int width, int box_rows);

namespace {

struct OzMaps {
  CUtensorMap a, b, bv, bt;
};

template <typename T> struct Num {
  static constexpr int S = sizeof(T) == 8 ? 8 : 4;
  typedef cpx<T> C;
};

int kpad_of(int k) { return ((k + oz::BK - 1) / oz::BK) * oz::BK; }
int rows128(int rows) { return ((rows + oz::BM - 1) / oz::BM) * oz::BM; }
int stacked_rows(int rows) { return 2 * (((rows + 63) / 64) * 64); }

template <typename T> cudaError_t attributes_of() {
  constexpr int S = Num<T>::S;
  cudaError_t e = cudaFuncSetAttribute(oz::k_dgemm_oz<S, true, T>, cudaFuncAttributeMaxDynamicSharedMemorySize, oz::Cfg<S>::SMEM);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(oz::k_dgemm_oz<S, false, T>, cudaFuncAttributeMaxDynamicSharedMemorySize, oz::Cfg<S>::SMEM);
  return e;
}

// of the current device: a function's attributes belong to one device
cudaError_t set_attributes() {
  static OncePerDevice once;
  int dev = 0;
  const cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  return once.run(dev, [] {
    const cudaError_t a = attributes_of<double>();
    return a == cudaSuccess ? attributes_of<float>() : a;
  });
}

// persistent blocks for `tiles` output tiles: one per SM
int oz_blocks(int tiles) {
  int dev = 0, n = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
    return tiles;
  return tiles < n ? tiles : n;
}

// C_z = A_z B_z^T over k values; arow: stacked (or plain) rows in use per product
template <typename T, bool STACKED>
cudaError_t launch_oz(const CUtensorMap &ta, const CUtensorMap &tb, int M, int N, int arow, int k, int arows, int brows,
                      const int *sa, const int *sb, void *C, int ldc, int *err, cudaStream_t st, int nz = 1, int za = 0,
                      int zb = 0, long long zc = 0) {
  constexpr int S = Num<T>::S, BN = oz::Cfg<S>::BN;
  oz::Product p;
  p.M = M;
  p.N = N;
  p.kblocks = kpad_of(k) / oz::BK;
  p.arows = arows;
  p.brows = brows;
  p.nbx = (N + BN - 1) / BN;
  p.nby = arow / oz::BM;
  p.nz = nz;
  p.za = za;
  p.zb = zb;
  p.zc = zc;
  p.ldc = ldc;
  oz::k_dgemm_oz<S, STACKED, T><<<oz_blocks(p.nbx * p.nby * nz), oz::THREADS, oz::Cfg<S>::SMEM, st>>>(
      ta, tb, p, sa, sb, static_cast<T *>(C), err);
  return cudaGetLastError();
}

int check_flag(int *err) {
  int flag = 0;
  if (cudaMemcpy(&flag, err, sizeof(int), cudaMemcpyDeviceToHost) != cudaSuccess) return LTMP2_ERR_CUDA;
  if (flag) {
    cudaMemset(err, 0, sizeof(int));
    return LTMP2_ERR_TIMEOUT;
  }
  return LTMP2_OK;
}

// rows of the A slices: a slab's states, or a Green's function
size_t a_rows(int rows_cap, int npw, int nz, bool cplx) {
  return (size_t)nz * std::max(stacked_rows(rows_cap), cplx ? stacked_rows(npw) : rows128(npw));
}
int k_pad(int npw, int nv, bool cplx) { return kpad_of((cplx ? 2 : 1) * std::max(npw, nv)); }

}  // namespace

size_t oz_bytes(int slices, int rows_cap, int npw, int nv, int nz, bool cplx) {
  const size_t rows = a_rows(rows_cap, npw, nz, cplx) + (size_t)nz * npw * 2 + (cplx ? 0 : (size_t)nv);
  return (sizeof(__half) * k_pad(npw, nv, cplx) * slices + sizeof(int)) * rows + 4096;
}

cudaError_t oz_init(OzResources &r, void *mem, int slices, int rows_cap, int npw, int nv, int nz, bool cplx) {
  cudaError_t e = set_attributes();
  if (e != cudaSuccess) return e;
  r.slices = slices;
  r.rows_cap = rows_cap;
  r.npw = npw;
  r.nv = nv;
  r.nz = nz;
  r.cplx = cplx;
  r.kpad = k_pad(npw, nv, cplx);
  r.arows = (int)a_rows(rows_cap, npw, nz, cplx);
  char *p = static_cast<char *>(mem);
  auto take = [&](size_t bytes) {
    char *q = p;
    p += (bytes + 255) / 256 * 256;
    return q;
  };
  const size_t row = sizeof(__half) * r.kpad * slices;
  const int brows = nz * npw, vrows = cplx ? 0 : nv;
  r.a = take(row * r.arows);
  r.b = take(row * brows);
  r.bt = take(row * brows);
  r.bv = take(row * vrows);
  r.sa = reinterpret_cast<int *>(take(sizeof(int) * r.arows));
  r.sb = reinterpret_cast<int *>(take(sizeof(int) * brows));
  r.sbt = reinterpret_cast<int *>(take(sizeof(int) * brows));
  r.sbv = reinterpret_cast<int *>(take(sizeof(int) * vrows));
  r.err = reinterpret_cast<int *>(take(sizeof(int)));
  if ((e = cudaMemset(r.err, 0, sizeof(int))) != cudaSuccess) return e;
  OzMaps *m = new OzMaps();
  const int bn = 512 / slices;
  if (tc_make_map_slices(&m->a, r.a, slices / 2, r.arows, 2 * r.kpad, oz::BM) ||
      tc_make_map_slices(&m->b, r.b, slices / 2, brows, 2 * r.kpad, bn) ||
      tc_make_map_slices(&m->bt, r.bt, slices / 2, brows, 2 * r.kpad, bn) ||
      (vrows > 0 && tc_make_map_slices(&m->bv, r.bv, slices / 2, vrows, 2 * r.kpad, bn))) {
    delete m;
    return cudaErrorInvalidValue;
  }
  r.maps = m;
  return cudaSuccess;
}

void oz_release(OzResources &r) {
  delete static_cast<OzMaps *>(r.maps);
  r.maps = nullptr;
}

namespace {
template <typename T>
cudaError_t split_rows(const OzResources &r, const T *x, int nrows, int k, int ld, const T *cscale, int prows, void *planes,
                       int *scale, int blocks, cudaStream_t st) {
  oz::k_oz_split_rows<Num<T>::S, T><<<blocks, 256, 0, st>>>(x, nrows, k, ld, cscale, kpad_of(k), r.kpad, prows,
                                                            static_cast<__half *>(planes), scale);
  return cudaGetLastError();
}
template <typename T>
cudaError_t split_stacked(const OzResources &r, const void *x, int rows, int k, int ld, const T *cscale, cudaStream_t st) {
  typedef typename Num<T>::C C;
  oz::k_oz_split_stacked<Num<T>::S, T, C><<<stacked_rows(rows) / 2, 256, 0, st>>>(
      static_cast<const C *>(x), rows, k, ld, cscale, kpad_of(k), r.kpad, r.arows, static_cast<__half *>(r.a), r.sa);
  return cudaGetLastError();
}
// complex operands of all nz products: stacked rows of A, or rows of B
template <typename T, bool STACKED>
cudaError_t split_cplx(const OzResources &r, const void *x, int rows, int k, int ld, long long zx, const T *cscale, int zscale,
                       bool conj, void *planes, int *scale, cudaStream_t st) {
  typedef typename Num<T>::C C;
  const int zrows = STACKED ? stacked_rows(rows) : rows;
  oz::k_oz_split_cplx<Num<T>::S, STACKED, T, C><<<dim3(STACKED ? zrows / 2 : rows, r.nz), 256, 0, st>>>(
      static_cast<const C *>(x), rows, k, ld, zx, cscale, zscale, conj, kpad_of(2 * k), r.kpad,
      STACKED ? r.arows : r.nz * r.npw, zrows, static_cast<__half *>(planes), scale);
  return cudaGetLastError();
}
}  // namespace

template <typename T> cudaError_t oz_set_virtuals(const OzResources &r, const void *cv, const void *cvt, cudaStream_t st) {
  if (r.nv < 1) return cudaSuccess;
  if (r.cplx)
    return split_cplx<T, false>(r, cvt, r.npw, r.nv, r.nv, (long long)r.npw * r.nv, nullptr, 0, false, r.bt, r.sbt, st);
  cudaError_t e = split_rows<T>(r, (const T *)cv, r.nv, r.npw, r.npw, nullptr, r.nv, r.bv, r.sbv, r.nv, st);
  if (e != cudaSuccess) return e;
  return split_rows<T>(r, (const T *)cvt, r.npw, r.nv, r.nv, nullptr, r.npw, r.bt, r.sbt, r.npw, st);
}

template <typename T>
cudaError_t oz_green(const OzResources &r, const void *cvt, const void *dv, int zscale, int nv, void *pr, cudaStream_t st) {
  if (!r.maps || nv < 1 || nv > r.nv) return cudaErrorInvalidValue;
  const OzMaps &m = *static_cast<const OzMaps *>(r.maps);
  cudaError_t e;
  if (r.cplx) {
    // A = conj(C_v')^T D' (rows q, columns a < nv), B = C_v'^T: P^T = A B^T
    e = split_cplx<T, true>(r, cvt, r.npw, nv, r.nv, (long long)r.npw * r.nv, (const T *)dv, zscale, true, r.a, r.sa, st);
    if (e != cudaSuccess) return e;
    return launch_oz<T, true>(m.a, m.bt, r.npw, r.npw, stacked_rows(r.npw), 2 * nv, r.arows, r.nz * r.npw, r.sa, r.sbt, pr,
                              r.npw, r.err, st, r.nz, stacked_rows(r.npw), r.npw, (long long)r.npw * r.npw);
  }
  // A = R_v'^T D', B = R_v'^T: P_r = A B^T
  e = split_rows<T>(r, (const T *)cvt, r.npw, nv, r.nv, (const T *)dv, r.arows, r.a, r.sa, rows128(r.npw), st);
  if (e != cudaSuccess) return e;
  return launch_oz<T, false>(m.a, m.bt, r.npw, r.npw, rows128(r.npw), nv, r.arows, r.npw, r.sa, r.sbt, pr, r.npw, r.err, st);
}

template <typename T>
cudaError_t oz_virtual(const OzResources &r, const void *st_in, int rows, const void *dv, int nv, void *x, void *wt,
                       cudaStream_t st) {
  if (rows > r.rows_cap || !r.maps || r.cplx || nv < 1 || nv > r.nv) return cudaErrorInvalidValue;
  const OzMaps &m = *static_cast<const OzMaps *>(r.maps);
  const int ar = stacked_rows(rows);
  // X^T = (U S)^T R_v'^T: A = the gathered states (K = n_pw), B = the first nv rows of R_v
  cudaError_t e = split_stacked<T>(r, st_in, rows, r.npw, r.npw, nullptr, st);
  if (e != cudaSuccess) return e;
  if ((e = launch_oz<T, true>(m.a, m.bv, rows, nv, ar, r.npw, r.arows, r.nv, r.sa, r.sbv, x, nv, r.err, st)) != cudaSuccess)
    return e;
  // W^T = (X^T D') R_v': A = X D' (K = nv), B = R_v^T (rows p, columns a < nv)
  if ((e = split_stacked<T>(r, x, rows, nv, nv, (const T *)dv, st)) != cudaSuccess) return e;
  return launch_oz<T, true>(m.a, m.bt, rows, r.npw, ar, nv, r.arows, r.npw, r.sa, r.sbt, wt, r.npw, r.err, st);
}

template <typename T> cudaError_t oz_split_b(const OzResources &r, const void *pr, cudaStream_t st) {
  if (r.cplx)   // P^T is Hermitian: row n of P is the conjugate of row n of P^T
    return split_cplx<T, false>(r, pr, r.npw, r.npw, r.npw, (long long)r.npw * r.npw, nullptr, 0, true, r.b, r.sb, st);
  return split_rows<T>(r, (const T *)pr, r.npw, r.npw, r.npw, nullptr, r.npw, r.b, r.sb, r.npw, st);
}

template <typename T> cudaError_t oz_wgemm(const OzResources &r, const void *st_in, int rows, void *wt, cudaStream_t st) {
  if (rows > r.rows_cap || !r.maps) return cudaErrorInvalidValue;
  const OzMaps &m = *static_cast<const OzMaps *>(r.maps);
  const int ar = stacked_rows(rows);
  cudaError_t e;
  if (r.cplx) {
    e = split_cplx<T, true>(r, st_in, rows, r.npw, r.npw, (long long)rows * r.npw, nullptr, 0, false, r.a, r.sa, st);
    if (e != cudaSuccess) return e;
    return launch_oz<T, true>(m.a, m.b, rows, r.npw, ar, 2 * r.npw, r.arows, r.nz * r.npw, r.sa, r.sb, wt, r.npw, r.err, st,
                              r.nz, ar, r.npw, (long long)rows * r.npw);
  }
  if ((e = split_stacked<T>(r, st_in, rows, r.npw, r.npw, nullptr, st)) != cudaSuccess) return e;
  return launch_oz<T, true>(m.a, m.b, rows, r.npw, ar, r.npw, r.arows, r.npw, r.sa, r.sb, wt, r.npw, r.err, st);
}

#define LTMP2_OZ_INSTANTIATE(T)                                                                                        \
  template cudaError_t oz_set_virtuals<T>(const OzResources &, const void *, const void *, cudaStream_t);              \
  template cudaError_t oz_green<T>(const OzResources &, const void *, const void *, int, int, void *, cudaStream_t);   \
  template cudaError_t oz_virtual<T>(const OzResources &, const void *, int, const void *, int, void *, void *,        \
                                     cudaStream_t);                                                                    \
  template cudaError_t oz_split_b<T>(const OzResources &, const void *, cudaStream_t);                                 \
  template cudaError_t oz_wgemm<T>(const OzResources &, const void *, int, void *, cudaStream_t);
LTMP2_OZ_INSTANTIATE(double)
LTMP2_OZ_INSTANTIATE(float)

int oz_check(const OzResources &r) { return check_flag(r.err); }

}  // namespace ltmp2

extern "C" int ltmp2_dgemm_nt(int m, int n, int k, const double *a, int lda, const double *b, int ldb, double *c,
                              int ldc) {
  using namespace ltmp2;
  if (m < 1 || n < 1 || k < 1 || !a || !b || !c || lda < k || ldb < k || ldc < n) return LTMP2_ERR_INVALID_ARG;
  cudaError_t e = set_attributes();
  if (e != cudaSuccess) return LTMP2_ERR_CUDA;
  constexpr int S = 8;
  const int kpad = kpad_of(k), ar = rows128(m);
  __half *pa = nullptr, *pb = nullptr;
  int *sa = nullptr, *sb = nullptr;
  int *err = nullptr;
  int rc = LTMP2_OK;
  auto cleanup = [&] {
    cudaFree(pa);
    cudaFree(pb);
    cudaFree(sa);
    cudaFree(sb);
    cudaFree(err);
  };
  if (cudaMalloc(&pa, sizeof(__half) * (size_t)S * ar * kpad) != cudaSuccess ||
      cudaMalloc(&pb, sizeof(__half) * (size_t)S * n * kpad) != cudaSuccess ||
      cudaMalloc(&sa, sizeof(int) * ar) != cudaSuccess || cudaMalloc(&sb, sizeof(int) * n) != cudaSuccess ||
      cudaMalloc(&err, sizeof(int)) != cudaSuccess) {
    cudaGetLastError();
    cleanup();
    return LTMP2_ERR_OOM;
  }
  OzMaps maps;
  if (tc_make_map_slices(&maps.a, pa, S / 2, ar, 2 * kpad, oz::BM) ||
      tc_make_map_slices(&maps.b, pb, S / 2, n, 2 * kpad, oz::Cfg<S>::BN)) {
    cleanup();
    return LTMP2_ERR_INVALID_ARG;
  }
  cudaMemset(err, 0, sizeof(int));
  oz::k_oz_split_rows<S, double><<<ar, 256>>>(a, m, k, lda, nullptr, kpad, kpad, ar, pa, sa);
  oz::k_oz_split_rows<S, double><<<n, 256>>>(b, n, k, ldb, nullptr, kpad, kpad, n, pb, sb);
  e = launch_oz<double, false>(maps.a, maps.b, m, n, ar, k, ar, n, sa, sb, c, ldc, err, nullptr);
  if (e == cudaSuccess) e = cudaDeviceSynchronize();
  if (e != cudaSuccess) rc = LTMP2_ERR_CUDA;
  if (!rc) rc = check_flag(err);
  cleanup();
  return rc;
}
