// Products of FP64 or FP32 accuracy on the tcgen05 tensor cores (the Green's function and the
// transformed states of step (iii), Sec. III A), by exact integer slices (Ozaki's scheme):
//
//   each row of A and of B (C = A B^T, both K-major) is scaled by a power of two 2^e with
//   |x| < 2^e over the row and cut into S slices of 7 bits (8 for FP64, 4 for FP32),
//       a = 2^e_a sum_s d_s 2^{-7(s+1)},  d_s integers, |d_0| <= 128, |d_s| <= 64 (s >= 1),
//   every slice exactly representable in FP16.  Then
//       (A B^T)_ij = 2^{e_i + f_j} sum_{d=0}^{S-1} 2^{-7(d+2)} sum_{s+t=d} sum_k a_{s,ik} b_{t,jk}
//   with the pairs s + t >= S left out (per term at most 7 x 2^12 x 2^-70 x 2^{e_a + e_b}
//   <= 7 x 2^-56 max|a| max|b|, at the rounding of an FP64 product).  Each inner sum is a
//   sum of integer products; over 384 k it stays below 2^24 in magnitude (at most
//   2 x 128 x 64 + 6 x 64 x 64 = 2.5 x 2^14 per k for one order d), so every partial sum is an
//   integer that FP32 holds exactly and the tensor core's accumulation is exact, whatever its
//   rounding.  The accumulators of the 8 orders d live in tensor memory (8 x 64 columns = all
//   512) and are drained every 384 k into 64-bit integer register sums.  The only roundings
//   are those of the slicing and of the final conversion.
//
// What bounds it: 36 slice products per product (10 with 4 slices).  FP16 operands run at twice
// the TF32 rate and half the bytes of the same integers.  Slice s of A multiplies the slices
// t < S - s of B in MMAs of up to 256 columns: four (two) B slices lie one after another in shared
// memory and so do the orders s + t in tensor memory, so 12 instructions replace 36 and A is read
// from shared memory once per 256 columns instead of once per 64.  The drain runs on integers
// because the FP64 pipe (2 operations per clock and SM) needs 69,000 clocks per 128 x 64 tile and
// window (a conversion and an FMA for each of 8 orders) where the window's products take 27,600 at
// the nominal rate; 8 float-to-integer conversions an element take 4,100.  One persistent block per SM: the next tile's products run while a tile is written.
// 4501 x 3071 x 3039 on GB300: 12.9 ms with TF32 slices and FP64 drains, 4.0 ms with the above, 2.75
// ms with single-block stages, a producer thread of its own and waits that poll before they read
// the clock (1.6 ms is what the slice products take at the measured FP16 rate); the kernel itself
// takes 1.9 of the 2.75 ms, the tensor pipe active 67 % of them.
//
// Against FP64 (FP32) products: an entry below 2^-3 (2^-4) of its row's maximum keeps fewer bits than its
// own 53 (24), and the dropped orders are relative to the two rows' maxima; the sums, in return, are exact.
#pragma once
#include <cuda.h>
#include <cuda_fp16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "tcgen05.cuh"

namespace ltmp2 {
namespace oz {

constexpr int BITS = 7;                      // bits per slice
constexpr int BM = 128;                      // rows of A per tile (tensor-memory lanes)
constexpr int BK = 16;                       // k per block: one MMA deep
constexpr int A_TILE = BM * 64;              // bytes of one plane of an A tile (64-byte swizzle rows)
constexpr int TMEM_COLS = 512;               // one accumulator per slice order d = s + t: all of it
constexpr int EPI_WARPS = 8;
constexpr int THREADS = 32 * (EPI_WARPS + 2);
constexpr int EPI_COLS = 32;                 // columns staged per output round
constexpr int EPI_BYTES = BM * (EPI_COLS + 1) * (int)sizeof(double);
constexpr int GROUP_ROWS = 12;               // row tiles that run side by side (12 x 12 tiles share operands in L2)

// S slices per operand: 8 for FP64 (56 bits below the row's maximum), 4 for FP32 (28 bits).
// Two slices share a plane: plane p holds slices p and p + S / 2, 16 k of the one, then 16 k of
// the other, so that a 64-byte row of shared memory is one k block of both.  A stage is then a
// single k block (48 KB / 32 KB) and four / six of them are in flight; with one slice per row
// a stage held two k blocks and two stages left the loads 1.1 us to arrive, which they missed
// (tensor pipe 42 % active).
template <int S> struct Cfg {
  static constexpr int P = S / 2;                      // planes
  static constexpr int BN = 512 / S;                   // rows of B per tile (accumulator columns per order)
  static constexpr int B_TILE = BN * 64;
  static constexpr int STAGE = P * (A_TILE + B_TILE);
  static constexpr int STAGES = S == 8 ? 4 : 6;
  static constexpr int SMEM = STAGES * STAGE + EPI_BYTES + 1024;  // + alignment slack
  // k blocks between drains: order S - 1 grows by at most 2 x 128 x 64 + (S - 2) x 64 x 64 per k
  static constexpr int DRAIN_KB = S == 8 ? 24 : 40;    // 384 / 640 k
  static_assert((2 * 128 * 64 + (S - 2) * 64 * 64) * DRAIN_KB * BK < (1 << 24), "order sums exact in FP32");
  static_assert(P * BN == 256, "P slices of B per MMA");
};
// element (row, k) of slice s, rows of a plane `prows`, padded K `kpad`
template <int S> __device__ __forceinline__ size_t slice_at(int s, size_t row, int k, size_t prows, int kpad) {
  constexpr int P = S / 2;
  return ((size_t)(s % P) * prows + row) * (2 * (size_t)kpad) + (k / BK) * (2 * BK) + (s / P) * BK + k % BK;
}
// instruction descriptor: D fp32, A and B fp16, both K-major, M = 128, N columns
__host__ __device__ constexpr uint32_t idesc(int n) {
  return (1u << 4) | ((uint32_t)(n >> 3) << 17) | ((uint32_t)(BM >> 4) << 24);
}

// Magnitudes are compared as the integers of their bits (the FP64 pipe is the slowest of the
// SM): the same order for finite values, with infinities and NaN above them.
typedef unsigned long long Bits;
__device__ __forceinline__ Bits magnitude(double x) { return (Bits)__double_as_longlong(x) & 0x7fffffffffffffffull; }
constexpr Bits kInfBits = 0x7ff0000000000000ull;
// a float's bits with the exponent rebiased (a denormal counts as up to 2^-126)
__device__ __forceinline__ Bits magnitude(float x) {
  const unsigned b = (unsigned)__float_as_int(x) & 0x7fffffffu;
  return b == 0 ? 0 : b >= 0x7f800000u ? kInfBits : ((Bits)b << 29) + ((Bits)(1023 - 127) << 52);
}
// the smallest e with |x| < 2^e for every |x| <= m (0 for m = 0 and for rows that are not finite)
__device__ __forceinline__ int row_exponent(Bits m) {
  return m > 0 && m < kInfBits ? ilogb(__longlong_as_double((long long)m)) + 1 : 0;
}
// the exponent kept for a row: its products are NaN if it holds a NaN or an infinity
constexpr int kNotFinite = 1 << 20;
__device__ __forceinline__ int stored_exponent(Bits m, int e) { return m < kInfBits ? e : kNotFinite; }

// v 2^e on the exponent bits; results out of the normal range, and rows that are not finite, take ldexp
__device__ __forceinline__ double times_pow2(double v, int e) {
  const long long b = __double_as_longlong(v);
  const int x = (int)((b >> 52) & 0x7ff) + e;
  if (x > 0 && x < 2047 && (b << 1) != 0) return __longlong_as_double(b + ((long long)e << 52));
  return e >= kNotFinite / 2 ? __longlong_as_double(0x7ff8000000000000ll) : ldexp(v, e);
}
__device__ __forceinline__ float times_pow2(float v, int e) {
  const int b = __float_as_int(v);
  const int x = ((b >> 23) & 0xff) + e;
  if (x > 0 && x < 255 && (b << 1) != 0) return __int_as_float(b + (e << 23));
  return e >= kNotFinite / 2 ? __int_as_float(0x7fc00000) : ldexpf(v, e);
}

// times 2^s, in two factors for rows of denormal numbers (one alone would overflow)
template <typename T> struct RowScale {
  T f1, f2;
  bool two;
  __device__ __forceinline__ explicit RowScale(int s) {
    const int lim = sizeof(T) == 8 ? 1000 : 120;
    const int a = min(max(s, -lim), lim);
    f1 = (T)ldexp(1.0, a);
    f2 = (T)ldexp(1.0, s - a);
    two = s != a;
  }
  __device__ __forceinline__ T operator()(T x) const {
    x *= f1;
    return two ? x * f2 : x;
  }
};

// x 2^(7 S - e) rounded to an integer, |x| < 2^e, as S balanced digits of 7 bits, top digit first:
// x = 2^e sum_s d_s 2^{-7(s+1)} + r, |r| <= 2^{e - 7 S - 1}; |d_0| <= 128, -64 <= d_s < 64 after
template <int S, typename T> __device__ __forceinline__ void slice(T x, const RowScale<T> &f, int (&d)[S]) {
  if constexpr (S == 8) {
    long long v = __double2ll_rn((double)f(x));
#pragma unroll
    for (int s = S - 1; s > 0; --s) {
      const int lo = (((int)v + 64) & 127) - 64;
      d[s] = lo;
      v = (v - lo) >> BITS;
    }
    d[0] = (int)v;
  } else {
    int v = __float2int_rn((float)f(x));   // at most 2^28
#pragma unroll
    for (int s = S - 1; s > 0; --s) {
      const int lo = ((v + 64) & 127) - 64;
      d[s] = lo;
      v = (v - lo) >> BITS;
    }
    d[0] = v;
  }
}
__device__ __forceinline__ __half2 pair16(int a, int b) { return __halves2half2(__int2half_rn(a), __int2half_rn(b)); }

// block-wide max of v over blockDim.x threads (blockDim.x a multiple of 32, <= 1024)
__device__ __forceinline__ Bits block_max(Bits v) {
  __shared__ Bits red[32];
  for (int o = 16; o > 0; o >>= 1) v = max(v, __shfl_xor_sync(0xffffffffu, v, o));
  const int w = threadIdx.x / 32, nw = blockDim.x / 32;
  __syncthreads();
  if (threadIdx.x % 32 == 0) red[w] = v;
  __syncthreads();
  Bits m = 0;
  for (int i = 0; i < nw; ++i) m = max(m, red[i]);
  return m;
}

// Slices of the rows of a real matrix X [nrows][ld], columns q < k, each times cscale[q]
// when cscale is not null: slice s at slice_at(s, r, q) for q < kfill (zero past k);
// scale[r] = e_r.  One block per row r < prows.  kfill is even.
template <int S, typename T>
__global__ void k_oz_split_rows(const T *__restrict__ x, int nrows, int k, int ld, const T *__restrict__ cscale,
                                int kfill, int kpad, int prows, __half *__restrict__ planes, int *__restrict__ scale) {
  const int r = blockIdx.x;
  const T *row = x + (size_t)r * ld;
  auto at = [&](int q) { return r < nrows && q < k ? (cscale ? row[q] * cscale[q] : row[q]) : T(0); };
  Bits m = 0;
  for (int q = threadIdx.x; q < k; q += blockDim.x) m = max(m, magnitude(at(q)));
  m = block_max(m);
  const int e = row_exponent(m);
  if (threadIdx.x == 0) scale[r] = stored_exponent(m, e);
  const RowScale<T> f(S * BITS - e);
  for (int q = 2 * threadIdx.x; q < kfill; q += 2 * blockDim.x) {
    int d0[S], d1[S];
    slice<S>(at(q), f, d0);
    slice<S>(at(q + 1), f, d1);
#pragma unroll
    for (int s = 0; s < S; ++s)
      *reinterpret_cast<__half2 *>(planes + slice_at<S>(s, r, q, prows, kpad)) = pair16(d0[s], d1[s]);
  }
}

// Slices of the stacked rows of a complex matrix X [rows][ld] (columns q < k, each times
// cscale[q] when cscale is not null): complex row m gives stacked row 128 (m / 64) + m % 64 (its
// real part) and that + 64 (its imaginary part), each with its own scale, for q < kfill.  One
// block per complex row m (rows past `rows` are zero).
template <int S, typename T, typename T2>
__global__ void k_oz_split_stacked(const T2 *__restrict__ x, int rows, int k, int ld, const T *__restrict__ cscale,
                                   int kfill, int kpad, int prows, __half *__restrict__ planes,
                                   int *__restrict__ scale) {
  const int m = blockIdx.x;
  const size_t r1 = (size_t)128 * (m / 64) + (m % 64), r2 = r1 + 64;
  const T2 *row = x + (size_t)m * ld;
  auto at = [&](int q) {
    T2 v{T(0), T(0)};
    if (m < rows && q < k) {
      v = row[q];
      if (cscale) {
        v.x *= cscale[q];
        v.y *= cscale[q];
      }
    }
    return v;
  };
  Bits mr = 0, mi = 0;
  for (int q = threadIdx.x; q < k; q += blockDim.x) {
    const T2 v = at(q);
    mr = max(mr, magnitude(v.x));
    mi = max(mi, magnitude(v.y));
  }
  mr = block_max(mr);
  mi = block_max(mi);
  const int er = row_exponent(mr), ei = row_exponent(mi);
  if (threadIdx.x == 0) {
    scale[r1] = stored_exponent(mr, er);
    scale[r2] = stored_exponent(mi, ei);
  }
  const RowScale<T> fr(S * BITS - er), fi(S * BITS - ei);
  for (int q = 2 * threadIdx.x; q < kfill; q += 2 * blockDim.x) {
    const T2 v0 = at(q), v1 = at(q + 1);
    int a0[S], a1[S];
    slice<S>(v0.x, fr, a0);
    slice<S>(v1.x, fr, a1);
#pragma unroll
    for (int s = 0; s < S; ++s)
      *reinterpret_cast<__half2 *>(planes + slice_at<S>(s, r1, q, prows, kpad)) = pair16(a0[s], a1[s]);
    slice<S>(v0.y, fi, a0);
    slice<S>(v1.y, fi, a1);
#pragma unroll
    for (int s = 0; s < S; ++s)
      *reinterpret_cast<__half2 *>(planes + slice_at<S>(s, r2, q, prows, kpad)) = pair16(a0[s], a1[s]);
  }
}

// General (complex) orbitals: C = X Y^T with X [rows][k] and Y [N][k] complex, over 2 k interleaved
// real products: (Re C | Im C) = ((Re X, -Im X) | (Im X, Re X)) (Re Y, Im Y)^T.
// X form (STACKED): complex row m gives the stacked rows of its real and imaginary part.
// Y form: row r, one row.  conj: of X / Y.  blockIdx.y: one of gridDim.y matrices, zx elements
// apart in x, zscale in cscale, zrows in the slices' rows.
template <int S, bool STACKED, typename T, typename T2>
__global__ void k_oz_split_cplx(const T2 *__restrict__ x, int rows, int k, int ld, long long zx,
                                const T *__restrict__ cscale, int zscale, bool conj, int kfill, int kpad, int prows,
                                int zrows, __half *__restrict__ planes, int *__restrict__ scale) {
  const int m = blockIdx.x, z = blockIdx.y;
  const size_t base = (size_t)z * zrows;
  const size_t r1 = STACKED ? base + (size_t)128 * (m / 64) + (m % 64) : base + m, r2 = r1 + 64;
  const T2 *row = x + z * zx + (size_t)m * ld;
  const T *cs = cscale ? cscale + (size_t)z * zscale : nullptr;
  auto at = [&](int q) {
    T2 v{T(0), T(0)};
    if (m < rows && q < k) {
      v = row[q];
      if (cs) {
        v.x *= cs[q];
        v.y *= cs[q];
      }
      if (conj) v.y = -v.y;
    }
    return v;
  };
  Bits mx = 0;
  for (int q = threadIdx.x; q < k; q += blockDim.x) {
    const T2 v = at(q);
    mx = max(mx, max(magnitude(v.x), magnitude(v.y)));
  }
  mx = block_max(mx);
  const int e = row_exponent(mx);
  if (threadIdx.x == 0) {
    scale[r1] = stored_exponent(mx, e);
    if (STACKED) scale[r2] = scale[r1];
  }
  const RowScale<T> f(S * BITS - e);
  for (int q = threadIdx.x; 2 * q < kfill; q += blockDim.x) {
    const T2 v = at(q);
    int re[S], im[S];
    slice<S>(v.x, f, re);
    slice<S>(v.y, f, im);
#pragma unroll
    for (int s = 0; s < S; ++s) {
      *reinterpret_cast<__half2 *>(planes + slice_at<S>(s, r1, 2 * q, prows, kpad)) =
          pair16(re[s], STACKED ? -im[s] : im[s]);
      if (STACKED) *reinterpret_cast<__half2 *>(planes + slice_at<S>(s, r2, 2 * q, prows, kpad)) = pair16(im[s], re[s]);
    }
  }
}

// 8 consecutive fp32 accumulator columns of this thread's tensor-memory lane, not yet waited for
__device__ __forceinline__ void tmem_ld8(uint32_t taddr, uint32_t (&r)[8]) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
               : "r"(taddr));
}

// true in every thread of the 8 epilogue warps if it is true in all of them
__device__ __forceinline__ bool epilogue_all(bool v) {
  uint32_t r;
  asm volatile(
      "{\n .reg .pred p, q;\n setp.ne.u32 p, %1, 0;\n bar.red.and.pred q, 1, 256, p;\n selp.u32 %0, 1, 0, q;\n}"
      : "=r"(r)
      : "r"(v ? 1u : 0u)
      : "memory");
  return r != 0;
}

// What one launch computes: C_z = A_z B_z^T for z < nz, from slices of arows / brows rows per slice
struct Product {
  int M, N;                // rows of C (complex rows if stacked) and columns
  int kblocks;
  int arows, brows;        // rows per slice plane
  int nbx, nby, nz;        // column tiles, row tiles, products
  int za, zb;              // rows between the products' operands
  long long zc;            // elements of C between them (complex ones if stacked)
  int ldc;
};

// C = A B^T from the slices.  Persistent: block b takes tiles b, b + gridDim.x, ... of the
// nz x nbx x nby tiles (BN columns x 128 stacked rows).  One thread of warp 9 issues the TMA copies,
// one of warp 8 the MMAs; warps 0-7 drain the accumulators every DRAIN_KB k blocks (warp w: lanes
// 32 (w % 4) on, the first or second half of the columns) and write the tile.
// STACKED: A rows are stacked real / imaginary rows and C is complex [M][ldc] (M complex rows);
// else C is real [M][ldc].  Every wait is bounded: on expiry the block raises *err, waits
// (bounded) for its own copies, writes nothing more, frees its tensor memory and returns.
template <int S, bool STACKED, typename T>
__global__ void __launch_bounds__(THREADS, 1)
    k_dgemm_oz(const __grid_constant__ CUtensorMap ta, const __grid_constant__ CUtensorMap tb, const Product pr,
               const int *__restrict__ sa, const int *__restrict__ sb, T *__restrict__ C, int *__restrict__ err) {
  using namespace tc;
  typedef Cfg<S> F;
  constexpr int BN = F::BN, STAGES = F::STAGES;
  extern __shared__ unsigned char smem_raw[];
  __shared__ uint64_t full_bar[STAGES], empty_bar[STAGES], accf_bar, acce_bar, done_bar;
  __shared__ uint32_t tmem_slot;
  __shared__ int row_exp[BM];
  unsigned char *smem = reinterpret_cast<unsigned char *>(
      (reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~static_cast<uintptr_t>(1023));
  const int warp = threadIdx.x / 32, lane = threadIdx.x % 32;
  const int per_z = pr.nbx * pr.nby, ntiles = per_z * pr.nz, kblocks = pr.kblocks;
  // tile -> (z, bx, by): groups of GROUP_ROWS row tiles, rows fastest within a group
  auto tile_at = [&](int t, int &bz, int &bx, int &by) {
    bz = t / per_z;
    t -= bz * per_z;
    const int per = GROUP_ROWS * pr.nbx, g = t / per, r = t - g * per;
    const int rows = min(GROUP_ROWS, pr.nby - g * GROUP_ROWS);
    by = g * GROUP_ROWS + r % rows;
    bx = r / rows;
  };
  const int nwin = (kblocks + F::DRAIN_KB - 1) / F::DRAIN_KB;

  if (warp == 0) tmem_alloc(&tmem_slot, TMEM_COLS);
  if (threadIdx.x == 0) {
    for (int s = 0; s < STAGES; ++s) {
      mbar_init(&full_bar[s], 1);
      mbar_init(&empty_bar[s], 1);
    }
    mbar_init(&accf_bar, 1);
    mbar_init(&acce_bar, 32 * EPI_WARPS);
    mbar_init(&done_bar, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  fence_before();
  __syncthreads();
  fence_after();
  const uint32_t tmem = tmem_slot;
  bool ok = true;

  // k blocks are counted over all tiles of this block: block kb of tile i is i kblocks + kb
  const int mine = (int)blockIdx.x < ntiles ? (ntiles - (int)blockIdx.x + (int)gridDim.x - 1) / (int)gridDim.x : 0;
  const int total = mine * kblocks;
  if (warp == EPI_WARPS + 1) {
    if (lane == 0) {   // TMA producer
      int g = 0;
      for (int tile = blockIdx.x; tile < ntiles && ok; tile += gridDim.x) {
        int bz, bx, by;
        tile_at(tile, bz, bx, by);
        const int arow0 = bz * pr.za + by * BM, brow0 = bz * pr.zb + bx * BN;
        for (int kb = 0; kb < kblocks; ++kb, ++g) {
          const int st = g % STAGES;
          // the stage is free once the MMAs of k block g - STAGES are done
          if (g >= STAGES && !mbar_wait(&empty_bar[st], (uint32_t)((g / STAGES - 1) & 1))) { ok = false; break; }
          unsigned char *p = smem + st * F::STAGE;
          mbar_expect_tx(&full_bar[st], F::STAGE);
          tma_load_3d(p, &ta, &full_bar[st], kb * 2 * BK, arow0, 0);                      // P planes of 128 rows
          tma_load_3d(p + F::P * A_TILE, &tb, &full_bar[st], kb * 2 * BK, brow0, 0);      // P planes of BN rows
        }
      }
      if (!ok) atomicExch(err, 1);
      // its own copies land before the block leaves, also when the MMAs gave up on them
      drain_issued<STAGES>(full_bar, max(0, g - STAGES), g);
    }
  } else if (warp == EPI_WARPS) {
    if (lane == 0) {   // MMA issuer
      int win = 0, kb = 0;
      for (int g = 0; g < total; ++g) {
        const int st = g % STAGES;
        const bool first = kb % F::DRAIN_KB == 0;
        if (!mbar_wait(&full_bar[st], (uint32_t)((g / STAGES) & 1))) { ok = false; break; }
        // the accumulators are free once the previous window has been drained
        if (first && win >= 1 && !mbar_wait(&acce_bar, (uint32_t)((win - 1) & 1))) { ok = false; break; }
        fence_after();
        // one descriptor per stage; a tile's descriptor adds its byte offset / 16 (the stage
        // lies below 256 KB of shared memory, so the 14-bit address field cannot overflow)
        const uint64_t d0 = sdesc_sw64(smem_u32(smem + st * F::STAGE));
#pragma unroll
        for (int s = 0; s < S; ++s)
#pragma unroll
          for (int t = 0; t < S - s; t += F::P) {
            const int n = (S - s - t < F::P ? S - s - t : F::P) * BN;   // up to 256 columns
            mma_f16(tmem + (uint32_t)((s + t) * BN), d0 + (uint64_t)(((s % F::P) * A_TILE + (s / F::P) * 32) >> 4),
                    d0 + (uint64_t)((F::P * A_TILE + (t / F::P) * 32) >> 4), idesc(n), (first && s == 0) ? 0u : 1u);
          }
        mma_commit(&empty_bar[st]);
        if (++kb == kblocks || kb % F::DRAIN_KB == 0) {
          mma_commit(&accf_bar);
          ++win;
          if (kb == kblocks) kb = 0;
        }
      }
      mma_commit(&done_bar);
      if (!ok) atomicExch(err, 1);
    }
  } else {
    constexpr int HALF = BN / 2;              // columns of this warp
    constexpr int NACC = S / 4;               // 64-bit sums per element: orders 4 a .. 4 a + 3 in sum a
    const int quad = warp % 4, half = warp / 4;
    const uint32_t t_base = tmem + ((uint32_t)(quad * 32) << 16) + (uint32_t)(half * HALF);
    T *stage = reinterpret_cast<T *>(smem + STAGES * F::STAGE);   // [128][EPI_COLS + 1]
    int win = 0;
    for (int tile = blockIdx.x; tile < ntiles && ok; tile += gridDim.x) {
      // sum[a][j] = sum over the windows of sum_{d < 4} acc_{4 a + d} 2^{7 (3 - d)}
      long long sum[NACC][HALF];
#pragma unroll
      for (int a = 0; a < NACC; ++a)
#pragma unroll
        for (int j = 0; j < HALF; ++j) sum[a][j] = 0;
      for (int w = 0; w < nwin; ++w, ++win) {
        if (!__all_sync(0xffffffffu, mbar_wait(&accf_bar, (uint32_t)(win & 1)))) { ok = false; break; }
        fence_after();
#pragma unroll
        for (int c = 0; c < HALF / 8; ++c) {   // 8 columns at a time: the sums leave 40 registers of 168
          uint32_t a[8], b[8];
#pragma unroll
          for (int q = 0; q < S / 2; ++q) {
            tmem_ld8(t_base + (uint32_t)(2 * q * BN + c * 8), a);
            tmem_ld8(t_base + (uint32_t)((2 * q + 1) * BN + c * 8), b);
            asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
            for (int j = 0; j < 8; ++j) {
              // below 2^31: at most (36,864 x 384 or 20,480 x 640) x 128 + 2^24
              const int pair = __float2int_rn(__uint_as_float(a[j])) * (1 << BITS) + __float2int_rn(__uint_as_float(b[j]));
              sum[q / 2][c * 8 + j] += (q % 2 == 0) ? (long long)pair * (1 << (2 * BITS)) : (long long)pair;
            }
          }
        }
        fence_before();
        mbar_arrive(&acce_bar);
      }
      // a warp whose wait ran out takes the others with it (they share the barriers below)
      if (!(ok = epilogue_all(ok))) break;
      int bz, bx, by;
      tile_at(tile, bz, bx, by);
      const int row = quad * 32 + lane;           // stacked row within the tile
      // the two exponents meet in one step: their sum may be in range where one alone is not
      if (half == 0) row_exp[row] = sa[(size_t)bz * pr.za + by * BM + row] - BITS * (S + 1);
      const int *sbz = sb + (size_t)bz * pr.zb;
      T *Cz = C + (STACKED ? 2 : 1) * bz * pr.zc;
#pragma unroll
      for (int h = 0; h < 2; ++h) {
#pragma unroll
        for (int c0 = 0; c0 < HALF; c0 += EPI_COLS) {
          if (half == h) {
#pragma unroll
            for (int j = 0; j < EPI_COLS; ++j) {
              T v = (T)sum[0][c0 + j];
              if constexpr (NACC == 2) v = fma(v, (T)(1ll << (4 * BITS)), (T)sum[NACC - 1][c0 + j]);
              stage[row * (EPI_COLS + 1) + j] = v;
            }
          }
          asm volatile("bar.sync 1, 256;" ::: "memory");
          const int n0 = bx * BN + h * HALF + c0;
          if (STACKED) {
            // complex rows: real parts in rows 0-63 of the tile, imaginary parts in 64-127
            for (int e = threadIdx.x; e < 64 * EPI_COLS; e += 32 * EPI_WARPS) {
              const int rr = e / EPI_COLS, cc = e % EPI_COLS;
              const int gm = by * 64 + rr, gn = n0 + cc;
              if (gm < pr.M && gn < pr.N) {
                const int eb = sbz[gn];
                T *dst = Cz + 2 * ((size_t)gm * pr.ldc + gn);
                const T re = times_pow2(stage[rr * (EPI_COLS + 1) + cc], row_exp[rr] + eb);
                const T im = times_pow2(stage[(rr + 64) * (EPI_COLS + 1) + cc], row_exp[rr + 64] + eb);
                if constexpr (sizeof(T) == 8) *reinterpret_cast<double2 *>(dst) = make_double2(re, im);
                else *reinterpret_cast<float2 *>(dst) = make_float2(re, im);
              }
            }
          } else {
            for (int e = threadIdx.x; e < BM * EPI_COLS; e += 32 * EPI_WARPS) {
              const int rr = e / EPI_COLS, cc = e % EPI_COLS;
              const int gm = by * BM + rr, gn = n0 + cc;
              if (gm < pr.M && gn < pr.N)
                Cz[(size_t)gm * pr.ldc + gn] = times_pow2(stage[rr * (EPI_COLS + 1) + cc], row_exp[rr] + sbz[gn]);
            }
          }
          asm volatile("bar.sync 1, 256;" ::: "memory");
        }
      }
    }
    if (!mbar_wait(&done_bar, 0)) ok = false;
    if (!ok) atomicExch(err, 1);
  }
  fence_before();
  __syncthreads();
  fence_after();
  if (warp == 0) tmem_dealloc(tmem, TMEM_COLS);
}

}  // namespace oz
}  // namespace ltmp2
