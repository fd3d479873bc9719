// FP64-accurate products on the tcgen05 tensor cores (the FP64 path's Green's function and
// transformed states of step (iii), Sec. III A), by exact integer slices (Ozaki's scheme):
//
//   each row of A and of B (C = A B^T, both K-major) is scaled by a power of two 2^e with
//   |x| < 2^e over the row and cut into S = 8 slices of 7 bits,
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
// What bounds it: 36 slice products per product.  FP16 operands run at twice the TF32 rate and
// half the bytes of the same integers.  Slice s of A multiplies the slices t < S - s of B in
// MMAs of up to 256 columns: the B slices lie one after another in shared memory and so do
// the orders s + t in tensor memory, so 12 instructions replace 36 and A is read from shared
// memory once per 256 columns instead of once per 64.  The drain runs on integers because the
// FP64 pipe (2 operations per clock and SM) needed 69,000 clocks per 128 x 64 tile and window
// where the window's products take 27,600; 8 float-to-integer conversions an element take 4,100.
// One persistent block per SM: the next tile's products run while a tile is written.
// 4501 x 3071 x 3039 on GB300: 12.9 ms with TF32 slices and FP64 drains, 4.0 ms now (1.6 ms is
// what the slice products take at the measured FP16 rate).
#pragma once
#include <cuda.h>
#include <cuda_fp16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "tcgen05.cuh"

namespace ltmp2 {
namespace oz {

constexpr int S = 8;                         // slices per operand
constexpr int BITS = 7;                      // bits per slice
constexpr int BM = 128;                      // rows of A per tile (tensor-memory lanes)
constexpr int BN = 64;                       // rows of B per tile (accumulator columns)
constexpr int BK = 32;                       // fp16 per k block (one 64-byte swizzle row)
constexpr int A_TILE = BM * 64;              // bytes of one A slice tile
constexpr int B_TILE = BN * 64;
constexpr int STAGE = S * (A_TILE + B_TILE); // 96 KB
constexpr int STAGES = 2;
constexpr int EPI_COLS = 32;                 // columns staged per output round
constexpr int EPI_BYTES = BM * (EPI_COLS + 1) * (int)sizeof(double);
constexpr int SMEM = STAGES * STAGE + EPI_BYTES + 1024;  // + alignment slack
constexpr int TMEM_COLS = S * BN;            // one accumulator per slice order d = s + t
constexpr int DRAIN_KB = 12;                 // k blocks between drains (384 k: sums below 2^24)
constexpr int EPI_WARPS = 8;
constexpr int THREADS = 32 * (EPI_WARPS + 1);
constexpr int GROUP_ROWS = 12;               // row tiles that run side by side (12 x 12 tiles share operands in L2)
static_assert((2 * 128 * 64 + 6 * 64 * 64) * DRAIN_KB * BK < (1 << 24), "order sums exact in FP32");
// instruction descriptor: D fp32, A and B fp16, both K-major, M = 128, N columns
__host__ __device__ constexpr uint32_t idesc(int n) {
  return (1u << 4) | ((uint32_t)(n >> 3) << 17) | ((uint32_t)(BM >> 4) << 24);
}

// Magnitudes are compared as the integers of their bits (the FP64 pipe is the slowest of the
// SM): the same order for finite values, with infinities and NaN above them.
typedef unsigned long long Bits;
constexpr Bits kInfBits = 0x7ff0000000000000ull;
__device__ __forceinline__ Bits magnitude(double x) { return (Bits)__double_as_longlong(x) & 0x7fffffffffffffffull; }
// the smallest e with |x| < 2^e for every |x| <= m (0 for m = 0 and for rows that are not finite)
__device__ __forceinline__ int row_exponent(Bits m) {
  return m > 0 && m < kInfBits ? ilogb(__longlong_as_double((long long)m)) + 1 : 0;
}
// the row's scale 2^e; NaN for a row that holds a NaN or an infinity, whose products are NaN
__device__ __forceinline__ double stored_scale(Bits m, int e) {
  return m < kInfBits ? ldexp(1.0, e) : __longlong_as_double(0x7ff8000000000000ll);
}

// times 2^s, in two factors for rows of denormal numbers (one alone would overflow)
struct RowScale {
  double f1, f2;
  bool two;
  __device__ __forceinline__ explicit RowScale(int s) {
    const int a = min(max(s, -1000), 1000);
    f1 = ldexp(1.0, a);
    f2 = ldexp(1.0, s - a);
    two = s != a;
  }
  __device__ __forceinline__ double operator()(double x) const {
    x *= f1;
    return two ? x * f2 : x;
  }
};

// x 2^(56 - e) rounded to an integer, |x| < 2^e, as S balanced digits of 7 bits, top digit first:
// x = 2^e sum_s d_s 2^{-7(s+1)} + r, |r| <= 2^{e-57}; |d_0| <= 128, -64 <= d_s < 64 after
__device__ __forceinline__ void slice(double x, const RowScale &f, __half (&d)[S]) {
  long long v = __double2ll_rn(f(x));
#pragma unroll
  for (int s = S - 1; s > 0; --s) {
    const int lo = (((int)v + 64) & 127) - 64;
    d[s] = __int2half_rn(lo);
    v = (v - lo) >> BITS;
  }
  d[0] = __int2half_rn((int)v);
}

// block-wide max of v over blockDim.x threads (blockDim.x a multiple of 32, <= 1024)
__device__ __forceinline__ Bits block_max(Bits v, Bits *red) {
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
// when cscale is not null: plane s row r at planes[(s * prows + r) * pitch + q] for
// q < kfill (zero past k); scale[r] = 2^e_r.  One block per row r < prows.  kfill and pitch are even.
__global__ void k_oz_split_rows(const double *__restrict__ x, int nrows, int k, int ld, const double *__restrict__ cscale,
                                int kfill, int pitch, int prows, __half *__restrict__ planes, double *__restrict__ scale) {
  __shared__ Bits red[32];
  const int r = blockIdx.x;
  const double *row = x + (size_t)r * ld;
  auto at = [&](int q) { return r < nrows && q < k ? (cscale ? row[q] * cscale[q] : row[q]) : 0.0; };
  Bits m = 0;
  for (int q = threadIdx.x; q < k; q += blockDim.x) m = max(m, magnitude(at(q)));
  m = block_max(m, red);
  const int e = row_exponent(m);
  if (threadIdx.x == 0) scale[r] = stored_scale(m, e);
  const RowScale f(S * BITS - e);
  for (int q = 2 * threadIdx.x; q < kfill; q += 2 * blockDim.x) {
    __half d0[S], d1[S];
    slice(at(q), f, d0);
    slice(at(q + 1), f, d1);
#pragma unroll
    for (int s = 0; s < S; ++s)
      *reinterpret_cast<__half2 *>(planes + ((size_t)s * prows + r) * pitch + q) = __halves2half2(d0[s], d1[s]);
  }
}

// Slices of the stacked rows of a complex matrix X [rows][ld] (columns q < k): complex row
// m gives stacked row 128 (m / 64) + m % 64 (its real part) and that + 64 (its imaginary
// part), each with its own scale; plane s row r at planes[(s * prows + r) * pitch + q] for
// q < kfill.  One block per complex row m < prows / 2 (rows past `rows` are zero).
__global__ void k_oz_split_stacked(const double2 *__restrict__ x, int rows, int k, int ld, int kfill, int pitch,
                                   int prows, __half *__restrict__ planes, double *__restrict__ scale) {
  __shared__ Bits red[32];
  const int m = blockIdx.x;
  const size_t r1 = (size_t)128 * (m / 64) + (m % 64), r2 = r1 + 64;
  Bits mr = 0, mi = 0;
  if (m < rows)
    for (int q = threadIdx.x; q < k; q += blockDim.x) {
      const double2 v = x[(size_t)m * ld + q];
      mr = max(mr, magnitude(v.x));
      mi = max(mi, magnitude(v.y));
    }
  mr = block_max(mr, red);
  mi = block_max(mi, red);
  const int er = row_exponent(mr), ei = row_exponent(mi);
  if (threadIdx.x == 0) {
    scale[r1] = stored_scale(mr, er);
    scale[r2] = stored_scale(mi, ei);
  }
  const RowScale fr(S * BITS - er), fi(S * BITS - ei);
  for (int q = 2 * threadIdx.x; q < kfill; q += 2 * blockDim.x) {
    double2 v0 = make_double2(0.0, 0.0), v1 = v0;
    if (m < rows && q < k) v0 = x[(size_t)m * ld + q];
    if (m < rows && q + 1 < k) v1 = x[(size_t)m * ld + q + 1];
    __half a0[S], a1[S];
    slice(v0.x, fr, a0);
    slice(v1.x, fr, a1);
#pragma unroll
    for (int s = 0; s < S; ++s)
      *reinterpret_cast<__half2 *>(planes + ((size_t)s * prows + r1) * pitch + q) = __halves2half2(a0[s], a1[s]);
    slice(v0.y, fi, a0);
    slice(v1.y, fi, a1);
#pragma unroll
    for (int s = 0; s < S; ++s)
      *reinterpret_cast<__half2 *>(planes + ((size_t)s * prows + r2) * pitch + q) = __halves2half2(a0[s], a1[s]);
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

// C = A B^T from the slices.  Persistent: block b takes tiles b, b + gridDim.x, ... of the
// nbx x nby tiles (64 columns x 128 stacked rows).  Warp 8 (one elected thread) issues the TMA copies and the
// MMAs; warps 0-7 drain the 8 accumulators every DRAIN_KB k blocks (warp w: lanes 32 (w % 4) on,
// columns 32 (w / 4) on) and write the tile.
// STACKED: A rows are the stacked real / imaginary rows of k_oz_split_stacked and C is
// complex [M][ldc] (M complex rows); else C is real [M][ldc].  Every wait is bounded: on
// expiry the block raises *err, waits (bounded) for its own copies, writes nothing more, frees its
// tensor memory and returns.
template <bool STACKED>
__global__ void __launch_bounds__(THREADS, 1)
    k_dgemm_oz(const __grid_constant__ CUtensorMap ta, const __grid_constant__ CUtensorMap tb, int M, int N,
               int kblocks, int arows, int brows, int nbx, int nby, const double *__restrict__ sa,
               const double *__restrict__ sb, double *__restrict__ C, int ldc, int *__restrict__ err) {
  using namespace tc;
  extern __shared__ unsigned char smem_raw[];
  __shared__ uint64_t full_bar[STAGES], empty_bar[STAGES], accf_bar, acce_bar, done_bar;
  __shared__ uint32_t tmem_slot;
  unsigned char *smem = reinterpret_cast<unsigned char *>(
      (reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~static_cast<uintptr_t>(1023));
  const int warp = threadIdx.x / 32, lane = threadIdx.x % 32;
  const int ntiles = nbx * nby;
  // tile -> (bx, by): groups of GROUP_ROWS row tiles, rows fastest within a group
  auto tile_at = [&](int t, int &bx, int &by) {
    const int per = GROUP_ROWS * nbx, g = t / per, r = t - g * per;
    const int rows = min(GROUP_ROWS, nby - g * GROUP_ROWS);
    by = g * GROUP_ROWS + r % rows;
    bx = r / rows;
  };
  const int nwin = (kblocks + DRAIN_KB - 1) / DRAIN_KB;

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

  if (warp == EPI_WARPS) {
    if (lane == 0) {
      // k blocks are counted over all tiles of this block: block kb of tile i is i kblocks + kb
      const int mine = (int)blockIdx.x < ntiles ? (ntiles - (int)blockIdx.x + (int)gridDim.x - 1) / (int)gridDim.x : 0;
      const int total = mine * kblocks;
      int ld_tile = blockIdx.x, ld_kb = 0, arow0 = 0, brow0 = 0;
      auto place = [&] {
        int bx, by;
        tile_at(ld_tile, bx, by);
        arow0 = by * BM;
        brow0 = bx * BN;
      };
      if (total > 0) place();
      auto issue = [&](int g) {   // k block g, called in order
        unsigned char *p = smem + (g % STAGES) * STAGE;
        uint64_t *bar = &full_bar[g % STAGES];
        mbar_expect_tx(bar, STAGE);
        const int x = ld_kb * BK;
        for (int s = 0; s < S; ++s) tma_load_2d(p + s * A_TILE, &ta, bar, x, s * arows + arow0);
        for (int t = 0; t < S; ++t) tma_load_2d(p + S * A_TILE + t * B_TILE, &tb, bar, x, t * brows + brow0);
        if (++ld_kb == kblocks) {
          ld_kb = 0;
          ld_tile += gridDim.x;
          if (ld_tile < ntiles) place();
        }
      };
      int issued = 0, consumed = 0, win = 0, kb = 0;
      for (; issued < STAGES && issued < total; ++issued) issue(issued);
      for (int g = 0; g < total; ++g) {
        const int st = g % STAGES;
        const bool first = kb % DRAIN_KB == 0;
        if (!mbar_wait(&full_bar[st], (uint32_t)((g / STAGES) & 1))) { ok = false; break; }
        consumed = g + 1;
        // the accumulators are free once the previous window has been drained
        if (first && win >= 1 && !mbar_wait(&acce_bar, (uint32_t)((win - 1) & 1))) { ok = false; break; }
        fence_after();
        // one descriptor per stage; a tile's descriptor adds its byte offset / 16 (the stage
        // lies below 256 KB of shared memory, so the 14-bit address field cannot overflow)
        const uint64_t d0 = sdesc_sw64(smem_u32(smem + st * STAGE));
#pragma unroll
        for (int k16 = 0; k16 < BK / 16; ++k16)
#pragma unroll
          for (int s = 0; s < S; ++s)
#pragma unroll
            for (int t = 0; t < S - s; t += 4) {
              const int n = (S - s - t < 4 ? S - s - t : 4) * BN;   // up to 256 columns
              mma_f16(tmem + (uint32_t)((s + t) * BN), d0 + (uint64_t)((s * A_TILE + k16 * 32) >> 4),
                      d0 + (uint64_t)((S * A_TILE + t * B_TILE + k16 * 32) >> 4), idesc(n),
                      (first && s == 0 && k16 == 0) ? 0u : 1u);
            }
        mma_commit(&empty_bar[st]);
        if (++kb == kblocks || kb % DRAIN_KB == 0) {
          mma_commit(&accf_bar);
          ++win;
          if (kb == kblocks) kb = 0;
        }
        // refill the stage of k block g - 1 once its MMAs are done (those of g are queued)
        if (g >= 1 && issued < total) {
          if (!mbar_wait(&empty_bar[(g - 1) % STAGES], (uint32_t)(((g - 1) / STAGES) & 1))) { ok = false; break; }
          issue(issued++);
        }
      }
      mma_commit(&done_bar);
      if (!ok) {
        atomicExch(err, 1);
        drain_issued<STAGES>(full_bar, consumed, issued);
      }
    }
  } else {
    const int quad = warp % 4, half = warp / 4;
    const uint32_t t_base = tmem + ((uint32_t)(quad * 32) << 16) + (uint32_t)(half * EPI_COLS);
    double *stage = reinterpret_cast<double *>(smem + STAGES * STAGE);   // [128][EPI_COLS + 1]
    int win = 0;
    for (int tile = blockIdx.x; tile < ntiles && ok; tile += gridDim.x) {
      // orders 0-3 and 4-7 of the lane's row, 32 columns: sum_d acc_d 2^{7 (3 - d)} and 2^{7 (7 - d)}
      long long hi[EPI_COLS], lo[EPI_COLS];
#pragma unroll
      for (int j = 0; j < EPI_COLS; ++j) hi[j] = lo[j] = 0;
      for (int w = 0; w < nwin; ++w, ++win) {
        if (!__all_sync(0xffffffffu, mbar_wait(&accf_bar, (uint32_t)(win & 1)))) { ok = false; break; }
        fence_after();
#pragma unroll
        for (int c = 0; c < EPI_COLS / 8; ++c) {   // 8 columns at a time: 2 x 64 sums leave 40 registers of 168
          uint32_t a[8], b[8];
#pragma unroll
          for (int q = 0; q < S / 2; ++q) {
            tmem_ld8(t_base + (uint32_t)(2 * q * BN + c * 8), a);
            tmem_ld8(t_base + (uint32_t)((2 * q + 1) * BN + c * 8), b);
            asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
            for (int j = 0; j < 8; ++j) {
              // below 2^31: order 6's 36,864 x 384 x 128 + order 7's 40,960 x 384
              const int pair = __float2int_rn(__uint_as_float(a[j])) * (1 << BITS) + __float2int_rn(__uint_as_float(b[j]));
              long long &sum = q < 2 ? hi[c * 8 + j] : lo[c * 8 + j];
              sum += (q % 2 == 0) ? (long long)pair * (1 << (2 * BITS)) : (long long)pair;
            }
          }
        }
        fence_before();
        mbar_arrive(&acce_bar);
      }
      // a warp whose wait ran out takes the others with it (they share the barriers below)
      if (!(ok = epilogue_all(ok))) break;
      int bx, by;
      tile_at(tile, bx, by);
      const int row = quad * 32 + lane;           // stacked row within the tile
      const double fa = sa[by * BM + row] * ldexp(1.0, -BITS * (S + 1));
#pragma unroll 1
      for (int h = 0; h < BN / EPI_COLS; ++h) {
        if (half == h) {
#pragma unroll
          for (int j = 0; j < EPI_COLS; ++j)
            stage[row * (EPI_COLS + 1) + j] = fma((double)hi[j], (double)(1ll << (4 * BITS)), (double)lo[j]) * fa;
        }
        asm volatile("bar.sync 1, 256;" ::: "memory");
        const int n0 = bx * BN + h * EPI_COLS;
        if (STACKED) {
          // complex rows: real parts in rows 0-63 of the tile, imaginary parts in 64-127
          for (int e = threadIdx.x; e < 64 * EPI_COLS; e += 32 * EPI_WARPS) {
            const int rr = e / EPI_COLS, cc = e % EPI_COLS;
            const int gm = by * 64 + rr, gn = n0 + cc;
            if (gm < M && gn < N) {
              const double fb = sb[gn];
              reinterpret_cast<double2 *>(C)[(size_t)gm * ldc + gn] =
                  make_double2(stage[rr * (EPI_COLS + 1) + cc] * fb, stage[(rr + 64) * (EPI_COLS + 1) + cc] * fb);
            }
          }
        } else {
          for (int e = threadIdx.x; e < BM * EPI_COLS; e += 32 * EPI_WARPS) {
            const int rr = e / EPI_COLS, cc = e % EPI_COLS;
            const int gm = by * BM + rr, gn = n0 + cc;
            if (gm < M && gn < N) C[(size_t)gm * ldc + gn] = stage[rr * (EPI_COLS + 1) + cc] * sb[gn];
          }
        }
        asm volatile("bar.sync 1, 256;" ::: "memory");
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
