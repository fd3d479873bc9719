// Whole energies by the exchange symmetry of the pairs.
//
// Without the occupied factors, S_ij(G, G') = <i| e^{-iGr} P_v(tau) e^{-iG'r} |j> obeys
//     S_ji(G, G') = S_ij(G', G)                     (real orbitals),
//     S_ji(G, G') = conj S_ij(-G', -G)              (general orbitals),
// because P_v(tau) is Hermitian (and real for real orbitals), so the co-densities of (j, i) are
// those of (i, j) with the two momenta exchanged.  When every G' is summed (a range of G' has no
// such partner), only the items i <= j are transformed, half of the plane and column work, and
//     sum_{G'} v(G') X_ij(G') = sum_{G, G'} v(G) v(G') S_ij(G, G') conj S_ij(G', G) d_i d_j
// with d_i = e^{(e_i - mu) tau}: the exchange term is a matrix times its own transpose, element by
// element, and its terms (G, G') and (G', G) are each other's conjugates, so half of them are summed.
// The direct term is sum v v' S_ii conj S_jj (real; general: S_jj at (-G, -G')), symmetric in the
// same way.
//
// S_ij is kept over an index set: the primary G' of real orbitals (two planes: S(p, g') and
// S(-p, g'); S(-G, -G') = conj S(G, G') holds the rest), every G != 0 of general orbitals (one
// plane, G and -G side by side).  The set is sorted by |G|^2, so that the nested auxiliary spheres of
// the cutoff extrapolation are prefixes of it: row g' of the lower triangle (columns p <= g') belongs
// to the spheres that contain g', and a level's sum is the sum of its rows.
//
// Measured against the slabs of G' (whole energies on GB300): 20^3 FP64 260 -> 165 ms (planes
// 148 -> 94, column 38 -> 25 with the contraction, direct 28 -> 3.5, sums 4 -> 0), 24^3 FP32 302 ->
// 219 (planes 165 -> 97, column 51 -> 53, direct and sums 19 -> 8.5).
#pragma once
#include "kernels.cuh"

namespace ltmp2 {

// pair slot of a pass -> (i, j): the orbitals j of the pass in turn, i <= j
__device__ __forceinline__ void sym_pair(const Plan &p, int t, int &i, int &j) {
  j = p.sym_j0;
  while (t > j) t -= ++j;
  i = t;
}
__device__ __forceinline__ size_t sym_pair_slot(const Plan &p, int i, int j) {
  const int a = j - p.sym_j0;
  return (size_t)a * p.sym_j0 + (size_t)a * (a + 1) / 2 + i;
}
// pairs left out of the exchange (learned form)
__device__ __forceinline__ bool sym_screened(const Plan &p, int i, int j) {
  return p.pair_keep && i != j && !p.pair_keep[i * p.n_occ + j];
}
template <typename T> __device__ __forceinline__ cpx<T> *sym_matrix(const Plan &p, int i, int j) {
  const size_t n2 = (size_t)p.sym_planes * p.n_idx * p.n_idx;
  return i == j ? (cpx<T> *)p.mdsym + j * n2 : (cpx<T> *)p.msym + sym_pair_slot(p, i, j) * n2;
}

// Column kernel of a pass: block (i, column).  z transform of the item's aux-disk columns, the kept
// points gathered by index in shared memory and written as row g' of S_ij's planes.
template <typename T, int N>
__global__ void __launch_bounds__(256) k_zsym(Plan p, int gp0) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  typedef typename Codensity<T>::W W;
  cpx<T> *row = reinterpret_cast<cpx<T> *>(smem_raw);   // [sym_planes n_idx]
  const int i = blockIdx.x, col = blockIdx.y;
  const int j = col_orbital(p, col);
  if (i > j || sym_screened(p, i, j)) return;
  const int g = gp0 + col / p.sym_nj;
  const cpx<W> *src0 = (const cpx<W> *)p.tbuf + item_of(p, col, i) * N * p.n_daux;
  const T sc = Codensity<T>::scale(p, i, col);
  for (int d = threadIdx.x; d < p.n_daux; d += blockDim.x) {
    const int4 c = p.daux[d];
    const int off = p.daux_off[d];
    cpx<W> a[N];
#pragma unroll
    for (int k = 0; k < N; ++k) a[k] = src0[(size_t)k * p.n_daux + d];
    LineFFT<W, N, -1>::run(a);
#pragma unroll
    for (int k = 0; k < N; ++k) {
      const int m = freq_of<N>(k);
      if (m >= c.z && m <= c.w) {
        const int q = p.sym_pos[off + m - c.z];
        if (q >= 0) row[q] = cscale(Codensity<T>::real(a[k]), sc);
      }
    }
  }
  __syncthreads();
  cpx<T> *S = sym_matrix<T>(p, i, j) + (size_t)g * p.n_idx;
  for (int pl = 0; pl < p.sym_planes; ++pl)
    for (int q = threadIdx.x; q < p.n_idx; q += blockDim.x)
      S[(size_t)pl * p.n_idx * p.n_idx + q] = row[pl * p.n_idx + q];
}

// Exchange sums of a pass: block (pair, row tile); rows[pair][g'] = v(g') sum_{p <= g'} c v(p)
// Re[S(p, g') conj S(g', p)] (second plane: Re[S(-p, g') S(-g', p)]), c = 2 below the diagonal and 1
// on it.  32 x 32 tiles, the transposed one through shared memory; every term is added in FP64.  Bound by reading S once (12.7 GB per Laplace point of the
// 24^3 system in FP64).
template <typename T> __global__ void __launch_bounds__(256) k_xsym(Plan p, double *__restrict__ rows) {
  __shared__ cpx<T> tile[2][32][33];
  const int nt = (p.n_idx + 31) / 32, R = nt - 1 - (int)blockIdx.y, pair = blockIdx.x;
  const int n = p.n_idx;
  int i, j;
  sym_pair(p, pair, i, j);
  if (sym_screened(p, i, j)) return;
  const cpx<T> *S = sym_matrix<T>(p, i, j);
  const size_t n2 = (size_t)n * n;
  const bool two = p.sym_planes == 2;
  const T *v = vtab<T>(p);
  const int tx = threadIdx.x % 32, ty = threadIdx.x / 32;
  double acc[4] = {0, 0, 0, 0};
  for (int C = 0; C <= R; ++C) {
    const int col = C * 32 + tx;
    const T vc = col < n ? v[p.sym_order[col]] : T(0);
    cpx<T> x[2][4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const int r = C * 32 + ty + 8 * k, c = R * 32 + tx;     // the transposed tile's rows
      const int row = R * 32 + ty + 8 * k;
      const bool in_t = r < n && c < n, in_x = row < n && col < n;
      const cpx<T> zero{T(0), T(0)};
      tile[0][ty + 8 * k][tx] = in_t ? S[(size_t)r * n + c] : zero;
      x[0][k] = in_x ? S[(size_t)row * n + col] : zero;
      if (two) {
        tile[1][ty + 8 * k][tx] = in_t ? S[n2 + (size_t)r * n + c] : zero;
        x[1][k] = in_x ? S[n2 + (size_t)row * n + col] : zero;
      }
    }
    __syncthreads();
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const int row = R * 32 + ty + 8 * k;
      const cpx<T> y = tile[0][tx][ty + 8 * k];
      T t = x[0][k].x * y.x + x[0][k].y * y.y;
      if (two) {
        const cpx<T> z = tile[1][tx][ty + 8 * k];
        t += x[1][k].x * z.x - x[1][k].y * z.y;
      }
      if (col <= row) acc[k] += (double)(vc * (col < row ? t + t : t));
    }
    __syncthreads();
  }
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    for (int o = 16; o > 0; o >>= 1) acc[k] += __shfl_xor_sync(0xffffffffu, acc[k], o);
    const int row = R * 32 + ty + 8 * k;
    if (tx == 0 && row < n) rows[(size_t)pair * n + row] = acc[k] * p.v_aux64[p.sym_order[row]];
  }
}

// e^x_ij += f d_i d_j sum of the pair's rows (level n: its first lev_rows[n] rows), fixed order; one
// block of 128 per pair
template <typename T> __global__ void k_xsym_sum(Plan p, const double *__restrict__ rows, double f) {
  int i, j;
  sym_pair(p, blockIdx.x, i, j);
  if (sym_screened(p, i, j)) return;
  const T *d = (const T *)p.dscale;
  const double scale = f * (double)d[i] * (double)d[j];
  const double *r = rows + (size_t)blockIdx.x * p.n_idx;
  const int no = p.n_occ;
  for (int n = 0; n < (p.n_lev > 1 ? p.n_lev : 1); ++n) {
    const int end = n == 0 ? p.n_idx : p.lev_rows[n];
    double s = 0.0;
    for (int k = threadIdx.x; k < end; k += blockDim.x) s += r[k];
    s = block_sum(s) * scale;
    if (threadIdx.x == 0) {
      double *ex = n == 0 ? p.ex : p.exl + (size_t)n * no * no;
      ex[i * no + j] += s;
      if (i != j) ex[j * no + i] += s;
    }
  }
}

// Direct term: block (row group, 4 x 4 block of (i, j)); part[group][i][j] = sum over the group's
// rows g' of v(g') sum_{p <= g'} c v(p) Re[S_ii conj S_jj] (general orbitals: Re[S_ii(p, g')
// S_jj(-p, -g')], whose index is the neighbour's; c = 1 within the pair of rows g', -g').  p and q: the
// two channels' plans (the same one for a closed shell; then only blocks with j >= i are there).
// The warps take the rows' 32-column chunks in turn, a lane a column: no product is padded, which in
// FP64 (2 FMA per clock and SM) is what counts: 32 x 32 tiles through shared memory took 1.7 ms
// per Laplace point on the 8^3 system with 2 occupied.  FP32: sums of 64 products, added in FP64.
template <typename T>
__global__ void __launch_bounds__(256) k_dsym(Plan p, Plan q, bool triangle, double *__restrict__ part) {
  constexpr int B = 4;
  __shared__ double red[8][B * B];
  const int n = p.n_idx, ni = p.n_occ, nj = q.n_occ;
  const int nbj = (nj + B - 1) / B;
  int bi = 0, bj = blockIdx.y;
  if (triangle)
    while (bj >= nbj - bi) bj -= nbj - bi++;
  else {
    bi = bj / nbj;
    bj -= bi * nbj;
  }
  const int i0 = bi * B, j0 = (triangle ? bi + bj : bj) * B;
  const size_t n2 = (size_t)n * n, stride = p.sym_planes * n2;
  const bool gen = p.sym_planes == 1;
  const T *v = vtab<T>(p);
  const int warp = threadIdx.x / 32, lane = threadIdx.x % 32;
  constexpr bool kFp32 = std::is_same<T, float>::value;
  T acc[B * B];
  double sum[kFp32 ? B * B : 1];
#pragma unroll
  for (int k = 0; k < B * B; ++k) {
    acc[k] = T(0);
    if (kFp32) sum[k] = 0.0;
  }
  auto carry = [&] {
#pragma unroll
    for (int k = 0; k < B * B; ++k) {
      sum[k] += (double)acc[k];
      acc[k] = T(0);
    }
  };
  const int2 rows = p.sym_groups[blockIdx.x];
  const cpx<T> *Ma = (const cpx<T> *)p.mdsym + i0 * stride, *Mb = (const cpx<T> *)q.mdsym + j0 * stride;
  // the rows' 32-column chunks go round the warps
  int chunk = 0, count = 0;
  for (int g = rows.x; g < rows.y; ++g) {
    const T vg = v[p.sym_order[g]];
    const int end = gen ? (g | 1) + 1 : g + 1;            // columns of the lower triangle
    const int gj = gen ? g ^ 1 : g, twice = gen ? (g & ~1) : g;
    for (int c0 = ((warp - chunk) & 7) * 32; c0 < end; c0 += 256) {
      const int c = c0 + lane;
      if (c >= end) continue;
      const T w = v[p.sym_order[c]] * vg * (c < twice ? T(2) : T(1));
      const int cj = gen ? c ^ 1 : c;
      for (int pl = 0; pl < p.sym_planes; ++pl) {
        const cpx<T> *ra = Ma + pl * n2 + (size_t)g * n + c, *rb = Mb + pl * n2 + (size_t)gj * n + cj;
        cpx<T> x[B], y[B];
#pragma unroll
        for (int k = 0; k < B; ++k) {
          x[k] = i0 + k < ni ? ra[k * stride] : cpx<T>{T(0), T(0)};
          y[k] = j0 + k < nj ? rb[k * stride] : cpx<T>{T(0), T(0)};
        }
#pragma unroll
        for (int a = 0; a < B; ++a) {
          if (i0 + a >= ni) continue;
          const T xr = w * x[a].x, xi = gen ? -(w * x[a].y) : w * x[a].y;
#pragma unroll
          for (int b = 0; b < B; ++b)
            if (j0 + b < nj) acc[a * B + b] = fma(xr, y[b].x, fma(xi, y[b].y, acc[a * B + b]));
        }
      }
      if (kFp32 && (++count & 15) == 0) carry();   // at most 64 products in plain FP32 (a lane past the end skips a turn)
    }
    chunk += (end + 31) / 32;
  }
  double s;
  if constexpr (kFp32) {
    carry();
    s = warp_sum16(sum);
  } else {
    s = warp_sum16(acc);
  }
  if (lane % 2 == 0) red[warp][lane / 2] = s;
  __syncthreads();
  if (threadIdx.x < B * B) {
    double s = 0.0;
    for (int k = 0; k < 8; ++k) s += red[k][threadIdx.x];
    const int i = i0 + threadIdx.x / B, j = j0 + threadIdx.x % B;
    if (i < ni && j < nj) part[((size_t)blockIdx.x * ni + i) * nj + j] = s;
  }
}

// acc[i][j] += f d_i d_j sum of the groups (level n: those whose rows are in it), fixed order, one warp per
// (i, j).  symmetric: only blocks with j >= i were summed, and acc is written both ways.
template <typename T>
__global__ void k_dsym_sum(Plan p, Plan q, bool symmetric, const double *__restrict__ part, double f,
                           double *__restrict__ acc, double *__restrict__ acc_lev) {
  const int ni = p.n_occ, nj = q.n_occ;
  const int ij = (blockIdx.x * blockDim.x + threadIdx.x) / 32, lane = threadIdx.x % 32;
  if (ij >= ni * nj) return;
  const int i = ij / nj, j = ij % nj;
  if (symmetric && j < i) return;
  const double scale = f * (double)((const T *)p.dscale)[i] * (double)((const T *)q.dscale)[j];
  for (int n = 0; n < (acc_lev && p.n_lev > 1 ? p.n_lev : 1); ++n) {
    const int end = n == 0 ? p.n_idx : p.lev_rows[n];
    double s = 0.0;
    for (int g = lane; g < p.n_groups; g += 32)
      if (p.sym_groups[g].y <= end) s += part[(size_t)g * ni * nj + ij];
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    s *= scale;
    if (lane == 0) {
      double *a = n == 0 ? acc : acc_lev + (size_t)n * ni * nj;
      a[i * nj + j] += s;
      if (symmetric && i != j) a[j * nj + i] += s;
    }
  }
}

}  // namespace ltmp2
