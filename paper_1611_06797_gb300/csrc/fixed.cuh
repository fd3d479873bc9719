// 64-bit fixed-point line FFTs for the FP64 path's co-density transforms (Eq. SCHovrlp).
//
// GB300 issues 2 FP64 operations per clock and SM, but 64 integer ones: a 64-bit integer
// addition runs about 25 times as fast as an FP64 one and a 64 x 64 -> 64 bit product (three
// IMAD.WIDE) 2.5 times as fast (measured, per SM and clock: 50 additions and 4.7 products
// against 1.9 FP64 operations).  An FFT is mostly additions, so the line transforms of the
// co-densities run on integers here.  A plane or line carries one power-of-two scale chosen
// from its 2-norms (Cauchy-Schwarz bounds every partial sum), so that no sum can overflow and
// about 61 bits stay below the bound: the transform's error is that of rounding to 2^-61 of the
// bound, at or below the rounding of the same transform in FP64.  Additions are exact;
// products round to nearest (the rounding constants cancel the mean of the dropped low parts).
#pragma once
#include <type_traits>
#include <utility>

#include "fft.cuh"

namespace ltmp2 {

// ---------------------------------------------------------------- constants
// cos / sin of 2 pi e / n and tangents as integers times 2^-62, by Taylor series in 128-bit
// integers at compile time (a few units of 2^-62 off)
namespace fxc {
typedef __int128 i128;
constexpr i128 kOne = (i128)1 << 62;
constexpr i128 kTwoPi = (i128)14488038916154245685ull * 2;   // 2 pi 2^62
constexpr i128 mul(i128 a, i128 b) { return (a * b) >> 62; }
constexpr i128 taylor(i128 x, bool sine) {
  i128 term = sine ? x : kOne, sum = term;
  const i128 x2 = mul(x, x);
  for (int k = sine ? 1 : 0; k < 40; k += 2) {
    term = -(mul(term, x2) / ((k + 1) * (k + 2)));
    if (term == 0) break;
    sum += term;
  }
  return sum;
}
// e / n of a turn, 0 <= e < n; angles above an eighth of a turn reduce to it
constexpr i128 cosn(int e, int n);
constexpr i128 sinn(int e, int n) {
  if (2 * e > n) return -sinn(n - e, n);
  if (4 * e > n) return cosn(4 * e - n, 4 * n);
  if (8 * e > n) return taylor(kTwoPi / 4 - kTwoPi * e / n, false);
  return taylor(kTwoPi * e / n, true);
}
constexpr i128 cosn(int e, int n) {
  if (2 * e > n) return cosn(n - e, n);
  if (4 * e > n) return -sinn(4 * e - n, 4 * n);
  if (8 * e > n) return taylor(kTwoPi / 4 - kTwoPi * e / n, true);
  return taylor(kTwoPi * e / n, false);
}
}  // namespace fxc

// x * c for |x| < 2^62 and a compile-time constant 0 <= c < 2^62 (times 2^-62).  Constants
// above 5/8 multiply by 1 - c instead, which keeps the sum of the two cross products inside 64 bits.
template <long long C> __host__ __device__ __forceinline__ long long fx_mulc(long long x) {
  static_assert(C >= 0 && C <= (1ll << 62), "constant range");
  if constexpr (C == (1ll << 62)) {
    return x;
  } else if constexpr (C > 5ll << 59) {
    return x - fx_mulc<(1ll << 62) - C>(x);
  } else {
    // c = (h + l 2^-32) 2^-31 with l in [-2^31, 2^31)
    constexpr long long c63 = C << 1;
    constexpr int h = (int)((c63 + (1ll << 31)) >> 32);
    constexpr int l = (int)(c63 - ((long long)h << 32));
    const int xh = (int)(x >> 32);
    const unsigned xl = (unsigned)x;
    // + 2^30 rounds; + l / 2 is the mean of the dropped product of the low halves
    constexpr long long r = (1ll << 30) + l / 2;
    const long long t = (long long)((unsigned long long)xl * (unsigned)h) + ((long long)xh * l + r);
    const long long p = (long long)xh * h;
    return p + p + (t >> 31);
  }
}
// A fixed-point value v, |v| <= 2^61, as v = hi 2^31 + lo with lo in [-2^30, 2^30): both halves are
// signed, so a product of two split values is three signed 32 x 32 -> 64 bit products.
struct alignas(8) fx2 { int lo, hi; };
__host__ __device__ __forceinline__ fx2 fx_split(long long v) {
  const int hi = (int)((v + (1ll << 30)) >> 31);
  return {(int)(v - ((long long)hi << 31)), hi};
}
// a * b * 2^-61, rounded; the product of the low halves is dropped (at most half a unit, mean zero)
__host__ __device__ __forceinline__ long long fx_mul61(fx2 a, fx2 b) {
  const long long t = (long long)a.hi * b.lo + ((long long)a.lo * b.hi + (1ll << 29));
  const long long q = (long long)a.hi * b.hi;
  return q + q + (t >> 30);
}
// x / 2^s rounded to nearest, 0 <= s < 63
__host__ __device__ __forceinline__ long long fx_shr(long long x, int s) {
  return s > 0 ? (x + (1ll << (s - 1))) >> s : x;
}

// ---------------------------------------------------------------- scales
constexpr int kFxBits = 61;          // |fixed-point value| <= 2^61, the bound given by the 2-norms
constexpr int kFxNotFinite = 1 << 20;   // exponent of a state with a NaN or an infinity
// e with 2^e > sqrt(norm2); smaller squares than 2^-962 count as that
__host__ __device__ __forceinline__ int fx_exponent(double norm2) {
  if (!(norm2 < 1e300)) return kFxNotFinite;
  return norm2 < 0x1p-962 ? -480 : (ilogb(norm2) >> 1) + 1;
}

// ---------------------------------------------------------------- radix kernels
template <int DIR> struct Radix<long long, 3, DIR> {
  typedef cpx<long long> C;
  static __host__ __device__ __forceinline__ void run(C (&v)[3]) {
    constexpr long long s3 = (long long)fxc::sinn(1, 3);
    const C t = cadd(v[1], v[2]), d = csub(v[1], v[2]);
    const C m = {v[0].x - (t.x >> 1), v[0].y - (t.y >> 1)};
    const C r = mul_i<DIR>(C{fx_mulc<s3>(d.x), fx_mulc<s3>(d.y)});
    v[0] = cadd(v[0], t);
    v[1] = cadd(m, r);
    v[2] = csub(m, r);
  }
};
// cos(2 pi / 5) + cos(4 pi / 5) = -1/2 and their difference is sqrt(5) / 2, so the cosine part
// takes one product; the sine part takes three
template <int DIR> struct Radix<long long, 5, DIR> {
  typedef cpx<long long> C;
  template <long long K> static __host__ __device__ __forceinline__ C mulc(C a) { return {fx_mulc<K>(a.x), fx_mulc<K>(a.y)}; }
  static __host__ __device__ __forceinline__ void run(C (&v)[5]) {
    constexpr long long h5 = (long long)((fxc::cosn(1, 5) - fxc::cosn(2, 5)) / 2);   // sqrt(5) / 4
    constexpr long long s1 = (long long)fxc::sinn(1, 5), s2 = (long long)fxc::sinn(2, 5);
    const C t1 = cadd(v[1], v[4]), t2 = cadd(v[2], v[3]), t3 = csub(v[1], v[4]), t4 = csub(v[2], v[3]);
    const C a = cadd(t1, t2), b = mulc<h5>(csub(t1, t2));
    const C m = {v[0].x - (a.x >> 2), v[0].y - (a.y >> 2)};
    const C b1 = cadd(m, b), b2 = csub(m, b);
    // q1 = s1 t3 + s2 t4 = s2 (t3 + t4) + (s1 - s2) t3,  q2 = s2 t3 - s1 t4 = s2 (t3 + t4) - (s1 + s2) t4
    const C s = mulc<s2>(cadd(t3, t4));
    const C q1 = cadd(s, mulc<s1 - s2>(t3));
    const C q2 = csub(csub(s, t4), mulc<s1 + s2 - (1ll << 62)>(t4));
    const C r1 = mul_i<DIR>(q1), r2 = mul_i<DIR>(q2);
    v[0] = cadd(v[0], a);
    v[1] = cadd(b1, r1);
    v[4] = csub(b1, r1);
    v[2] = cadd(b2, r2);
    v[3] = csub(b2, r2);
  }
};

// v * exp(DIR * 2 pi i E / NT): eighths of a turn take two products, other angles three
// shears (tan(t/2), sin t, tan(t/2)) after a quarter turn that brings |t| to at most 1/8 turn
template <int NT, int E, int DIR> __host__ __device__ __forceinline__ cpx<long long> ct_twiddle(cpx<long long> v) {
  constexpr int e = E % NT;
  if constexpr ((4 * e) % NT == 0) {
    constexpr int q = (4 * e) / NT;
    if constexpr (q == 0) return v;
    else if constexpr (q == 1) return mul_i<DIR>(v);
    else if constexpr (q == 2) return {-v.x, -v.y};
    else return mul_i<-DIR>(v);
  } else if constexpr (8 * e > NT) {
    // turn by a quarter and go on with what is left, in (-1/8, 1/8] of a turn
    constexpr int quarters = (8 * e + NT) / (2 * NT);          // nearest number of quarter turns
    const cpx<long long> u = ct_twiddle<4, quarters % 4, DIR>(v);
    constexpr int rest = 4 * e - quarters * NT;                // of 4 NT
    if constexpr (rest == 0) return u;
    else if constexpr (rest > 0) return ct_twiddle<4 * NT, rest, DIR>(u);
    else return ct_twiddle<4 * NT, -rest, -DIR>(u);
  } else if constexpr (8 * e == NT) {
    constexpr long long r2 = (long long)fxc::sinn(1, 8);
    return DIR > 0 ? cpx<long long>{fx_mulc<r2>(v.x - v.y), fx_mulc<r2>(v.x + v.y)}
                   : cpx<long long>{fx_mulc<r2>(v.x + v.y), fx_mulc<r2>(v.y - v.x)};
  } else {
    constexpr fxc::i128 sn = fxc::sinn(e, NT), cs = fxc::cosn(e, NT);
    constexpr long long s = (long long)sn, t = (long long)((sn << 62) / (fxc::kOne + cs));
    if constexpr (DIR > 0) {
      v.x -= fx_mulc<t>(v.y);
      v.y += fx_mulc<s>(v.x);
      v.x -= fx_mulc<t>(v.y);
    } else {
      v.x += fx_mulc<t>(v.y);
      v.y -= fx_mulc<s>(v.x);
      v.x += fx_mulc<t>(v.y);
    }
    return v;
  }
}

// f(integral_constant<int, 0>) ... f(integral_constant<int, N - 1>)
template <typename F, int... I> __host__ __device__ __forceinline__ void fx_each(F &&f, std::integer_sequence<int, I...>) {
  (f(std::integral_constant<int, I>{}), ...);
}

// The line FFT with compile-time twiddles, by the splits of LineFFT: fixed-point values V (and the
// packed pairs of pair.cuh, which bring their own ct_twiddle)
template <typename V, int N, int DIR> struct CtLineFFT {
  typedef cpx<V> C;
  static __host__ __device__ __forceinline__ void run(C (&a)[N]) {
    constexpr int P1 = pfa_n1(N);
    if constexpr (P1 > 0) {
      constexpr int N1 = P1, N2 = N / P1;
      constexpr int A = inv_mod(N2 % N1, N1), B = inv_mod(N1 % N2, N2);
      C t[N];
#pragma unroll
      for (int n2 = 0; n2 < N2; ++n2) {
        C v[N1];
#pragma unroll
        for (int n1 = 0; n1 < N1; ++n1) v[n1] = a[(N2 * n1 + N1 * n2) % N];
        CtLineFFT<V, N1, DIR>::run(v);
#pragma unroll
        for (int k1 = 0; k1 < N1; ++k1) t[k1 * N2 + n2] = v[k1];
      }
#pragma unroll
      for (int k1 = 0; k1 < N1; ++k1) {
        C u[N2];
#pragma unroll
        for (int n2 = 0; n2 < N2; ++n2) u[n2] = t[k1 * N2 + n2];
        CtLineFFT<V, N2, DIR>::run(u);
#pragma unroll
        for (int k2 = 0; k2 < N2; ++k2) a[(N2 * A * k1 + N1 * B * k2) % N] = u[k2];
      }
    } else {
      constexpr int R = pick_radix(N), M = N / R;
      static_assert(R == 2 || R == 3 || R == 4 || R == 5, "line length must be 5-smooth");
      C t[N];
      fx_each([&](auto n2c) {
        constexpr int n2 = decltype(n2c)::value;
        C v[R];
#pragma unroll
        for (int n1 = 0; n1 < R; ++n1) v[n1] = a[M * n1 + n2];
        Radix<V, R, DIR>::run(v);
        fx_each([&](auto k1c) {
          constexpr int k1 = decltype(k1c)::value;
          t[M * k1 + n2] = ct_twiddle<N, n2 * k1, DIR>(v[k1]);
        }, std::make_integer_sequence<int, R>{});
      }, std::make_integer_sequence<int, M>{});
#pragma unroll
      for (int k1 = 0; k1 < R; ++k1) {
        C u[M];
#pragma unroll
        for (int n2 = 0; n2 < M; ++n2) u[n2] = t[M * k1 + n2];
        if constexpr (M > 1) CtLineFFT<V, M, DIR>::run(u);
#pragma unroll
        for (int k2 = 0; k2 < M; ++k2) a[k1 + R * k2] = u[k2];
      }
    }
  }
};
template <int N, int DIR, int NT> struct LineFFT<long long, N, DIR, NT> : CtLineFFT<long long, N, DIR> {};

}  // namespace ltmp2
