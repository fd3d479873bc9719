// Host check of the fixed-point line FFTs and products (csrc/fixed.cuh, compiled for the CPU
// through their __host__ paths): every supported length, both directions, on integers whose
// absolute sum is just below 2^61, against the exact integer DFT.  Prints one line per
// case: N DIR max|X - X_ref| in units, then the constants and the product.
#include <cmath>
#include <cstdio>
#include <cstdint>

#include "fixed.cuh"

using namespace ltmp2;

static uint64_t rng = 88172645463325252ull;
static uint64_t next() { rng ^= rng << 13; rng ^= rng >> 7; rng ^= rng << 17; return rng; }
static double uni() { return (double)(next() >> 11) / 9007199254740992.0 * 2.0 - 1.0; }

template <int N, int DIR> double check(int kind) {
  cpx<long long> a[N];
  double re[N], im[N], sum = 0;
  for (int n = 0; n < N; ++n) {
    re[n] = kind == 2 ? (n == 3 % N ? 1.0 : 0.0) : uni();
    im[n] = kind == 1 ? 0.0 : kind == 2 ? 0.0 : uni();
    if (kind == 1) re[n] = std::fabs(re[n]);
    sum += std::hypot(re[n], im[n]);
  }
  const double f = 2305843009213693952.0 / sum * 0.999999;
  for (int n = 0; n < N; ++n) a[n] = {(long long)(re[n] * f), (long long)(im[n] * f)};
  if (kind != 2)
    for (int n = 0; n < N; ++n) { a[n].x += (long long)(next() & 255); if (kind == 0) a[n].y -= (long long)(next() & 255); }
  cpx<long long> x[N];
  for (int n = 0; n < N; ++n) x[n] = a[n];
  LineFFT<long long, N, DIR>::run(a);
  double worst = 0;
  for (int k = 0; k < N; ++k) {
    __int128 sr = 0, si = 0;   // times 2^62
    for (int n = 0; n < N; ++n) {
      const int e = (k * n) % N;
      const __int128 c = fxc::cosn(e, N), s = DIR * fxc::sinn(e, N);
      sr += (__int128)x[n].x * c - (__int128)x[n].y * s;
      si += (__int128)x[n].x * s + (__int128)x[n].y * c;
    }
    const double dr = (double)(((__int128)a[k].x << 62) - sr) / 4611686018427387904.0;
    const double di = (double)(((__int128)a[k].y << 62) - si) / 4611686018427387904.0;
    worst = std::fmax(worst, std::fmax(std::fabs(dr), std::fabs(di)));
  }
  return worst;
}

template <int N> void row() {
  for (int dir = -1; dir <= 1; dir += 2) {
    double w = 0;
    for (int rep = 0; rep < 40; ++rep)
      for (int kind = 0; kind < 3; ++kind) w = std::fmax(w, dir < 0 ? check<N, -1>(kind) : check<N, 1>(kind));
    std::printf("%d %d %.3f\n", N, dir, w);
  }
}

int main() {
  row<8>(); row<10>(); row<12>(); row<16>(); row<18>(); row<20>(); row<24>();
  row<25>(); row<27>(); row<30>(); row<32>(); row<36>(); row<40>();
  // the table constants against the host's cosine
  double tw = 0;
  for (int n : {8, 25, 27, 32, 36, 40, 160})
    for (int e = 0; e < n; ++e) {
      const long double t = 6.283185307179586476925286766559005768L * e / n;
      tw = std::fmax(tw, (double)std::fabs((long double)fxc::cosn(e, n) / 4611686018427387904.0L - std::cos(t)));
      tw = std::fmax(tw, (double)std::fabs((long double)fxc::sinn(e, n) / 4611686018427387904.0L - std::sin(t)));
    }
  std::printf("const 0 %.3e\n", tw);
  // products: |x|, |y| <= 2^61 of every magnitude, and the ends of the range
  double mean = 0, worst = 0, back = 0;
  const int n = 200000;
  auto err = [&](long long x, long long y) {
    const fx2 a = fx_split(x), b = fx_split(y);
    back = std::fmax(back, std::fabs((double)(((__int128)a.hi << 31) + a.lo - x)));
    return (double)(((__int128)fx_mul61(a, b) << 61) - (__int128)x * y) / 2305843009213693952.0;
  };
  for (int i = 0; i < n; ++i) {
    const int sa = (int)(next() % 40), sb = (int)(next() % 40);
    const double d = err(((long long)next() >> 2) >> sa, ((long long)next() >> 2) >> sb);
    mean += d / n;
    worst = std::fmax(worst, std::fabs(d));
  }
  const long long top = 1ll << 61;
  for (long long x : {top, -top, top - 1, 0ll, (1ll << 30) - 1, 1ll << 30, -(1ll << 30)})
    for (long long y : {top, -top, top - 1, 0ll, (1ll << 30) - 1, 1ll << 30, -(1ll << 30)})
      worst = std::fmax(worst, std::fabs(err(x, y)));
  std::printf("mul %.4f %.4f %.1f\n", mean, worst, back);
  return 0;
}
