// Host check of the packed FP32 line FFTs (csrc/pair.cuh through their __host__ paths): both
// lines of a pair, every supported length and direction, against the DFT in double.  Prints one
// line per case: N DIR ||X - X_ref||_2 / ||X_ref||_2.
#include <cmath>
#include <cstdio>

#include "pair.cuh"

using namespace ltmp2;

template <int N, int DIR> void check() {
  cpx<f2> a[N];
  double x[2][N][2];
  unsigned s = 12345u + N;
  for (int n = 0; n < N; ++n) {
    float v[4];
    for (float &q : v) {
      s = s * 1664525u + 1013904223u;
      q = (float)(s >> 8) / 8388608.0f - 1.0f;
    }
    a[n] = {f2_make(v[0], v[1]), f2_make(v[2], v[3])};
    for (int l = 0; l < 2; ++l) {
      x[l][n][0] = v[l];
      x[l][n][1] = v[2 + l];
    }
  }
  LineFFT<f2, N, DIR>::run(a);
  double worst = 0;
  for (int l = 0; l < 2; ++l) {
    double err = 0, ref = 0;
    for (int k = 0; k < N; ++k) {
      double re = 0, im = 0;
      for (int n = 0; n < N; ++n) {
        const double t = DIR * 2 * M_PI * ((k * n) % N) / N, c = std::cos(t), q = std::sin(t);
        re += x[l][n][0] * c - x[l][n][1] * q;
        im += x[l][n][0] * q + x[l][n][1] * c;
      }
      float u[2], v[2];
      f2_get(a[k].x, u[0], u[1]);
      f2_get(a[k].y, v[0], v[1]);
      err += std::pow(u[l] - re, 2) + std::pow(v[l] - im, 2);
      ref += re * re + im * im;
    }
    worst = std::fmax(worst, std::sqrt(err / ref));
  }
  std::printf("%d %d %.3e\n", N, DIR, worst);
}
template <int... I> void all(std::integer_sequence<int, I...>) {
  (check<tw_size_at(I), -1>(), ...);
  (check<tw_size_at(I), +1>(), ...);
}
int main() { all(std::make_integer_sequence<int, kNumFftSizes>{}); }
