// Two lines at once in FP32: f2 holds the same value of two lines, and its arithmetic is the
// packed add / sub / mul / fma on two floats (one issue for two operations; the scalar transforms
// of the co-densities were bound by issue slots and by shared-memory accesses, not by the FP32
// lanes).  The line FFT is the compile-time form of fixed.cuh.
#pragma once
#include <cstring>

#include "fixed.cuh"

namespace ltmp2 {

struct f2 { unsigned long long v; };   // the two floats, the first in the low half

__host__ __device__ __forceinline__ f2 f2_make(float a, float b) {
#ifdef __CUDA_ARCH__
  f2 r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r.v) : "f"(a), "f"(b));
  return r;
#else
  unsigned lo, hi;
  std::memcpy(&lo, &a, 4);
  std::memcpy(&hi, &b, 4);
  return {(unsigned long long)hi << 32 | lo};
#endif
}
__host__ __device__ __forceinline__ void f2_get(f2 r, float &a, float &b) {
#ifdef __CUDA_ARCH__
  asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(r.v));
#else
  const unsigned lo = (unsigned)r.v, hi = (unsigned)(r.v >> 32);
  std::memcpy(&a, &lo, 4);
  std::memcpy(&b, &hi, 4);
#endif
}
#ifdef __CUDA_ARCH__
#define LTMP2_F2_BODY(ptx, expr)                                                                     \
  f2 r;                                                                                              \
  asm(ptx ".rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(u.v), "l"(v.v));                                 \
  return r;
#else
#define LTMP2_F2_BODY(ptx, expr)                                                                     \
  float a, b, c, d;                                                                                  \
  f2_get(u, a, b);                                                                                   \
  f2_get(v, c, d);                                                                                   \
  return f2_make(a expr c, b expr d);
#endif
__host__ __device__ __forceinline__ f2 operator+(f2 u, f2 v) { LTMP2_F2_BODY("add", +) }
__host__ __device__ __forceinline__ f2 operator-(f2 u, f2 v) { LTMP2_F2_BODY("sub", -) }
__host__ __device__ __forceinline__ f2 operator*(f2 u, f2 v) { LTMP2_F2_BODY("mul", *) }
#undef LTMP2_F2_BODY
// c v + w for one c
__host__ __device__ __forceinline__ f2 f2_fma(float c, f2 v, f2 w) {
#ifdef __CUDA_ARCH__
  f2 r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r.v) : "l"(f2_make(c, c).v), "l"(v.v), "l"(w.v));
  return r;
#else
  float a, b, d, e;
  f2_get(v, a, b);
  f2_get(w, d, e);
  return f2_make(fmaf(c, a, d), fmaf(c, b, e));
#endif
}
__host__ __device__ __forceinline__ f2 f2_mul(float c, f2 v) { return f2_make(c, c) * v; }

// one 128-bit access to shared memory (left to the compiler it becomes two of 64 bits, which conflict
// two ways)
__device__ __forceinline__ cpx<f2> f2_load(const cpx<f2> *p) {
  cpx<f2> r;
  asm volatile("ld.shared.v2.b64 {%0, %1}, [%2];" : "=l"(r.x.v), "=l"(r.y.v) : "r"((unsigned)__cvta_generic_to_shared(p)) : "memory");
  return r;
}
__device__ __forceinline__ void f2_store(cpx<f2> *p, cpx<f2> v) {
  asm volatile("st.shared.v2.b64 [%0], {%1, %2};" ::"r"((unsigned)__cvta_generic_to_shared(p)), "l"(v.x.v), "l"(v.y.v) : "memory");
}

// cos / sin of 2 pi e / n, rounded from 2^-62
constexpr float f2_cosn(int e, int n) { return (float)((double)(long long)fxc::cosn(e, n) / 4611686018427387904.0); }
constexpr float f2_sinn(int e, int n) { return (float)((double)(long long)fxc::sinn(e, n) / 4611686018427387904.0); }

// v + c (DIR i) u
template <int DIR> __host__ __device__ __forceinline__ cpx<f2> f2_add_i(float c, cpx<f2> u, cpx<f2> v) {
  return {f2_fma(-DIR * c, u.y, v.x), f2_fma(DIR * c, u.x, v.y)};
}

template <int DIR> struct Radix<f2, 4, DIR> {
  typedef cpx<f2> C;
  static __host__ __device__ __forceinline__ void run(C (&v)[4]) {
    const C s02 = cadd(v[0], v[2]), d02 = csub(v[0], v[2]), s13 = cadd(v[1], v[3]), d = csub(v[1], v[3]);
    v[0] = cadd(s02, s13);
    v[2] = csub(s02, s13);
    const C p = {d02.x + d.y, d02.y - d.x}, q = {d02.x - d.y, d02.y + d.x};
    v[1] = DIR < 0 ? p : q;
    v[3] = DIR < 0 ? q : p;
  }
};
template <int DIR> struct Radix<f2, 3, DIR> {
  typedef cpx<f2> C;
  static __host__ __device__ __forceinline__ void run(C (&v)[3]) {
    constexpr float s3 = f2_sinn(1, 3);
    const C t = cadd(v[1], v[2]), d = csub(v[1], v[2]);
    const C m = {f2_fma(-0.5f, t.x, v[0].x), f2_fma(-0.5f, t.y, v[0].y)};
    v[0] = cadd(v[0], t);
    v[1] = f2_add_i<DIR>(s3, d, m);
    v[2] = f2_add_i<-DIR>(s3, d, m);
  }
};
template <int DIR> struct Radix<f2, 5, DIR> {
  typedef cpx<f2> C;
  static __host__ __device__ __forceinline__ C two(float c, C u, float d, C v) {   // c u + d v
    return {f2_fma(c, u.x, f2_mul(d, v.x)), f2_fma(c, u.y, f2_mul(d, v.y))};
  }
  static __host__ __device__ __forceinline__ void run(C (&v)[5]) {
    constexpr float c1 = f2_cosn(1, 5), c2 = f2_cosn(2, 5), s1 = f2_sinn(1, 5), s2 = f2_sinn(2, 5);
    const C t1 = cadd(v[1], v[4]), t2 = cadd(v[2], v[3]), t3 = csub(v[1], v[4]), t4 = csub(v[2], v[3]);
    const C b1 = {f2_fma(c1, t1.x, f2_fma(c2, t2.x, v[0].x)), f2_fma(c1, t1.y, f2_fma(c2, t2.y, v[0].y))};
    const C b2 = {f2_fma(c2, t1.x, f2_fma(c1, t2.x, v[0].x)), f2_fma(c2, t1.y, f2_fma(c1, t2.y, v[0].y))};
    const C q1 = two(s1, t3, s2, t4), q2 = two(s2, t3, -s1, t4);
    v[0] = cadd(v[0], cadd(t1, t2));
    const C p1 = {b1.x + q1.y, b1.y - q1.x}, m1 = {b1.x - q1.y, b1.y + q1.x};
    const C p2 = {b2.x + q2.y, b2.y - q2.x}, m2 = {b2.x - q2.y, b2.y + q2.x};
    v[1] = DIR < 0 ? p1 : m1;
    v[4] = DIR < 0 ? m1 : p1;
    v[2] = DIR < 0 ? p2 : m2;
    v[3] = DIR < 0 ? m2 : p2;
  }
};

template <int NT, int E, int DIR> __host__ __device__ __forceinline__ cpx<f2> ct_twiddle(cpx<f2> v) {
  constexpr int e = E % NT;
  if constexpr (e == 0) {
    return v;
  } else if constexpr ((4 * e) % NT == 0) {
    constexpr int q = DIR > 0 ? (4 * e) / NT : 4 - (4 * e) / NT;   // times i^q
    if constexpr (q == 1) return {f2_mul(-1.0f, v.y), v.x};
    else if constexpr (q == 2) return {f2_mul(-1.0f, v.x), f2_mul(-1.0f, v.y)};
    else return {v.y, f2_mul(-1.0f, v.x)};
  } else if constexpr (e * 8 == NT || e * 8 == 3 * NT) {
    // (+-1 +- i) sqrt(1/2): the sum and the difference, scaled
    constexpr float r = f2_sinn(1, 8);
    constexpr float c = e * 8 == NT ? r : -r, s = DIR > 0 ? r : -r;
    // c x - s y, s x + c y with |c| = |s|
    const f2 p = v.x + v.y, m = v.x - v.y;
    if constexpr (c > 0 && s > 0) return {f2_mul(r, m), f2_mul(r, p)};
    else if constexpr (c > 0) return {f2_mul(r, p), f2_mul(-r, m)};
    else if constexpr (s > 0) return {f2_mul(-r, p), f2_mul(r, m)};
    else return {f2_mul(-r, m), f2_mul(-r, p)};
  } else {
    constexpr float c = f2_cosn(e, NT), s = DIR * f2_sinn(e, NT);
    return {f2_fma(c, v.x, f2_mul(-s, v.y)), f2_fma(s, v.x, f2_mul(c, v.y))};
  }
}

template <int N, int DIR, int NT> struct LineFFT<f2, N, DIR, NT> : CtLineFFT<f2, N, DIR> {};

}  // namespace ltmp2
