// Register DFTs: one thread holds the whole sequence.  Forward uses W = exp(-2 pi i / Q); inverse conjugates.
#pragma once
#include <math.h>

#include "pcb_internal.cuh"

namespace pcb {

// exp(-2 pi i k / 96), every root of the register DFTs (Q | 96), with a compile-time index: cos(2 pi k / 96),
// k = 0 .. 24, rounded to FP64, and the octant symmetries.  They fold into the instructions.
__device__ __forceinline__ constexpr double cos96(int k) {
  constexpr double c[25] = {
    1.0, 0.9978589232386035, 0.9914448613738104, 0.9807852804032304,
    0.9659258262890683, 0.9469301294951057, 0.9238795325112867, 0.8968727415326883,
    0.8660254037844386, 0.8314696123025452, 0.7933533402912352, 0.7518398074789774,
    0.7071067811865476, 0.6593458151000688, 0.6087614290087207, 0.5555702330196022,
    0.5, 0.4422886902190013, 0.3826834323650898, 0.3214394653031616,
    0.25881904510252074, 0.19509032201612828, 0.1305261922200516, 0.06540312923014306,
    0.0};
  return k <= 24 ? c[k] : k <= 48 ? -c[48 - k] : k <= 72 ? -c[k - 48] : c[96 - k];
}
template <typename R> __device__ __forceinline__ constexpr cx<R> root96(int k) {   // exp(-2 pi i k / 96)
  cx<R> w{};
  w.x = (R)cos96(k);
  w.y = (R)(k <= 72 ? -cos96((k + 72) % 96) : -cos96(k - 24));
  return w;
}

// exp(-2 pi i k / 64), 0 <= k < 64, with a compile-time index (the zeta = pi twist of the time lines)
__device__ __forceinline__ constexpr double cos64(int k) {
  constexpr double c[17] = {
    1.0, 0.9951847266721969, 0.9807852804032304, 0.9569403357322088,
    0.9238795325112867, 0.881921264348355, 0.8314696123025452, 0.773010453362737,
    0.7071067811865476, 0.6343932841636455, 0.5555702330196022, 0.47139673682599764,
    0.3826834323650898, 0.2902846772544624, 0.19509032201612828, 0.0980171403295606,
    0.0};
  return k <= 16 ? c[k] : -c[32 - k];
}
template <typename R> __device__ __forceinline__ constexpr cx<R> root64(int k) {
  cx<R> w{};
  const int j = k % 32;
  const double s = k < 32 ? 1.0 : -1.0;
  w.x = (R)(s * cos64(j));
  w.y = (R)(-s * (j <= 16 ? cos64(16 - j) : cos64(j - 16)));
  return w;
}

template <typename T>
__device__ __forceinline__ void r2(T& a, T& b) { T t = cadd(a, b); b = csub(a, b); a = t; }

template <typename T>
__device__ __forceinline__ void r4(T* a, bool inv) {
  T t0 = cadd(a[0], a[2]), t1 = csub(a[0], a[2]);
  T t2 = cadd(a[1], a[3]), t3 = csub(a[1], a[3]);
  t3 = inv ? cmul_pi(t3) : cmul_mi(t3);
  a[0] = cadd(t0, t2); a[2] = csub(t0, t2);
  a[1] = cadd(t1, t3); a[3] = csub(t1, t3);
}

template <typename T, typename R>
__device__ __forceinline__ void r3(T* a, bool inv) {
  const R s = (R)0.86602540378443864676;
  T t1 = cadd(a[1], a[2]), t2 = csub(a[1], a[2]);
  T m1 = csub(a[0], cscale(t1, (R)0.5));
  T st = cscale(t2, s);
  T ist = inv ? cmul_pi(st) : cmul_mi(st);
  a[0] = cadd(a[0], t1);
  a[1] = cadd(m1, ist);
  a[2] = csub(m1, ist);
}

template <typename T, typename R>
__device__ __forceinline__ void r8(T* a, bool inv) {
  T e[4] = {a[0], a[2], a[4], a[6]};
  T o[4] = {a[1], a[3], a[5], a[7]};
  r4(e, inv); r4(o, inv);
  const R h = (R)0.70710678118654752440;
  o[1] = cmul(o[1], mk<R>(h, inv ? h : -h));
  o[2] = inv ? cmul_pi(o[2]) : cmul_mi(o[2]);
  o[3] = cmul(o[3], mk<R>(-h, inv ? h : -h));
#pragma unroll
  for (int k = 0; k < 4; ++k) { a[k] = cadd(e[k], o[k]); a[k + 4] = csub(e[k], o[k]); }
}

// Primitive DFT of size Q on x[0..Q) in place, natural output order.
template <typename T, typename R, int Q>
__device__ __forceinline__ void prim(T* x, bool inv) {
  if (Q == 2) r2(x[0], x[1]);
  else if (Q == 3) r3<T, R>(x, inv);
  else if (Q == 4) r4(x, inv);
  else if (Q == 8) r8<T, R>(x, inv);
}

// Register DFT of size Q = A*B (A, B primitive) or primitive Q.  Output X[k] is left in
// register pos<Q>(k): identity for primitive sizes, (k / A) + B * (k % A) for composites.
template <int Q> struct Split { static constexpr int A = Q, B = 1; };
template <> struct Split<6> { static constexpr int A = 2, B = 3; };
template <> struct Split<12> { static constexpr int A = 4, B = 3; };
template <> struct Split<16> { static constexpr int A = 4, B = 4; };
template <> struct Split<24> { static constexpr int A = 8, B = 3; };
template <> struct Split<32> { static constexpr int A = 4, B = 8; };

template <int Q> __device__ __forceinline__ constexpr int pos(int k) {
  return Split<Q>::B == 1 ? k : (k / Split<Q>::A) + Split<Q>::B * (k % Split<Q>::A);
}

template <typename T, typename R, int Q>
__device__ __forceinline__ void reg_dft(T* x, bool inv) {
  constexpr int A = Split<Q>::A, B = Split<Q>::B;
  if constexpr (B == 1) {
    prim<T, R, Q>(x, inv);
  } else {
  // step 1: for each b, A-point DFT over x[b + B a]; result Y_b[k1] stays at x[b + B k1]
#pragma unroll
  for (int b = 0; b < B; ++b) {
    T t[A > 1 ? A : 1];
#pragma unroll
    for (int a = 0; a < A; ++a) t[a] = x[b + B * a];
    prim<T, R, A>(t, inv);
#pragma unroll
    for (int k1 = 0; k1 < A; ++k1) {
      T v = t[k1];
      if (b * k1) {
        const int k = (b * k1 * (96 / Q)) % 96;
        if (k == 24) {                       // a quarter turn is exact
          v = inv ? cmul_pi(v) : cmul_mi(v);
        } else {
          T w = root96<R>(k);
          if (inv) w.y = -w.y;
          v = cmul(v, w);
        }
      }
      x[b + B * k1] = v;
    }
  }
  // step 2: for each k1, B-point DFT over the contiguous chunk x[B k1 .. B k1 + B)
#pragma unroll
  for (int k1 = 0; k1 < A; ++k1) prim<T, R, B>(x + B * k1, inv);
  }
}

// DFT at the half frequencies (the twisted time lines): X[k] = sum_q x[q] exp(-i pi q (2k + 1) / A), both in
// natural order.  The first radix-2 step takes x[q] -/+ i x[q + A/2], and the twist and the step's twiddle
// are one factor per value: A - 2 complex products, where a twist before the plain DFT takes A - 1 and its
// first step's twiddles.  FP64 time pass at N = 191, n = 128 (no coupling): 0.52 -> 0.49 ms.
template <typename T, typename R, int A>
__device__ __forceinline__ void odd_dft(T* x) {
  constexpr int H = A / 2, S = 32 / A;
  T e[H], o[H];
#pragma unroll
  for (int q = 0; q < H; ++q) {
    const T b = cmul_mi(x[q + H]);
    e[q] = cadd(x[q], b);
    o[q] = csub(x[q], b);
    if (q) {
      e[q] = cmul(e[q], root64<R>(q * S));
      o[q] = cmul(o[q], root64<R>(3 * q * S));
    }
  }
  reg_dft<T, R, H>(e, false);
  reg_dft<T, R, H>(o, false);
#pragma unroll
  for (int k = 0; k < H; ++k) {
    x[2 * k] = e[pos<H>(k)];
    x[2 * k + 1] = o[pos<H>(k)];
  }
}
// its inverse without the factor 1/A
template <typename T, typename R, int A>
__device__ __forceinline__ void odd_idft(T* x) {
  constexpr int H = A / 2, S = 32 / A;
  T e[H], o[H];
#pragma unroll
  for (int k = 0; k < H; ++k) {
    e[k] = x[2 * k];
    o[k] = x[2 * k + 1];
  }
  reg_dft<T, R, H>(e, true);
  reg_dft<T, R, H>(o, true);
#pragma unroll
  for (int q = 0; q < H; ++q) {
    T a = e[pos<H>(q)], b = o[pos<H>(q)];
    if (q) {
      T w = root64<R>(q * S), v = root64<R>(3 * q * S);
      w.y = -w.y;
      v.y = -v.y;
      a = cmul(a, w);
      b = cmul(b, v);
    }
    x[q] = cadd(a, b);
    x[q + H] = cmul_pi(csub(a, b));
  }
}

}  // namespace pcb
