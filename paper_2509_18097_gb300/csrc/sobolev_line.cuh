// Line transforms of the grid Sobolev preconditioner (Sec. 3.2, Eq. 3): DCT-II and its
// inverse of n = 2^a 3^b <= 256 points, two real lines at a time.
//
// Two lines are packed as the real and imaginary parts of one complex sequence after the
// even/odd reordering that turns a DCT-II into a DFT (valid for odd n too).  The complex FFT is
// a two-stage Cooley-Tukey split n = N1 x N2: N1 register DFTs of N2 points, twiddles, an
// exchange through shared memory, N2 register DFTs of N1 points.  A block transforms P line
// pairs together; a work item is one register DFT of one pair, with the pair index fastest
// across the lanes, so every shared-memory access of the stages is a contiguous row of pairs.
//
// Shared rows.  Position e of a line and frequency k are row e and row k.  Forward, stage 1 item t
// (of N1) takes x[j], j = t + N1 m, and leaves its N2 outputs in rows N2 t + k2; stage 2 item k2
// (of N2) rewrites rows k2 + N2 t in place, which puts the spectrum in natural order.  The inverse
// runs the same split backwards: N2 items of N1 points in place, then N1 items of N2 points.
// Twiddles come from a per-level table laid out so that an item's N2 (or N1) factors are at
// compile-time offsets from one pointer: twm[k2 N1 + t] = exp(-2 pi i t k2 / n).
#pragma once
#include <utility>

#include "kernels.h"

namespace pdg {

// ------------------------------------------------------------------------------ constants

// cos / sin of 2 pi k / n at compile time: the Taylor series at an angle in (-pi, pi], where 30
// terms are far below double rounding
__host__ __device__ constexpr double series_cos(double x) {
  double s = 1.0, t = 1.0;
  for (int i = 1; i < 30; ++i) {
    t *= -x * x / ((2 * i - 1) * (2 * i));
    s += t;
  }
  return s;
}
__host__ __device__ constexpr double series_sin(double x) {
  double s = x, t = x;
  for (int i = 1; i < 30; ++i) {
    t *= -x * x / ((2 * i) * (2 * i + 1));
    s += t;
  }
  return s;
}
__host__ __device__ constexpr double turn(int k, int n) {
  const int r = ((k % n) + n) % n;
  return 6.283185307179586476925 * (2 * r > n ? r - n : r) / n;
}

// threadIdx.x, opaque to the compiler: the kernels switch over the level sizes inside their item
// loop, and hoisting every size's thread-dependent addresses out of it spills registers
__device__ __forceinline__ int thread_here() {
  int t;
  asm volatile("mov.u32 %0, %%tid.x;" : "=r"(t));
  return t;
}

template <class F, int... I>
__device__ __forceinline__ void sfor_seq(F&& f, std::integer_sequence<int, I...>) {
  (f(std::integral_constant<int, I>{}), ...);
}
// f(0), f(1), .. f(N - 1) with the index a compile-time constant
template <int N, class F>
__device__ __forceinline__ void sfor(F&& f) {
  sfor_seq(static_cast<F&&>(f), std::make_integer_sequence<int, N>{});
}

__device__ __forceinline__ float2 cadd(float2 a, float2 b) { return make_float2(a.x + b.x, a.y + b.y); }
__device__ __forceinline__ float2 csub(float2 a, float2 b) { return make_float2(a.x - b.x, a.y - b.y); }
__device__ __forceinline__ float2 cmulf(float2 a, float2 b) {
  return make_float2(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x);
}

// a times exp(-2 pi i K / N) (forward) or its conjugate (INV)
template <int K, int N, bool INV>
__device__ __forceinline__ float2 cmul_const(float2 a) {
  constexpr int k = K % N;
  if constexpr (k == 0) return a;
  else if constexpr (2 * k == N) return make_float2(-a.x, -a.y);
  else if constexpr (4 * k == N) return INV ? make_float2(-a.y, a.x) : make_float2(a.y, -a.x);
  else if constexpr (4 * k == 3 * N) return INV ? make_float2(a.y, -a.x) : make_float2(-a.y, a.x);
  else {
    constexpr float c = (float)series_cos(turn(k, N));
    constexpr float s = (float)(INV ? series_sin(turn(k, N)) : -series_sin(turn(k, N)));
    return make_float2(a.x * c - a.y * s, a.x * s + a.y * c);
  }
}

// k < A B with k = i mod A and k = b mod B (A, B coprime)
__host__ __device__ constexpr int crt(int A, int B, int i, int b) {
  int k = i;
  while (k % B != b) k += A;
  return k;
}

// DFT of R = 2^a 3^b points in registers, natural order in and out.  Coprime factors are taken
// without twiddles (the Good-Thomas prime-factor map): fewer roundings, RMS error of a 36-point line
// 8.3e-8 with twiddles, 7.5e-8 without.
template <int R, bool INV>
__device__ __forceinline__ void dft(float2 (&a)[R]) {
  if constexpr (R == 2) {
    const float2 t = a[1];
    a[1] = csub(a[0], t);
    a[0] = cadd(a[0], t);
  } else if constexpr (R == 3) {
    constexpr float h = INV ? -0.866025403784438647f : 0.866025403784438647f;
    const float2 s = cadd(a[1], a[2]), d = csub(a[1], a[2]);
    const float2 m = make_float2(a[0].x - 0.5f * s.x, a[0].y - 0.5f * s.y);
    a[0] = cadd(a[0], s);
    a[1] = make_float2(m.x + h * d.y, m.y - h * d.x);
    a[2] = make_float2(m.x - h * d.y, m.y + h * d.x);
  } else if constexpr (R == 4) {
    const float2 s0 = cadd(a[0], a[2]), d0 = csub(a[0], a[2]), s1 = cadd(a[1], a[3]), d1 = csub(a[1], a[3]);
    a[0] = cadd(s0, s1);
    a[2] = csub(s0, s1);
    const float2 r = INV ? make_float2(-d1.y, d1.x) : make_float2(d1.y, -d1.x);  // +-i d1
    a[1] = cadd(d0, r);
    a[3] = csub(d0, r);
  } else if constexpr (R % 6 == 0) {
    constexpr int A = R & -R, B = R / A;
    float2 y[A][B];
#pragma unroll
    for (int b = 0; b < B; ++b) {
      float2 t[A];
#pragma unroll
      for (int i = 0; i < A; ++i) t[i] = a[(B * i + A * b) % R];
      dft<A, INV>(t);
#pragma unroll
      for (int i = 0; i < A; ++i) y[i][b] = t[i];
    }
    sfor<A>([&](auto ic) {
      constexpr int i = decltype(ic)::value;
      dft<B, INV>(y[i]);
      sfor<B>([&](auto bc) {
        constexpr int b = decltype(bc)::value;
        a[crt(A, B, i, b)] = y[i][b];
      });
    });
  } else if constexpr (R > 4) {
    constexpr int A = R % 4 == 0 ? 4 : 3, B = R / A;
    static_assert(A * B == R, "R = 2^a 3^b");
    float2 y[A][B];
    sfor<B>([&](auto bc) {
      constexpr int b = decltype(bc)::value;
      float2 t[A];
#pragma unroll
      for (int i = 0; i < A; ++i) t[i] = a[b + B * i];
      dft<A, INV>(t);
      sfor<A>([&](auto ic) {
        constexpr int i = decltype(ic)::value;
        y[i][b] = cmul_const<b * i, R, INV>(t[i]);
      });
    });
#pragma unroll
    for (int i = 0; i < A; ++i) {
      dft<B, INV>(y[i]);
#pragma unroll
      for (int b = 0; b < B; ++b) a[i + A * b] = y[i][b];
    }
  }
}

// ------------------------------------------------------------------------------ sizes

template <int n>
struct Fac {
  static constexpr int N1 = line_n1(n), N2 = n / N1;
  static_assert(N1 * N2 == n, "factors");
};

// e with x[e] = v[j] at j = t + N1 m (t < N1): the even elements in order, then the odd ones
// backwards.  With N2 even the half is decided by m alone, so e is t times a constant plus one.
template <int n>
__device__ __forceinline__ int esrc(int t, int m) {
  constexpr int N1 = Fac<n>::N1, N2 = Fac<n>::N2;
  const int j = t + N1 * m;
  if (N2 % 2 == 0 ? m < N2 / 2 : 2 * j < n) return 2 * j;
  return 2 * (n - 1 - j) + 1;
}

// The z-planes of a level from the first with an active vertex to the last: (first, count); all of
// them without a mask.  By warp 0 of a block; the caller synchronises.
__device__ __forceinline__ void z_range(const Level& lv, int2* out) {
  if (threadIdx.x >= 32) return;
  int lo = lv.n, hi = -1;
  for (int z = threadIdx.x; z < lv.n; z += 32)
    if (!lv.zmask || __ldg(lv.zmask + z)) {
      lo = min(lo, z);
      hi = z;
    }
  lo = __reduce_min_sync(0xffffffffu, lo);
  hi = __reduce_max_sync(0xffffffffu, hi);
  if (threadIdx.x == 0) *out = make_int2(hi < 0 ? 0 : lo, hi < 0 ? 0 : hi - lo + 1);
}

// ------------------------------------------------------------------------------ stages

// FFT stages over the block's P line pairs; a thread keeps one pair (P divides THREADS) and
// takes items it0, it0 + THREADS / P, ..; S: float2 between rows, sm points at the pair.
// First stage of the forward transform on item t's values: DFT, twiddles, rows N2 t + k.
template <int n, int S>
__device__ __forceinline__ void fwd_stage1(float2 (&v)[Fac<n>::N2], float2* sm, int t, const float2* __restrict__ twm) {
  constexpr int N1 = Fac<n>::N1, N2 = Fac<n>::N2;
  dft<N2, false>(v);
  float2* o = sm + N2 * t * S;
  const float2* w = twm + t;
  o[0] = v[0];
#pragma unroll
  for (int k = 1; k < N2; ++k) o[k * S] = N1 > 1 ? cmulf(v[k], __ldg(w + k * N1)) : v[k];
}

template <int n, int S, int STEP>
__device__ __forceinline__ void fwd_stage2(float2* sm, int it0) {
  constexpr int N1 = Fac<n>::N1, N2 = Fac<n>::N2;
  if constexpr (N1 > 1)
#pragma unroll 1
    for (int k2 = it0; k2 < N2; k2 += STEP) {
      float2 v[N1];
      float2* r = sm + k2 * S;
#pragma unroll
      for (int t = 0; t < N1; ++t) v[t] = r[N2 * t * S];
      dft<N1, false>(v);
#pragma unroll
      for (int k = 0; k < N1; ++k) r[N2 * k * S] = v[k];
    }
}

template <int n, int S, int STEP>
__device__ __forceinline__ void inv_stage1(float2* sm, int it0, const float2* __restrict__ twm) {
  constexpr int N1 = Fac<n>::N1, N2 = Fac<n>::N2;
  if constexpr (N1 > 1)
#pragma unroll 1
    for (int t = it0; t < N2; t += STEP) {
      float2 v[N1];
      float2* r = sm + t * S;
      const float2* w = twm + t * N1;
#pragma unroll
      for (int m = 0; m < N1; ++m) v[m] = r[N2 * m * S];
      dft<N1, true>(v);
      r[0] = v[0];
#pragma unroll
      for (int k = 1; k < N1; ++k) {
        const float2 c = __ldg(w + k);
        r[N2 * k * S] = cmulf(v[k], make_float2(c.x, -c.y));
      }
    }
}

// Last stage of the inverse: item k's values, v[s] at position esrc(k, s)
template <int n, int S>
__device__ __forceinline__ void inv_stage2(float2 (&v)[Fac<n>::N2], const float2* sm, int k) {
  constexpr int N2 = Fac<n>::N2;
#pragma unroll
  for (int s = 0; s < N2; ++s) v[s] = sm[(N2 * k + s) * S];
  dft<N2, true>(v);
}

// ------------------------------------------------------------------------------ DCT ends

// Separates the two packed spectra: from Z_q and Z_{n-q}, X_A and X_B at q and at n - q.
// V_A = (Z_q + conj Z_{n-q}) / 2, V_B = (Z_q - conj Z_{n-q}) / 2i, X_q = Re(w V), and since
// w_{n-q} = -i conj(w_q) and V_{n-q} = conj(V_q), X_{n-q} = -Im(w V); w = exp(-i pi q / 2n).
__device__ __forceinline__ void dct2_ends(float2 zq, float2 zn, float2 w, float2& xq, float2& xn) {
  const float2 va = make_float2(0.5f * (zq.x + zn.x), 0.5f * (zq.y - zn.y));
  const float2 vb = make_float2(0.5f * (zq.y + zn.y), -0.5f * (zq.x - zn.x));
  const float2 ua = cmulf(w, va), ub = cmulf(w, vb);
  xq = make_float2(ua.x, ub.x);
  xn = make_float2(-ua.y, -ub.y);
}

// The inverse's input from the spectra (X_A, X_B) at q and n - q (0 there for q = 0):
// V_q = conj(w) (X_q - i X_{n-q}), V_{n-q} = conj(V_q), Z = V_A + i V_B.
__device__ __forceinline__ void dct3_ends(float2 xq, float2 xn, float2 w, float2& zq, float2& zn) {
  const float2 va = make_float2(w.x * xq.x - w.y * xn.x, -w.y * xq.x - w.x * xn.x);
  const float2 vb = make_float2(w.x * xq.y - w.y * xn.y, -w.y * xq.y - w.x * xn.y);
  zq = make_float2(va.x - vb.y, va.y + vb.x);
  zn = make_float2(va.x + vb.y, vb.x - va.y);
}

}  // namespace pdg
