// N-point DFTs in registers with compile-time structure, for the line-resident plane kernels.
//
// Dft<T, N, SG, MK>::run(v) replaces v[n] by X[k] = sum_n v[n] exp(SG 2 pi i n k / N), natural order
// in and out (all index maps are compile-time, so a permutation costs nothing in registers). MK is
// the mask of inputs that can be non-zero: the inverse transforms of a plane see only |n| <= N/4,
// and a butterfly on a known zero is a copy. The outputs a caller does not use (the forward
// transforms' |n| > N/4) are removed by the compiler, since they are dead.
//
// Composite lengths: coprime factors by the prime-factor map (Good 1958, Thomas 1963; no twiddle
// factors), powers by Cooley-Tukey with constant twiddles. The power-of-two factor comes first in
// the inverse and last in the forward transform, where the zero inputs and dead outputs are.
//
// Double-float sums stay unnormalised inside a transform: 8 FP32 operations a sum instead of 11, 4 a
// product instead of 7; the caller renormalises what it stores. With u = 2^-24 and A the sum of the
// inputs' magnitudes, the low part after k steps in a row is at most (k + 1) u A (each step adds a
// rounding error of the leading parts, u A at most), so a step's own rounding, of the low parts, is at most
// 2 (k + 1) u^2 A and that of the whole transform about k^2 u^2 A: k is at most 15 for the 32 points a lane
// holds, 8e-13 A if every rounding went one way. Measured against 64-bit arithmetic, A_v x on 96^3 is off
// by 4.1e-15 and on 64^3 by 3.2e-15 of its largest component, as with sums renormalised throughout.
#pragma once

#include <utility>

#include "common.cuh"

namespace wdf {
namespace ld {

typedef unsigned long long u64;

// exp(2 pi i k / n) at compile time: Taylor series on an angle of at most pi / 4
struct CS {
  double c, s;
};
constexpr CS cs_small(double x) {
  double c = 1, s = x, tc = 1, ts = x;
  const double x2 = x * x;
  for (int i = 1; i < 14; ++i) {
    tc *= -x2 / ((2 * i - 1) * (2.0 * i));
    ts *= -x2 / ((2.0 * i) * (2 * i + 1));
    c += tc;
    s += ts;
  }
  return {c, s};
}
constexpr CS unit_root(int k, int n) {
  k %= n;
  if (k < 0) k += n;
  const int oct = (8 * k + n / 2 >= 0) ? (2 * (4 * k + n / 2) / (2 * n)) % 4 : 0;  // nearest multiple of pi / 2
  const double x = 6.283185307179586476925286766559 * ((double)(4 * k - oct * n) / (4.0 * n));
  const CS r = cs_small(4 * k - oct * n > 2 * n ? x - 6.283185307179586476925286766559 : x);
  return oct == 0 ? CS{r.c, r.s} : oct == 1 ? CS{-r.s, r.c} : oct == 2 ? CS{-r.c, -r.s} : CS{r.s, -r.c};
}

// Complex arithmetic per number type: CA<T>::C and the operations below (S, SG = +-1).
//   add, sub, neg           a + b, a - b, -a
//   addi<S>                 a + S i b
//   rmul, rfma, rdot2       a k, a k + b, a k + b l for real constants
//   half_neg                x - t / 2
//   twiddle                 a w, or a conj(w)
//   norm                    what a caller stores (double-float: renormalised)
template <typename T> struct CA {
  typedef cplx<T> C;
  static __device__ __forceinline__ C zero() { return mkc<T>(0, 0); }
  static __device__ __forceinline__ C add(C a, C b) { return mkc<T>(a.x + b.x, a.y + b.y); }
  static __device__ __forceinline__ C sub(C a, C b) { return mkc<T>(a.x - b.x, a.y - b.y); }
  static __device__ __forceinline__ C neg(C a) { return mkc<T>(-a.x, -a.y); }
  template <int S> static __device__ __forceinline__ C muli(C a) { return S > 0 ? mkc<T>(-a.y, a.x) : mkc<T>(a.y, -a.x); }
  template <int S> static __device__ __forceinline__ C addi(C a, C b) {
    return S > 0 ? mkc<T>(a.x - b.y, a.y + b.x) : mkc<T>(a.x + b.y, a.y - b.x);
  }
  static __device__ __forceinline__ C rmul(C a, double k) { return mkc<T>(a.x * (T)k, a.y * (T)k); }
  static __device__ __forceinline__ C rfma(C a, double k, C b) { return mkc<T>(a.x * (T)k + b.x, a.y * (T)k + b.y); }
  static __device__ __forceinline__ C rdot2(C a, double k, C b, double l) {
    return mkc<T>(a.x * (T)k + b.x * (T)l, a.y * (T)k + b.y * (T)l);
  }
  static __device__ __forceinline__ C half_neg(C x, C t) { return mkc<T>(x.x - (T)0.5 * t.x, x.y - (T)0.5 * t.y); }
  static __device__ __forceinline__ C cmulk(C a, double c, double s) {
    return mkc<T>(a.x * (T)c - a.y * (T)s, a.x * (T)s + a.y * (T)c);
  }
  static __device__ __forceinline__ C twiddle(C a, C w, bool conj) { return conj ? cmulc<T>(a, w) : cmul<T>(a, w); }
  static __device__ __forceinline__ C scale(C a, T f) { return cscal<T>(a, f); }
  static __device__ __forceinline__ C norm(C a) { return a; }
  static __device__ __forceinline__ C get(cplx<T> a) { return a; }
  static __device__ __forceinline__ cplx<T> put(C a) { return a; }
  // x1 = u + i S s d, x2 = u - i S s d
  template <int S> static __device__ __forceinline__ void pm_imul(C u, C d, double s, C &x1, C &x2) {
    const T k = (T)(S * s);
    x1 = mkc<T>(u.x - k * d.y, u.y + k * d.x);
    x2 = mkc<T>(u.x + k * d.y, u.y - k * d.x);
  }
  // x1 = e + w o, x2 = e - w o for w = (1 + S i) / sqrt 2 (FIRST) or (-1 + S i) / sqrt 2
  template <int S, bool FIRST> static __device__ __forceinline__ void pm_w8(C e, C o, C &x1, C &x2) {
    const T h = (T)0.70710678118654752440;
    const T dx = FIRST ? (S > 0 ? o.x - o.y : o.x + o.y) : (S > 0 ? -o.x - o.y : o.y - o.x);
    const T dy = FIRST ? (S > 0 ? o.y + o.x : o.y - o.x) : (S > 0 ? o.x - o.y : -o.y - o.x);
    x1 = mkc<T>(h * dx + e.x, h * dy + e.y);
    x2 = mkc<T>(e.x - h * dx, e.y - h * dy);
  }
};

// Double-float complex numbers as two packed pairs, (re, im) of the high and of the low parts: each
// FP32 operation of the error-free transformations runs on both parts in one packed instruction
// (add, mul and fma .rn.f32x2: two IEEE results, so the values are those of the scalar code). The
// FP32 pipe takes as long as for two scalar instructions, but a transform has about half the
// instructions: the scalar form of these kernels waited for instruction fetch (2.6 "no instruction"
// stalls per issue at 96 x 96). Multiplication by i swaps the halves of a pair; its signs ride
// on a fused multiply-add with a +-1 pair, which is exact.
struct pdf {
  u64 h, l;
};
static __constant__ u64 kNegZero2 = 0x8000000080000000ull;
__device__ __forceinline__ u64 pk(float a, float b) {
  u64 r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
  return r;
}
__device__ __forceinline__ float2 upk(u64 a) {
  float2 v;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(v.x), "=f"(v.y) : "l"(a));
  return v;
}
__device__ __forceinline__ u64 add2(u64 a, u64 b) {
  u64 r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ u64 sub2(u64 a, u64 b) {
  u64 r;
  asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ u64 fma2(u64 a, u64 b, u64 c) {
  u64 r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
  return r;
}
// a b as a fused multiply-add with a -0 that the compiler cannot see through: it fuses a packed mul
// that feeds a packed add into one operation, rounding mode notwithstanding, and the error-free
// transformations would lose the product's rounding error
__device__ __forceinline__ u64 mul2(u64 a, u64 b) {
  return fma2(a, b, kNegZero2);
}

// FP32 complex numbers as one packed pair: a complex sum is one instruction, a product by a constant
// or a twiddle two. The FP32 pipe takes as long as for the scalar pairs, but half of the issue slots go to
// the loads, swaps and address arithmetic beside it: the V_loc product 5-18% faster than with
// scalar arithmetic (64 x 64 .127 -> .111 ms, 75 x 75 .316 -> .267, 80 x 80 .346 -> .287 per 128 pairs).
template <> struct CA<float> {
  typedef u64 C;
  static __device__ __forceinline__ u64 swap(u64 a) {
    const float2 v = upk(a);
    return pk(v.y, v.x);
  }
  static __device__ __forceinline__ u64 both(double k) { return pk((float)k, (float)k); }
  static __device__ __forceinline__ u64 alt(double k) { return pk(-(float)k, (float)k); }  // i k on a swapped pair
  static __device__ __forceinline__ C zero() { return 0ull; }
  static __device__ __forceinline__ C get(float2 a) { return pk(a.x, a.y); }
  static __device__ __forceinline__ float2 put(C a) { return upk(a); }
  static __device__ __forceinline__ C add(C a, C b) { return add2(a, b); }
  static __device__ __forceinline__ C sub(C a, C b) { return sub2(a, b); }
  static __device__ __forceinline__ C neg(C a) { return pmul(a, both(-1.0)); }
  static __device__ __forceinline__ C pmul(C a, C b) {
    u64 r;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
  }
  template <int S> static __device__ __forceinline__ C muli(C a) { return pmul(swap(a), alt(S)); }
  template <int S> static __device__ __forceinline__ C addi(C a, C b) { return fma2(swap(b), alt(S), a); }
  static __device__ __forceinline__ C rmul(C a, double k) { return pmul(a, both(k)); }
  static __device__ __forceinline__ C rfma(C a, double k, C b) { return fma2(a, both(k), b); }
  static __device__ __forceinline__ C rdot2(C a, double k, C b, double l) { return fma2(a, both(k), pmul(b, both(l))); }
  static __device__ __forceinline__ C half_neg(C x, C t) { return fma2(t, both(-0.5), x); }
  static __device__ __forceinline__ C cmulk(C a, double c, double s) { return fma2(a, both(c), pmul(swap(a), alt(s))); }
  static __device__ __forceinline__ C twiddle(C a, C w, bool conj) {
    const float2 v = upk(w);
    const float s = conj ? -v.y : v.y;
    return fma2(a, pk(v.x, v.x), pmul(swap(a), pk(-s, s)));
  }
  static __device__ __forceinline__ C scale(C a, float f) { return pmul(a, pk(f, f)); }
  static __device__ __forceinline__ C norm(C a) { return a; }
  template <int S> static __device__ __forceinline__ void pm_imul(C u, C d, double s, C &x1, C &x2) {
    const C t = swap(d);
    x1 = fma2(t, alt(S * s), u);
    x2 = fma2(t, alt(-S * s), u);
  }
  template <int S, bool FIRST> static __device__ __forceinline__ void pm_w8(C e, C o, C &x1, C &x2) {
    const C v = addi<S>(o, o);  // (1 + S i) o
    const double h = 0.70710678118654752440;
    if (FIRST) {
      x1 = fma2(v, both(h), e);
      x2 = fma2(v, both(-h), e);
    } else {  // (-1 + S i) = S i (1 + S i)
      const C t = swap(v);
      x1 = fma2(t, alt(S * h), e);
      x2 = fma2(t, alt(-S * h), e);
    }
  }
};

template <> struct CA<df64> {
  typedef pdf C;
  static __device__ __forceinline__ u64 swap(u64 a) {
    const float2 v = upk(a);
    return pk(v.y, v.x);
  }
  static __device__ __forceinline__ C zero() { return C{0ull, 0ull}; }
  static __device__ __forceinline__ C get(cplx<df64> a) { return C{pk(a.x.hi, a.y.hi), pk(a.x.lo, a.y.lo)}; }
  static __device__ __forceinline__ cplx<df64> put(C a) {
    const float2 h = upk(a.h), l = upk(a.l);
    return mkc<df64>(df64(h.x, l.x), df64(h.y, l.y));
  }
  // TwoSum of the high parts, the low parts added in FP32 (no renormalisation)
  static __device__ __forceinline__ C add(C a, C b) {
    const u64 s = add2(a.h, b.h), bb = sub2(s, a.h);
    const u64 e = add2(sub2(a.h, sub2(s, bb)), sub2(b.h, bb));
    return C{s, add2(e, add2(a.l, b.l))};
  }
  static __device__ __forceinline__ C sub(C a, C b) {
    const u64 s = sub2(a.h, b.h), bb = sub2(a.h, s);  // bb: the part of b that went into s
    const u64 e = sub2(sub2(a.h, add2(s, bb)), sub2(b.h, bb));
    return C{s, add2(e, sub2(a.l, b.l))};
  }
  // a + f b for a pair f of +-1 or +-1/2 (exact products)
  static __device__ __forceinline__ C add_scaled(C a, u64 bh, u64 bl, u64 f) {
    const u64 s = fma2(bh, f, a.h), nb = sub2(a.h, s);
    const u64 e = add2(sub2(a.h, add2(s, nb)), fma2(bh, f, nb));
    return C{s, add2(e, fma2(bl, f, a.l))};
  }
  static __device__ __forceinline__ C neg(C a) {
    const u64 m = pk(-1.f, -1.f);
    return C{mul2(a.h, m), mul2(a.l, m)};
  }
  template <int S> static __device__ __forceinline__ C muli(C a) {
    const u64 f = pk(S > 0 ? -1.f : 1.f, S > 0 ? 1.f : -1.f);
    return C{mul2(swap(a.h), f), mul2(swap(a.l), f)};
  }
  template <int S> static __device__ __forceinline__ C addi(C a, C b) {
    return add_scaled(a, swap(b.h), swap(b.l), pk(S > 0 ? -1.f : 1.f, S > 0 ? 1.f : -1.f));
  }
  static __device__ __forceinline__ C half_neg(C x, C t) { return add_scaled(x, t.h, t.l, pk(-0.5f, -0.5f)); }
  // the products of the halves of a with the halves of (kh + kl), nkh = -kh; not renormalised
  static __device__ __forceinline__ C mulp(u64 h, u64 l, u64 kh, u64 nkh, u64 kl) {
    u64 e = fma2(h, kh, mul2(h, nkh));
    e = fma2(h, kl, e);
    return C{mul2(h, kh), fma2(l, kh, e)};
  }
  static constexpr float hi(double k) { return (float)k; }
  static constexpr float lo(double k) { return (float)(k - (double)(float)k); }
  static __device__ __forceinline__ C rmul(C a, double k) {
    return mulp(a.h, a.l, pk(hi(k), hi(k)), pk(-hi(k), -hi(k)), pk(lo(k), lo(k)));
  }
  static __device__ __forceinline__ C rfma(C a, double k, C b) { return add(rmul(a, k), b); }
  static __device__ __forceinline__ C rdot2(C a, double k, C b, double l) { return add(rmul(a, k), rmul(b, l)); }
  static __device__ __forceinline__ C cmulk(C a, double c, double s) {
    return add(rmul(a, c), mulp(swap(a.h), swap(a.l), pk(-hi(s), hi(s)), pk(hi(s), -hi(s)), pk(-lo(s), lo(s))));
  }
  static __device__ __forceinline__ C twiddle(C a, C w, bool conj) {
    const float2 h = upk(w.h), l = upk(w.l);
    const float sh = conj ? -h.y : h.y, sl = conj ? -l.y : l.y;
    return add(mulp(a.h, a.l, pk(h.x, h.x), pk(-h.x, -h.x), pk(l.x, l.x)),
               mulp(swap(a.h), swap(a.l), pk(-sh, sh), pk(sh, -sh), pk(-sl, sl)));
  }
  static __device__ __forceinline__ C norm(C a) {
    const u64 s = add2(a.h, a.l);
    return C{s, sub2(a.l, sub2(s, a.h))};
  }
  static __device__ __forceinline__ C scale(C a, df64 f) {
    return norm(mulp(a.h, a.l, pk(f.hi, f.hi), pk(-f.hi, -f.hi), pk(f.lo, f.lo)));
  }
  template <int S> static __device__ __forceinline__ void pm_imul(C u, C d, double s, C &x1, C &x2) {
    const C v = rmul(d, s);
    x1 = addi<S>(u, v);
    x2 = addi<-S>(u, v);
  }
  template <int S, bool FIRST> static __device__ __forceinline__ void pm_w8(C e, C o, C &x1, C &x2) {
    const C v = rmul(addi<S>(o, o), 0.70710678118654752440);  // (1 + S i) o / sqrt 2
    x1 = FIRST ? add(e, v) : addi<S>(e, v);                    // (-1 + S i) = S i (1 + S i)
    x2 = FIRST ? sub(e, v) : addi<-S>(e, v);
  }
};

// a exp(2 pi i K / N)
template <typename T, int K, int N> __device__ __forceinline__ typename CA<T>::C mulw(typename CA<T>::C a) {
  constexpr int k = ((K % N) + N) % N;
  if constexpr (k == 0) {
    return a;
  } else if constexpr (4 * k == N) {
    return CA<T>::template muli<1>(a);
  } else if constexpr (2 * k == N) {
    return CA<T>::neg(a);
  } else if constexpr (4 * k == 3 * N) {
    return CA<T>::template muli<-1>(a);
  } else {
    constexpr CS w = unit_root(k, N);
    return CA<T>::cmulk(a, w.c, w.s);
  }
}

template <int I, int E, typename F> __device__ __forceinline__ void static_for(F &&f) {
  if constexpr (I < E) {
    f(std::integral_constant<int, I>{});
    static_for<I + 1, E>(std::forward<F>(f));
  }
}

// masks of the inputs that can be non-zero: a predicate on the index
struct Full {
  static constexpr bool at(int) { return true; }
};
// the inputs n = S m + O (mod NT) of a length-NT line that can be non-zero, |n| <= XB, for any of
// the offsets O .. O + W - 1
template <int NT, int XB, int S, int O, int W = 1> struct Band {
  static constexpr bool at(int m) {
    for (int w = 0; w < W; ++w) {
      const int n = (S * m + O + w) % NT;
      if (n <= XB || n >= NT - XB) return true;
    }
    return false;
  }
};
// the inputs (S m + O) mod R of a mask
template <typename MK, int S, int O, int R> struct Sub {
  static constexpr bool at(int m) { return MK::at((S * m + O) % R); }
};
// entry m stands for the sub-transform of COUNT inputs Sub<MK, S, ., R> started at (O m) mod R
template <typename MK, int S, int O, int R, int COUNT> struct Any {
  static constexpr bool at(int m) {
    for (int i = 0; i < COUNT; ++i)
      if (MK::at((S * i + O * m) % R)) return true;
    return false;
  }
};

// the first factor of a composite length (the power of two first); 0: a base case
constexpr int first_factor(int n) {
  switch (n) {
    case 2: case 3: case 4: case 5: case 8: return 0;
    case 6: return 2;
    case 9: return 3;
    case 10: return 2;
    case 12: return 4;
    case 15: return 3;
    case 16: return 8;
    case 18: return 2;
    case 20: return 4;
    case 24: return 8;
    case 25: return 5;
    case 27: return 3;
    case 30: return 2;
    case 32: return 8;
    case 36: return 4;
    case 40: return 8;
    case 45: return 9;
    case 48: return 16;
    case 50: return 2;
    case 54: return 2;
    case 60: return 4;
    case 64: return 8;
    case 72: return 8;
    case 75: return 3;
    case 80: return 16;
    case 96: return 32;
    default: return -1;
  }
}
constexpr int gcd_of(int a, int b) { return b == 0 ? a : gcd_of(b, a % b); }
constexpr int inverse_mod(int a, int m) {
  int x = 1;
  while ((a * x) % m != 1 % m) ++x;
  return x;
}

template <typename T, int N, int SG, typename MK = Full> struct Dft {
  typedef CA<T> O;
  typedef typename O::C C;
  static __device__ __forceinline__ void run(C (&v)[N]) {
    if constexpr (N == 1) {
    } else if constexpr (N == 2) {
      if constexpr (MK::at(0) && MK::at(1)) {
        const C a = v[0], b = v[1];
        v[0] = O::add(a, b);
        v[1] = O::sub(a, b);
      } else if constexpr (MK::at(0)) {
        v[1] = v[0];
      } else if constexpr (MK::at(1)) {
        v[0] = v[1];
        v[1] = O::neg(v[1]);
      }
    } else if constexpr (N == 4) {
      C e[2] = {v[0], v[2]}, o[2] = {v[1], v[3]};
      Dft<T, 2, SG, Sub<MK, 2, 0, 4>>::run(e);
      Dft<T, 2, SG, Sub<MK, 2, 1, 4>>::run(o);
      combine<2>(v, e, o);
    } else if constexpr (N == 8) {
      C e[4] = {v[0], v[2], v[4], v[6]}, o[4] = {v[1], v[3], v[5], v[7]};
      Dft<T, 4, SG, Sub<MK, 2, 0, 8>>::run(e);
      Dft<T, 4, SG, Sub<MK, 2, 1, 8>>::run(o);
      combine<4>(v, e, o);
    } else if constexpr (N == 3) {
      if constexpr (!MK::at(1) && !MK::at(2)) {
        v[1] = v[0];
        v[2] = v[0];
      } else {
        const C t = MK::at(1) ? (MK::at(2) ? O::add(v[1], v[2]) : v[1]) : v[2];
        const C d = MK::at(1) ? (MK::at(2) ? O::sub(v[1], v[2]) : v[1]) : O::neg(v[2]);
        const C u = O::half_neg(v[0], t);
        v[0] = MK::at(0) ? O::add(v[0], t) : t;
        O::template pm_imul<SG>(u, d, 0.86602540378443864676, v[1], v[2]);
      }
    } else if constexpr (N == 5) {
      if constexpr (!MK::at(1) && !MK::at(2) && !MK::at(3) && !MK::at(4)) {
        v[1] = v[2] = v[3] = v[4] = v[0];
      } else {
        constexpr double c1 = 0.30901699437494742410, c2 = -0.80901699437494742410;
        constexpr double s1 = 0.95105651629515357212, s2 = 0.58778525229247312917;
        const C a1 = O::add(v[1], v[4]), a2 = O::add(v[2], v[3]), b1 = O::sub(v[1], v[4]), b2 = O::sub(v[2], v[3]);
        const C p = O::rfma(a1, c1, O::rfma(a2, c2, v[0])), q = O::rfma(a1, c2, O::rfma(a2, c1, v[0]));
        const C u = O::rdot2(b1, s1, b2, s2), w = O::rdot2(b1, s2, b2, -s1);
        v[0] = O::add(v[0], O::add(a1, a2));
        v[1] = O::template addi<SG>(p, u);
        v[4] = O::template addi<-SG>(p, u);
        v[2] = O::template addi<SG>(q, w);
        v[3] = O::template addi<-SG>(q, w);
      }
    } else {
      constexpr int F = first_factor(N);
      static_assert(F > 1, "length without a factorisation");
      // inverse: factor F first; forward: last
      constexpr int A = SG > 0 ? F : N / F, B = N / A;
      if constexpr (gcd_of(A, B) == 1) pfa<A, B>(v);
      else ct<A, B>(v);
    }
  }

 private:
  // radix-2 combination of two half-length transforms, X[k] = e[k] + w^k o[k], w = exp(SG 2 pi i / 2H)
  template <int H> static __device__ __forceinline__ void combine(C (&v)[N], const C (&e)[H], const C (&o)[H]) {
    constexpr bool he = any(0), ho = any(1);
    static_for<0, H>([&](auto kk) {
      constexpr int k = kk();
      if constexpr (!ho) {
        v[k] = e[k];
        v[k + H] = e[k];
      } else if constexpr (he && 2 * k == H) {  // w = SG i
        v[k] = O::template addi<SG>(e[k], o[k]);
        v[k + H] = O::template addi<-SG>(e[k], o[k]);
      } else if constexpr (he && H == 4 && k % 2 == 1) {
        O::template pm_w8<SG, k == 1>(e[k], o[k], v[k], v[k + H]);
      } else {
        const C w = mulw<T, SG * k, 2 * H>(o[k]);
        if constexpr (he) {
          v[k] = O::add(e[k], w);
          v[k + H] = O::sub(e[k], w);
        } else {
          v[k] = w;
          v[k + H] = O::neg(w);
        }
      }
    });
  }
  static constexpr bool any(int parity) {
    for (int i = parity; i < N; i += 2)
      if (MK::at(i)) return true;
    return false;
  }
  // coprime A B: input n = (B n1 + A n2) mod N, output k = (B (B^-1 mod A) k1 + A (A^-1 mod B) k2) mod N
  template <int A, int B> static __device__ __forceinline__ void pfa(C (&v)[N]) {
    constexpr int cA = B * inverse_mod(B % A, A), cB = A * inverse_mod(A % B, B);
    C a[B][A];
    static_for<0, B>([&](auto j) {
      constexpr int n2 = j();
      static_for<0, A>([&](auto i) { a[n2][i()] = v[(B * i() + A * n2) % N]; });
      Dft<T, A, SG, Sub<MK, B, A * n2, N>>::run(a[n2]);
    });
    static_for<0, A>([&](auto i) {
      constexpr int k1 = i();
      C b[B];
      static_for<0, B>([&](auto j) { b[j()] = a[j()][k1]; });
      Dft<T, B, SG, Any<MK, B, A, N, A>>::run(b);
      static_for<0, B>([&](auto j) { v[(cA * k1 + cB * j()) % N] = b[j()]; });
    });
  }
  // Cooley-Tukey: n = n2 + B n1, k = k1 + A k2
  template <int A, int B> static __device__ __forceinline__ void ct(C (&v)[N]) {
    C a[B][A];
    static_for<0, B>([&](auto j) {
      constexpr int n2 = j();
      static_for<0, A>([&](auto i) { a[n2][i()] = v[n2 + B * i()]; });
      Dft<T, A, SG, Sub<MK, B, n2, N>>::run(a[n2]);
      static_for<1, A>([&](auto i) { a[n2][i()] = mulw<T, SG * n2 * i(), N>(a[n2][i()]); });
    });
    static_for<0, A>([&](auto i) {
      constexpr int k1 = i();
      C b[B];
      static_for<0, B>([&](auto j) { b[j()] = a[j()][k1]; });
      Dft<T, B, SG, Any<MK, B, 1, N, A>>::run(b);
      static_for<0, B>([&](auto j) { v[k1 + A * j()] = b[j()]; });
    });
  }
};

}  // namespace ld
}  // namespace wdf
