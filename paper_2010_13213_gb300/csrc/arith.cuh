// arith.cuh -- complex arithmetic in registers for the line transforms (lines.cuh).
//
// Ar<R> is a complex value V of the arithmetic R with the operations the transforms are written in, the
// memory form M of a V, a twiddle T and a real coefficient C:
//   float   V, M = one register pair (re, im); every operation is a packed f32x2 instruction;
//   df      V = two register pairs, h = (re.hi, im.hi) and l = (re.lo, im.lo): the two error-free chains of a
//           double-float complex operation run as one packed f32x2 chain;
//   double  V = (re, im).
// The packed instructions issue half as often for the same FP32 lanes.  A 16-point double-float FFT in
// registers (16 warps per SM) measured 1,480 clocks per warp packed against 1,731 as scalar chains: 91 % of
// the FP32 pipe instead of 80 %.
//
// Double-float sums and real products are left unnormalised (lazy: TwoSum of the high parts, plain sums of the low
// parts); callers renormalise (norm) before a value enters a complex product, which renormalises its result.  ArFine
// renormalises every sum.  Products by i swap the halves of a pair, with the sign folded into an exact multiply by
// (+1, -1) inside the following sum.
#pragma once
#include "common.cuh"

namespace lgf {

typedef unsigned long long f2;  // two packed floats

LGF_D f2 f2_pack(float a, float b) {
  f2 r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
  return r;
}
LGF_D void f2_unpack(f2 v, float &a, float &b) { asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(v)); }
LGF_D f2 f2_swap(f2 v) {
  float a, b;
  f2_unpack(v, a, b);
  return f2_pack(b, a);
}
LGF_D f2 f2_add(f2 a, f2 b) {
  f2 r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
LGF_D f2 f2_sub(f2 a, f2 b) {
  f2 r;
  asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
LGF_D f2 f2_mul(f2 a, f2 b) {
  f2 r;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
LGF_D f2 f2_fma(f2 a, f2 b, f2 c) {
  f2 r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
  return r;
}
LGF_D f2 f2_neg(f2 a) { return a ^ 0x8000000080000000ull; }
#define LGF_F2_PM 0xbf8000003f800000ull   // (+1, -1)
#define LGF_F2_MP 0x3f800000bf800000ull   // (-1, +1)
#define LGF_F2_MH 0xbf000000bf000000ull   // (-1/2, -1/2)

template <class R>
struct Ar;

// ------------------------------------------------------------------ double
template <>
struct Ar<double> {
  typedef double Real;
  struct V {
    double re, im;
  };
  typedef double2 M;
  typedef double2 T;  // (cos, -sin) of a forward twiddle
  static LGF_D V make(double re, double im) { return {re, im}; }
  static LGF_D double re(V a) { return a.re; }
  static LGF_D double im(V a) { return a.im; }
  static LGF_D V zero() { return {0.0, 0.0}; }
  static LGF_D V ld(const M *p) {
    const double2 v = *p;
    return {v.x, v.y};
  }
  static LGF_D void st(M *p, V a) { *p = make_double2(a.re, a.im); }
  static LGF_D V conj(V a) { return {a.re, -a.im}; }
  static LGF_D V add(V a, V b) { return {a.re + b.re, a.im + b.im}; }
  static LGF_D V sub(V a, V b) { return {a.re - b.re, a.im - b.im}; }
  static LGF_D V add_mi(V a, V b) { return {a.re + b.im, a.im - b.re}; }  // a - i b
  static LGF_D V add_pi(V a, V b) { return {a.re - b.im, a.im + b.re}; }  // a + i b
  static LGF_D V add_mh(V a, V b) { return {fma(-0.5, b.re, a.re), fma(-0.5, b.im, a.im)}; }  // a - b / 2
  static LGF_D V mul(V a, T w) { return {a.re * w.x - a.im * w.y, a.re * w.y + a.im * w.x}; }
  static LGF_D V swap(V a) { return {a.im, a.re}; }
  // acc + w.re a, and acc + i w.im v for s = swap(v)
  static LGF_D V fma_re(V acc, V a, T w) { return {fma(w.x, a.re, acc.re), fma(w.x, a.im, acc.im)}; }
  static LGF_D V fma_im(V acc, V s, T w) { return {fma(-w.y, s.re, acc.re), fma(w.y, s.im, acc.im)}; }
  static LGF_D V mul_im(V s, T w) { return {-w.y * s.re, w.y * s.im}; }  // i w.im v for s = swap(v)
  static LGF_D V mul_w8(V v, T w) {  // v e^{-i pi/4}, w.x = cos(pi/4)
    return {w.x * (v.re + v.im), w.x * (v.im - v.re)};
  }
  static LGF_D V norm(V a) { return a; }
  static LGF_D V scale_conj(V a, double g) { return {a.re * g, -(a.im * g)}; }
};

// ------------------------------------------------------------------ float
template <>
struct Ar<float> {
  typedef float Real;
  struct V {
    f2 v;
  };
  typedef f2 M;
  struct alignas(16) T {
    f2 re, im;  // (c, c) and (s, -s) for the forward twiddle c - i s: (-w.im, w.im)
  };
  static LGF_D V make(float re, float im) { return {f2_pack(re, im)}; }
  static LGF_D float re(V a) {
    float x, y;
    f2_unpack(a.v, x, y);
    return x;
  }
  static LGF_D float im(V a) {
    float x, y;
    f2_unpack(a.v, x, y);
    return y;
  }
  static LGF_D V zero() { return {0ull}; }
  static LGF_D V ld(const M *p) { return {*p}; }
  static LGF_D void st(M *p, V a) { *p = a.v; }
  static LGF_D V conj(V a) { return {a.v ^ 0x8000000000000000ull}; }
  static LGF_D V add(V a, V b) { return {f2_add(a.v, b.v)}; }
  static LGF_D V sub(V a, V b) { return {f2_sub(a.v, b.v)}; }
  static LGF_D V add_mi(V a, V b) { return {f2_fma(f2_swap(b.v), LGF_F2_PM, a.v)}; }
  static LGF_D V add_pi(V a, V b) { return {f2_fma(f2_swap(b.v), LGF_F2_MP, a.v)}; }
  static LGF_D V add_mh(V a, V b) { return {f2_fma(b.v, LGF_F2_MH, a.v)}; }
  static LGF_D V mul(V a, T w) { return {f2_fma(f2_swap(a.v), w.im, f2_mul(a.v, w.re))}; }
  static LGF_D V swap(V a) { return {f2_swap(a.v)}; }
  static LGF_D V fma_re(V acc, V a, T w) { return {f2_fma(a.v, w.re, acc.v)}; }
  static LGF_D V fma_im(V acc, V s, T w) { return {f2_fma(s.v, w.im, acc.v)}; }
  static LGF_D V mul_im(V s, T w) { return {f2_mul(s.v, w.im)}; }
  static LGF_D V mul_w8(V v, T w) { return {f2_mul(f2_fma(f2_swap(v.v), LGF_F2_PM, v.v), w.re)}; }
  static LGF_D V norm(V a) { return a; }
  static LGF_D V scale_conj(V a, float g) { return {f2_mul(a.v, f2_pack(g, -g))}; }
};

// ------------------------------------------------------------------ double-float
template <>
struct Ar<df> {
  typedef df Real;
  struct V {
    f2 h, l;
  };
  typedef ulonglong2 M;  // (re.hi, im.hi), (re.lo, im.lo)
  struct alignas(16) T {
    f2 reh, rel, imh, iml;  // (c, c) and (-w.im, w.im), high and low parts
  };
  static LGF_D V make(df re, df im) { return {f2_pack(re.hi, im.hi), f2_pack(re.lo, im.lo)}; }
  static LGF_D df re(V a) {
    df r;
    float t;
    f2_unpack(a.h, r.hi, t);
    f2_unpack(a.l, r.lo, t);
    return r;
  }
  static LGF_D df im(V a) {
    df r;
    float t;
    f2_unpack(a.h, t, r.hi);
    f2_unpack(a.l, t, r.lo);
    return r;
  }
  static LGF_D V zero() { return {0ull, 0ull}; }
  static LGF_D V ld(const M *p) {
    const ulonglong2 v = *p;
    return {v.x, v.y};
  }
  static LGF_D void st(M *p, V a) { *p = make_ulonglong2(a.h, a.l); }
  static LGF_D V conj(V a) { return {a.h ^ 0x8000000000000000ull, a.l ^ 0x8000000000000000ull}; }
  static LGF_D V add(V a, V b) {  // TwoSum with n = -(b's virtual part)
    const f2 s = f2_add(a.h, b.h), n = f2_sub(a.h, s);
    const f2 e = f2_add(f2_sub(a.h, f2_add(s, n)), f2_add(b.h, n));
    return {s, f2_add(e, f2_add(a.l, b.l))};
  }
  static LGF_D V sub(V a, V b) {
    const f2 s = f2_sub(a.h, b.h), n = f2_sub(a.h, s);
    const f2 e = f2_add(f2_sub(a.h, f2_add(s, n)), f2_sub(n, b.h));
    return {s, f2_add(e, f2_sub(a.l, b.l))};
  }
  // a + k * (bh, bl) for k of 0, +-1 or powers of two (exact products)
  static LGF_D V add_k(V a, f2 bh, f2 bl, f2 k) {
    const f2 s = f2_fma(bh, k, a.h), n = f2_sub(a.h, s);
    const f2 e = f2_add(f2_sub(a.h, f2_add(s, n)), f2_fma(bh, k, n));
    return {s, f2_add(e, f2_fma(bl, k, a.l))};
  }
  static LGF_D V add_mi(V a, V b) { return add_k(a, f2_swap(b.h), f2_swap(b.l), LGF_F2_PM); }
  static LGF_D V add_pi(V a, V b) { return add_k(a, f2_swap(b.h), f2_swap(b.l), LGF_F2_MP); }
  static LGF_D V add_mh(V a, V b) { return add_k(a, b.h, b.l, LGF_F2_MH); }
  static LGF_D V swap(V a) { return {f2_swap(a.h), f2_swap(a.l)}; }
  // Of a normalised value: both TwoProds, the four cross products folded into one correction, one TwoSum, one
  // renormalisation.
  static LGF_D V mul(V a, T w) {
    const f2 sh = f2_swap(a.h), sl = f2_swap(a.l);
    const f2 p1 = f2_mul(a.h, w.reh), e1 = f2_fma(a.h, w.reh, f2_neg(p1));
    const f2 p2 = f2_mul(sh, w.imh), e2 = f2_fma(sh, w.imh, f2_neg(p2));
    f2 x = f2_fma(a.l, w.reh, e1);
    x = f2_fma(a.h, w.rel, x);
    x = f2_fma(sl, w.imh, x);
    x = f2_fma(sh, w.iml, f2_add(x, e2));
    const f2 s = f2_add(p1, p2), n = f2_sub(p1, s);
    return norm({s, f2_add(f2_add(f2_sub(p1, f2_add(s, n)), f2_add(p2, n)), x)});
  }
  static LGF_D V mulr(V a, f2 ch, f2 cl) {  // componentwise product, left unnormalised
    const f2 p = f2_mul(a.h, ch);
    f2 e = f2_fma(a.h, ch, f2_neg(p));
    e = f2_fma(a.l, ch, e);
    return {p, f2_fma(a.h, cl, e)};
  }
  static LGF_D V fmar(V acc, V a, f2 ch, f2 cl) {
    const V q = mulr(a, ch, cl);
    return add(acc, q);
  }
  static LGF_D V fma_re(V acc, V a, T w) { return fmar(acc, a, w.reh, w.rel); }
  static LGF_D V fma_im(V acc, V s, T w) { return fmar(acc, s, w.imh, w.iml); }
  static LGF_D V mul_im(V s, T w) { return mulr(s, w.imh, w.iml); }
  static LGF_D V mul_w8(V v, T w) { return mulr(add_mi(v, v), w.reh, w.rel); }
  static LGF_D V norm(V a) {
    const f2 hi = f2_add(a.h, a.l);
    return {hi, f2_sub(a.l, f2_sub(hi, a.h))};
  }
  static LGF_D V scale_conj(V a, df g) { return mulr(a, f2_pack(g.hi, -g.hi), f2_pack(g.lo, -g.lo)); }
};

// The same arithmetic with every double-float sum and real product renormalised, 11 packed instructions a sum instead of
// 8: a sum of lazy sums rounds in proportion to low parts of several ulps.
template <class R>
struct ArFine : Ar<R> {};
template <>
struct ArFine<df> : Ar<df> {
  typedef Ar<df> L;
  static LGF_D V add(V a, V b) { return norm(L::add(a, b)); }
  static LGF_D V sub(V a, V b) { return norm(L::sub(a, b)); }
  static LGF_D V add_mi(V a, V b) { return norm(L::add_mi(a, b)); }
  static LGF_D V add_pi(V a, V b) { return norm(L::add_pi(a, b)); }
  static LGF_D V add_mh(V a, V b) { return norm(L::add_mh(a, b)); }
  static LGF_D V fma_re(V acc, V a, T w) { return norm(L::fma_re(acc, a, w)); }
  static LGF_D V fma_im(V acc, V s, T w) { return norm(L::fma_im(acc, s, w)); }
  static LGF_D V mul_im(V s, T w) { return norm(L::mul_im(s, w)); }
  static LGF_D V mul_w8(V v, T w) { return norm(mulr(add_mi(v, v), w.reh, w.rel)); }
};

// Host-side construction of a twiddle (re, im) from FP64 (T as above).
inline void make_T(double re, double im, Ar<double>::T &t) { t = make_double2(re, im); }
inline f2 host_pack(float a, float b) {
  union {
    float f[2];
    f2 v;
  } u;
  u.f[0] = a;
  u.f[1] = b;
  return u.v;
}
inline void make_T(double re, double im, Ar<float>::T &t) {
  t.re = host_pack((float)re, (float)re);
  t.im = host_pack(-(float)im, (float)im);
}
inline void make_T(double re, double im, Ar<df>::T &t) {
  const float rh = (float)re, rl = (float)(re - (double)rh), ih = (float)im, il = (float)(im - (double)ih);
  t.reh = host_pack(rh, rh);
  t.rel = host_pack(rl, rl);
  t.imh = host_pack(-ih, ih);
  t.iml = host_pack(-il, il);
}

// ------------------------------------------------------------------ small DFTs in registers
// Forward DFTs (e^{-2 pi i jk / N}), unnormalised, natural order in and out; A is Ar<R> or ArFine<R>.

// Twiddles of one launch, in the parameter bank: W_P^n, n < P = 2 NB, and the constants of the 16-point FFT.
#define LINE_P_MAX 32
template <class R>
struct LineTw {
  typename Ar<R>::T p[LINE_P_MAX];
  typename Ar<R>::T w16[4];  // W_16^1, W_16^2 (= W_8), W_16^3, W_16^9
  typename Ar<R>::T c3;      // (cos, -sin)(2 pi / 3)
};

// 4 points; the third and fourth input may come without their factor -i (M2, M3), folded into the sums.
template <class A, bool M2 = false, bool M3 = false>
LGF_D void dft4(typename A::V &a, typename A::V &b, typename A::V &c, typename A::V &d) {
  const typename A::V s02 = M2 ? A::add_mi(a, c) : A::add(a, c), d02 = M2 ? A::add_pi(a, c) : A::sub(a, c);
  const typename A::V s13 = M3 ? A::add_mi(b, d) : A::add(b, d), d13 = M3 ? A::add_pi(b, d) : A::sub(b, d);
  a = A::add(s02, s13);
  c = A::sub(s02, s13);
  b = A::add_mi(d02, d13);
  d = A::add_pi(d02, d13);
}

template <class T>
LGF_D void vswap(T &a, T &b) {
  const T t = a;
  a = b;
  b = t;
}

template <class A>
LGF_D void dft16(typename A::V (&x)[16], const LineTw<typename A::Real> &tw) {
#pragma unroll
  for (int i = 0; i < 4; ++i) dft4<A>(x[i], x[i + 4], x[i + 8], x[i + 12]);
  // x[a + 4 k] *= W_16^{a k}; W_16^4 = -i and the -i of W_16^6 = -i W_8 are folded into the second stage
  x[5] = A::mul(A::norm(x[5]), tw.w16[0]);
  x[9] = A::mul_w8(x[9], tw.w16[1]);
  x[13] = A::mul(A::norm(x[13]), tw.w16[2]);
  x[6] = A::mul_w8(x[6], tw.w16[1]);
  x[14] = A::mul_w8(x[14], tw.w16[1]);
  x[7] = A::mul(A::norm(x[7]), tw.w16[2]);
  x[11] = A::mul_w8(x[11], tw.w16[1]);
  x[15] = A::mul(A::norm(x[15]), tw.w16[3]);
  dft4<A>(x[0], x[1], x[2], x[3]);
  dft4<A>(x[4], x[5], x[6], x[7]);
  dft4<A, true, true>(x[8], x[9], x[10], x[11]);
  dft4<A, true, false>(x[12], x[13], x[14], x[15]);
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int j = i + 1; j < 4; ++j) vswap(x[4 * i + j], x[4 * j + i]);
}

template <class A>
LGF_D void dft8(typename A::V (&x)[8], const LineTw<typename A::Real> &tw) {
  dft4<A>(x[0], x[2], x[4], x[6]);  // even points: E_k in x[0], x[2], x[4], x[6]
  dft4<A>(x[1], x[3], x[5], x[7]);  // odd points
  const typename A::V o1 = A::mul_w8(x[3], tw.w16[1]), o3 = A::mul_w8(x[7], tw.w16[1]);
  const typename A::V e0 = x[0], e1 = x[2], e2 = x[4], e3 = x[6], o0 = x[1], o2 = x[5];
  x[0] = A::add(e0, o0);
  x[4] = A::sub(e0, o0);
  x[1] = A::add(e1, o1);
  x[5] = A::sub(e1, o1);
  x[2] = A::add_mi(e2, o2);  // W_8^2 = -i
  x[6] = A::add_pi(e2, o2);
  x[3] = A::add_mi(e3, o3);  // W_8^3 = -i W_8
  x[7] = A::add_pi(e3, o3);
}

template <class A>
LGF_D void dft3(typename A::V &a, typename A::V &b, typename A::V &c, const LineTw<typename A::Real> &tw) {
  const typename A::V u = A::add(b, c), v = A::swap(A::sub(b, c));
  const typename A::V m = A::add_mh(a, u), q = A::mul_im(v, tw.c3);  // q = -i sin(2 pi / 3) (b - c)
  a = A::add(a, u);
  b = A::add(m, q);
  c = A::sub(m, q);
}

// Odd N >= 5 by conjugate pairs with real coefficients; W_N^j = W_P^{j P / N} from the launch's table.
template <class A, int N, int P>
LGF_D void dft_odd(typename A::V (&x)[N], const LineTw<typename A::Real> &tw) {
  constexpr int H = (N - 1) / 2;
  typename A::V u[H], v[H], x0 = x[0];
#pragma unroll
  for (int j = 0; j < H; ++j) {
    u[j] = A::add(x[j + 1], x[N - 1 - j]);
    v[j] = A::swap(A::sub(x[j + 1], x[N - 1 - j]));
  }
  typename A::V sum = x0;
#pragma unroll
  for (int j = 0; j < H; ++j) sum = A::add(sum, u[j]);
  x[0] = sum;
#pragma unroll
  for (int k = 1; k <= H; ++k) {
    typename A::V a = x0, b = A::mul_im(v[0], tw.p[k * (P / N)]);
#pragma unroll
    for (int j = 1; j <= H; ++j) {
      const int q = (j * k) % N * (P / N);
      a = A::fma_re(a, u[j - 1], tw.p[q]);
      if (j > 1) b = A::fma_im(b, v[j - 1], tw.p[q]);
    }
    x[k] = A::add(a, b);
    x[N - k] = A::sub(a, b);
  }
}

// v W_N^r, r and N compile-time after unrolling; quarter turns as swaps and signs
template <class A, int N, int P>
LGF_D typename A::V rotate(typename A::V v, const LineTw<typename A::Real> &tw, int r) {
  r %= N;
  if (r == 0) return v;
  if (4 * r == N) return A::add_mi(A::zero(), v);
  if (2 * r == N) return A::sub(A::zero(), v);
  if (4 * r == 3 * N) return A::add_pi(A::zero(), v);
  return A::mul(A::norm(v), tw.p[r * (P / N)]);
}

constexpr int dft_radix(int n) { return n % 4 == 0 ? 4 : (n % 2 == 0 ? 2 : (n % 3 == 0 ? 3 : n)); }
constexpr int gcd_of(int a, int b) { return b == 0 ? a : gcd_of(b, a % b); }
constexpr int inverse_mod(int a, int n) {  // a^-1 mod n (0 for n = 1)
  for (int i = 0; i < n; ++i)
    if (a * i % n == 1 % n) return i;
  return 0;
}

// N points, N | P, P / N even or N in the direct list
template <class A, int N, int P>
struct Dft {
  typedef typename A::V V;
  static LGF_D void run(V (&x)[N], const LineTw<typename A::Real> &tw) {
    if constexpr (N == 1) {
    } else if constexpr (N == 2) {
      const V a = x[0];
      x[0] = A::add(a, x[1]);
      x[1] = A::sub(a, x[1]);
    } else if constexpr (N == 3) {
      dft3<A>(x[0], x[1], x[2], tw);
    } else if constexpr (N == 4) {
      dft4<A>(x[0], x[1], x[2], x[3]);
    } else if constexpr (N == 8) {
      dft8<A>(x, tw);
    } else if constexpr (N == 16) {
      dft16<A>(x, tw);
    } else {
      constexpr int F = dft_radix(N), Q = N / F;  // j = a + F b, k = k2 + Q k1
      if constexpr (Q == 1) {
        dft_odd<A, N, P>(x, tw);
      } else if constexpr (gcd_of(F, Q) == 1) {
        // coprime factors without twiddles: input j = (Q a + F b) mod N, output k = k1 mod F = k2 mod Q
        constexpr int CF = Q * inverse_mod(Q, F), CQ = F * inverse_mod(F, Q);
        V y[F][Q];
#pragma unroll
        for (int a = 0; a < F; ++a) {
#pragma unroll
          for (int b = 0; b < Q; ++b) y[a][b] = x[(Q * a + F * b) % N];
          Dft<A, Q, P>::run(y[a], tw);
        }
#pragma unroll
        for (int k2 = 0; k2 < Q; ++k2) {
          V z[F];
#pragma unroll
          for (int a = 0; a < F; ++a) z[a] = y[a][k2];
          Dft<A, F, P>::run(z, tw);
#pragma unroll
          for (int k1 = 0; k1 < F; ++k1) x[(CF * k1 + CQ * k2) % N] = z[k1];
        }
      } else {
        V y[F][Q];
#pragma unroll
        for (int a = 0; a < F; ++a) {
#pragma unroll
          for (int b = 0; b < Q; ++b) y[a][b] = x[a + F * b];
          Dft<A, Q, P>::run(y[a], tw);
#pragma unroll
          for (int k2 = 1; k2 < Q; ++k2)
            if (a > 0) y[a][k2] = rotate<A, N, P>(y[a][k2], tw, a * k2);
        }
#pragma unroll
        for (int k2 = 0; k2 < Q; ++k2) {
          V z[F];
#pragma unroll
          for (int a = 0; a < F; ++a) z[a] = y[a][k2];
          Dft<A, F, P>::run(z, tw);
#pragma unroll
          for (int k1 = 0; k1 < F; ++k1) x[k2 + Q * k1] = z[k1];
        }
      }
    }
  }
};

}  // namespace lgf
