// Complex arithmetic policies of the FFT kernels and compile-time register
// DFTs.
//
// Policies: P32 complex64 (float2), P64 complex128 (double2), PFF complex
// float-float (float4 = re.hi, im.hi, re.lo, im.lo; about 48 bits on the FP32
// pipes, see ff.h).  Every butterfly is written once over a policy.
//
// RegDFT<P, N, INV>::run(v) transforms N values held in registers (natural
// order in and out) by recursive decimation in time, N = R * M:
//   X[k2 + M q] = sum_j w_N^(j k2) E_j[k2] w_R^(j q),  E_j = DFT_M(x[R i + j]),
// with every index and every twiddle known at compile time.  The twiddle
// constants w_N^e = cos(2 pi e / N) - i sin(2 pi e / N) are evaluated by
// constexpr Taylor series (after an exact octant reduction of e / N), so no
// table is read and the float-float policy gets both halves of each constant
// folded into the instruction stream.
#pragma once

#include <cuda_runtime.h>

#include <type_traits>
#include <utility>

#include "common.h"
#include "ff.h"

namespace aim {

// ------------------------------------------------------------------ compile-time trigonometry
constexpr double kTwoPi = 6.283185307179586476925286766559;

// Taylor series for |x| <= pi/4 (the 16-term truncation error is far below 1e-20).
constexpr double cx_sin_small(double x) {
  double term = x, sum = x;
  for (int n = 1; n < 16; ++n) {
    term *= -x * x / ((2.0 * n) * (2.0 * n + 1.0));
    sum += term;
  }
  return sum;
}
constexpr double cx_cos_small(double x) {
  double term = 1.0, sum = 1.0;
  for (int n = 1; n < 16; ++n) {
    term *= -x * x / ((2.0 * n - 1.0) * (2.0 * n));
    sum += term;
  }
  return sum;
}
// cos and sin of 2 pi e / N for integers e, N > 0: reduce e / N to the first
// octant exactly in integer arithmetic (8 e mod 8 N), then use the series.
struct CS {
  double c, s;
};
constexpr CS cx_cossin_2pi(long e, long N) {
  e %= N;
  if (e < 0) e += N;
  const long e8 = 8 * e;       // angle in units of (2 pi / 8N) ... octant index = e8 / N
  const long oct = e8 / N;     // 0..7
  const long rem = e8 - oct * N;  // 0 <= rem < N, angle within the octant = (pi/4) rem / N
  double a = (kTwoPi / 8.0) * (double)rem / (double)N;
  // octants: angle = oct * pi/4 + a
  double c0 = cx_cos_small(a), s0 = cx_sin_small(a);
  double b = (kTwoPi / 8.0) - a;  // for odd octants use the complement for accuracy
  double c1 = cx_cos_small(b), s1 = cx_sin_small(b);
  switch (oct) {
    case 0: return CS{c0, s0};
    case 1: return CS{s1, c1};
    case 2: return CS{-s0, c0};
    case 3: return CS{-c1, s1};
    case 4: return CS{-c0, -s0};
    case 5: return CS{-s1, -c1};
    case 6: return CS{s0, -c0};
    default: return CS{c1, -s1};
  }
}

template <int B, int E, class F> AIM_HD __forceinline__ void static_for(F&& f) {
  if constexpr (B < E) {
    f(std::integral_constant<int, B>{});
    static_for<B + 1, E>(f);
  }
}

// ------------------------------------------------------------------ policies
struct P32 {
  using S = float2;  // storage
  using T = float2;  // work
  static constexpr int kTX = 16;
  __device__ static T ld(const S& s) { return s; }
  __device__ static S st(const T& t) { return t; }
  __device__ static T zero() { return make_float2(0.f, 0.f); }
  __device__ static T add(T a, T b) { return add2(a, b); }
  __device__ static T sub(T a, T b) { return sub2(a, b); }
  __device__ static T neg(T a) { return neg2(a); }
  __device__ static T mul(T a, T b) { return make_float2(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x); }
  __device__ static T mulr(T a, double, float c, float) { return mul2(a, both(c)); }
  __device__ static T madr(T m, T a, double, float c, float) { return fma2(a, both(c), m); }  // m + c a
  __device__ static T sub_half(T m, T a) { return fma2(a, both(-0.5f), m); }                  // m - a / 2
  __device__ static T neg_half(T a) { return mul2(a, both(-0.5f)); }
  // a * (c + i s) for compile-time constants
  __device__ static T mulc(T a, double, float c, float, double, float s, float) {
    return fma2(swap2(a), make_float2(-s, s), mul2(a, both(c)));
  }
  template <bool INV> __device__ static T mul_mi(T a) {
    return INV ? make_float2(-a.y, a.x) : make_float2(a.y, -a.x);
  }
  // m + sg * mul_mi(c d) and m + sg * mul_mi(d) (sg = +-1)
  template <bool INV, int SG> __device__ static T add_mi_scaled(T m, T d, double, float c, float) {
    const float cs = SG * (INV ? -c : c);
    return fma2(swap2(d), make_float2(cs, -cs), m);
  }
  template <bool INV, int SG> __device__ static T add_mi(T m, T d) {
    return add_mi_scaled<INV, SG>(m, d, 1.0, 1.f, 0.f);
  }
  __device__ static T conj_if(T w, bool c) { return c ? make_float2(w.x, -w.y) : w; }
};

struct P64 {
  using S = double2;
  using T = double2;
  static constexpr int kTX = 8;
  AIM_HD static T ld(const S& s) { return s; }
  AIM_HD static S st(const T& t) { return t; }
  AIM_HD static T zero() { return make_double2(0.0, 0.0); }
  AIM_HD static T add(T a, T b) { return make_double2(a.x + b.x, a.y + b.y); }
  AIM_HD static T sub(T a, T b) { return make_double2(a.x - b.x, a.y - b.y); }
  AIM_HD static T neg(T a) { return make_double2(-a.x, -a.y); }
  AIM_HD static T mul(T a, T b) { return make_double2(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x); }
  AIM_HD static T mulr(T a, double c, float, float) { return make_double2(a.x * c, a.y * c); }
  AIM_HD static T madr(T m, T a, double c, float, float) { return make_double2(fma(c, a.x, m.x), fma(c, a.y, m.y)); }
  AIM_HD static T sub_half(T m, T a) { return make_double2(fma(-0.5, a.x, m.x), fma(-0.5, a.y, m.y)); }
  AIM_HD static T neg_half(T a) { return make_double2(-0.5 * a.x, -0.5 * a.y); }
  AIM_HD static T mulc(T a, double c, float, float, double s, float, float) {
    return make_double2(a.x * c - a.y * s, a.x * s + a.y * c);
  }
  template <bool INV> AIM_HD static T mul_mi(T a) { return INV ? make_double2(-a.y, a.x) : make_double2(a.y, -a.x); }
  template <bool INV, int SG> AIM_HD static T add_mi_scaled(T m, T d, double c, float, float) {
    const double cs = SG * (INV ? -c : c);
    return make_double2(fma(cs, d.y, m.x), fma(-cs, d.x, m.y));
  }
  template <bool INV, int SG> AIM_HD static T add_mi(T m, T d) {
    const T t = mul_mi<INV>(d);
    return SG > 0 ? add(m, t) : sub(m, t);
  }
  AIM_HD static T conj_if(T w, bool c) { return c ? make_double2(w.x, -w.y) : w; }
};

struct PFF {
  using S = float4;  // (re.hi, im.hi, re.lo, im.lo)
  using T = cff2;
  static constexpr int kTX = 8;
  __device__ static T ld(const S& s) { return cff2_ld(s); }
  __device__ static S st(const T& t) { return cff2_st(t); }
  __device__ static T zero() { return cff2_zero(); }
  // additions without the closing renormalisation: every value feeds further arithmetic
  __device__ static T add(T a, T b) { return cff2_add_lazy(a, b); }
  __device__ static T sub(T a, T b) { return cff2_add_lazy(a, cff2_neg(b)); }
  __device__ static T neg(T a) { return cff2_neg(a); }
  __device__ static T mul(T a, T b) { return cff2_dot2(cff2_re(a), b, cff2_im(a), cff2_times_i(b)); }
  __device__ static T mulr(T a, double, float ch, float cl) {
    const float2 h = both(ch), p = mul2(a.hi, h);
    float2 e = fma2(a.hi, h, neg2(p));
    e = fma2(a.hi, both(cl), e);
    e = fma2(a.lo, h, e);
    return fast_two_sum2(p, e);
  }
  __device__ static T madr(T m, T a, double c, float ch, float cl) { return add(m, mulr(a, c, ch, cl)); }
  __device__ static T neg_half(T a) { return cff2{mul2(a.hi, both(-0.5f)), mul2(a.lo, both(-0.5f))}; }
  __device__ static T sub_half(T m, T a) { return add(m, neg_half(a)); }
  __device__ static T mulc(T a, double, float ch, float cl, double, float sh, float sl) {
    return cff2_dot2(a, cff2{both(ch), both(cl)}, cff2{swap2(a.hi), swap2(a.lo)},
                     cff2{make_float2(-sh, sh), make_float2(-sl, sl)});
  }
  template <bool INV> __device__ static T mul_mi(T a) { return INV ? cff2_times_i(a) : cff2_neg(cff2_times_i(a)); }
  template <bool INV, int SG> __device__ static T add_mi_scaled(T m, T d, double c, float ch, float cl) {
    return add_mi<INV, SG>(m, mulr(d, c, ch, cl));
  }
  template <bool INV, int SG> __device__ static T add_mi(T m, T d) {
    const T t = mul_mi<(SG > 0) == INV>(d);
    return add(m, t);
  }
  __device__ static T conj_if(T w, bool c) {
    return c ? cff2{make_float2(w.hi.x, -w.hi.y), make_float2(w.lo.x, -w.lo.y)} : w;
  }
};

// Real constants as (double value, float hi, float lo).
#define AIM_RC(c) (c), (float)(c), (float)((c) - (double)(float)(c))

// ------------------------------------------------------------------ small butterflies
// Each takes a mask Z of the inputs that are not known to be zero (bit i:
// v[i]); the others are neither read nor added.  A zero-padded transform
// whose upper half is zero drops the additions of its first stage this way.
template <class P, bool A, bool B> AIM_HD __forceinline__ typename P::T add_z(typename P::T a, typename P::T b) {
  if constexpr (A && B) return P::add(a, b);
  else if constexpr (A) return a;
  else if constexpr (B) return b;
  else return P::zero();
}
template <class P, bool A, bool B> AIM_HD __forceinline__ typename P::T sub_z(typename P::T a, typename P::T b) {
  if constexpr (A && B) return P::sub(a, b);
  else if constexpr (A) return a;
  else if constexpr (B) return P::neg(b);
  else return P::zero();
}
// m + sg * mul_mi(d)
template <class P, bool INV, int SG, bool M, bool D>
AIM_HD __forceinline__ typename P::T add_mi_z(typename P::T m, typename P::T d) {
  if constexpr (M && D) return P::template add_mi<INV, SG>(m, d);
  else if constexpr (M) return m;
  else if constexpr (D) return P::template mul_mi<(SG > 0) == INV>(d);
  else return P::zero();
}
constexpr bool has(unsigned long long z, int i) { return (z >> i) & 1; }
constexpr unsigned long long all_mask(int n) { return n >= 64 ? ~0ull : (1ull << n) - 1; }

template <class P, bool INV, unsigned long long Z = 3> AIM_HD __forceinline__ void dft2(typename P::T* v) {
  const typename P::T a = v[0], b = v[1];
  v[0] = add_z<P, has(Z, 0), has(Z, 1)>(a, b);
  v[1] = sub_z<P, has(Z, 0), has(Z, 1)>(a, b);
}
template <class P, bool INV, unsigned long long Z = 7> AIM_HD __forceinline__ void dft3(typename P::T* v) {
  using T = typename P::T;
  constexpr bool z0 = has(Z, 0), z1 = has(Z, 1), z2 = has(Z, 2), zs = z1 || z2;
  const T a = v[0], s = add_z<P, z1, z2>(v[1], v[2]), d = sub_z<P, z1, z2>(v[1], v[2]);
  v[0] = add_z<P, z0, zs>(a, s);
  if constexpr (zs) {
    T m;
    if constexpr (z0) m = P::sub_half(a, s);
    else m = P::neg_half(s);
    // v1, v2 = m +- (-i) sin(2 pi / 3) d (forward; +i inverse), each a fused multiply-add
    v[1] = P::template add_mi_scaled<INV, 1>(m, d, AIM_RC(0.86602540378443864676));
    v[2] = P::template add_mi_scaled<INV, -1>(m, d, AIM_RC(0.86602540378443864676));
  } else {
    v[1] = v[2] = a;
  }
}
template <class P, bool INV, unsigned long long Z = 15> AIM_HD __forceinline__ void dft4(typename P::T* v) {
  using T = typename P::T;
  constexpr bool z0 = has(Z, 0), z1 = has(Z, 1), z2 = has(Z, 2), z3 = has(Z, 3), ze = z0 || z2, zo = z1 || z3;
  const T s02 = add_z<P, z0, z2>(v[0], v[2]), d02 = sub_z<P, z0, z2>(v[0], v[2]);
  const T s13 = add_z<P, z1, z3>(v[1], v[3]), d13 = sub_z<P, z1, z3>(v[1], v[3]);
  v[0] = add_z<P, ze, zo>(s02, s13);
  v[2] = sub_z<P, ze, zo>(s02, s13);
  v[1] = add_mi_z<P, INV, 1, ze, zo>(d02, d13);
  v[3] = add_mi_z<P, INV, -1, ze, zo>(d02, d13);
}
template <class P, bool INV, unsigned long long Z = 31> AIM_HD __forceinline__ void dft5(typename P::T* v) {
  using T = typename P::T;
  constexpr bool z0 = has(Z, 0), z1 = has(Z, 1), z2 = has(Z, 2), z3 = has(Z, 3), z4 = has(Z, 4);
  constexpr bool za = z1 || z4, zb = z2 || z3;
  const T a0 = v[0];
  if constexpr (!za && !zb) {
    v[1] = v[2] = v[3] = v[4] = a0;
    return;
  }
  const T t1 = add_z<P, z1, z4>(v[1], v[4]), t2 = add_z<P, z2, z3>(v[2], v[3]);
  const T t3 = sub_z<P, z1, z4>(v[1], v[4]), t4 = sub_z<P, z2, z3>(v[2], v[3]);
  // cos(2pi/5), cos(4pi/5), sin(2pi/5), sin(4pi/5)
  T b1, b2, u1, u2;
  if constexpr (za && zb) {
    b1 = P::madr(P::mulr(t1, AIM_RC(0.30901699437494742410)), t2, AIM_RC(-0.80901699437494742410));
    b2 = P::madr(P::mulr(t1, AIM_RC(-0.80901699437494742410)), t2, AIM_RC(0.30901699437494742410));
    u1 = P::madr(P::mulr(t3, AIM_RC(0.95105651629515357212)), t4, AIM_RC(0.58778525229247312917));
    u2 = P::madr(P::mulr(t3, AIM_RC(0.58778525229247312917)), t4, AIM_RC(-0.95105651629515357212));
  } else if constexpr (za) {
    b1 = P::mulr(t1, AIM_RC(0.30901699437494742410));
    b2 = P::mulr(t1, AIM_RC(-0.80901699437494742410));
    u1 = P::mulr(t3, AIM_RC(0.95105651629515357212));
    u2 = P::mulr(t3, AIM_RC(0.58778525229247312917));
  } else {
    b1 = P::mulr(t2, AIM_RC(-0.80901699437494742410));
    b2 = P::mulr(t2, AIM_RC(0.30901699437494742410));
    u1 = P::mulr(t4, AIM_RC(0.58778525229247312917));
    u2 = P::mulr(t4, AIM_RC(-0.95105651629515357212));
  }
  b1 = add_z<P, z0, true>(a0, b1);
  b2 = add_z<P, z0, true>(a0, b2);
  v[0] = add_z<P, z0, true>(a0, add_z<P, za, zb>(t1, t2));
  v[1] = P::template add_mi<INV, 1>(b1, u1);
  v[4] = P::template add_mi<INV, -1>(b1, u1);
  v[2] = P::template add_mi<INV, 1>(b2, u2);
  v[3] = P::template add_mi<INV, -1>(b2, u2);
}

// ------------------------------------------------------------------ register DFT
constexpr int first_factor(int n) {
  return (n % 4 == 0) ? 4 : (n % 3 == 0) ? 3 : (n % 5 == 0) ? 5 : (n % 2 == 0) ? 2 : n;
}
constexpr int gcd_c(int a, int b) { return b == 0 ? a : gcd_c(b, a % b); }
// A radix R in {4, 3, 5, 2} with N = R M and gcd(R, M) = 1 (a prime-factor
// split, which needs no twiddle factors), or 0 when N has none.
constexpr int coprime_factor(int n) {
  const int rs[4] = {4, 3, 5, 2};
  for (int i = 0; i < 4; ++i)
    if (n % rs[i] == 0 && n / rs[i] > 1 && gcd_c(rs[i], n / rs[i]) == 1) return rs[i];
  return 0;
}
// a^-1 mod m for gcd(a, m) = 1
constexpr int inv_mod(int a, int m) {
  for (int x = 1; x < m; ++x)
    if ((a * x) % m == 1) return x;
  return m == 1 ? 0 : -1;
}

// x * w_N^E (forward) or x * conj(w_N^E) (inverse), E compile-time
template <class P, int N, int E, bool INV> AIM_HD __forceinline__ typename P::T twiddle_c(typename P::T x) {
  constexpr int e = E % N;
  if constexpr (e == 0) {
    return x;
  } else if constexpr (2 * e == N) {
    return P::neg(x);
  } else if constexpr (4 * e == N) {
    return P::template mul_mi<INV>(x);  // w^(N/4) = -i
  } else if constexpr (4 * e == 3 * N) {
    return P::template mul_mi<!INV>(x);  // w^(3N/4) = +i
  } else {
    constexpr CS cs = cx_cossin_2pi(e, N);
    constexpr double c = cs.c;
    constexpr double s = INV ? cs.s : -cs.s;  // forward: exp(-i theta)
    return P::mulc(x, c, (float)c, (float)(c - (double)(float)c), s, (float)s, (float)(s - (double)(float)s));
  }
}

// The mask of the inputs first, first + step, ... (count of them, mod n) of a DFT of length n
constexpr unsigned long long sub_mask(unsigned long long z, int n, int first, int step, int count) {
  unsigned long long m = 0;
  for (int i = 0; i < count; ++i)
    if (has(z, (first + step * i) % n)) m |= 1ull << i;
  return m;
}
// Bit j: whether the sub-transform j (inputs base j + step i mod n, i < count) has a nonzero input
constexpr unsigned long long group_mask(unsigned long long z, int n, int groups, int base, int step, int count) {
  unsigned long long m = 0;
  for (int j = 0; j < groups; ++j)
    if (sub_mask(z, n, (base * j) % n, step, count)) m |= 1ull << j;
  return m;
}

// Z: the inputs that are not known to be zero (see the butterflies).
template <class P, int N, bool INV, unsigned long long Z = all_mask(N)> struct RegDFT {
  using T = typename P::T;
  AIM_HD __forceinline__ static void run(T* v) {
    if constexpr (N == 1) {
    } else if constexpr (N == 2) {
      dft2<P, INV, Z>(v);
    } else if constexpr (N == 3) {
      dft3<P, INV, Z>(v);
    } else if constexpr (N == 4) {
      dft4<P, INV, Z>(v);
    } else if constexpr (N == 5) {
      dft5<P, INV, Z>(v);
    } else if constexpr (coprime_factor(N) != 0) {
      // Good-Thomas prime-factor split N = R M, gcd(R, M) = 1: input index
      // n = (M j + R i) mod N, output index k = (M a k1 + R b k2) mod N with
      // a = M^-1 mod R, b = R^-1 mod M; the two DFT stages need no twiddles.
      constexpr int R = coprime_factor(N);
      constexpr int M = N / R;
      constexpr int A = inv_mod(M % R, R), B = inv_mod(R % M, M);
      constexpr unsigned long long ZG = group_mask(Z, N, R, M, R, M);
      T sub[R][M];
      static_for<0, R>([&](auto j) {
        static_for<0, M>([&](auto i) { sub[j][i] = v[(M * decltype(j)::value + R * decltype(i)::value) % N]; });
        constexpr unsigned long long ZS = sub_mask(Z, N, (M * decltype(j)::value) % N, R, M);
        if constexpr (ZS != 0) RegDFT<P, M, INV, ZS>::run(sub[j]);
      });
      static_for<0, M>([&](auto k2) {
        T t[R];
        static_for<0, R>([&](auto j) { t[j] = sub[j][k2]; });
        RegDFT<P, R, INV, ZG>::run(t);
        static_for<0, R>([&](auto k1) {
          v[(M * A * decltype(k1)::value + R * B * decltype(k2)::value) % N] = t[k1];
        });
      });
    } else {
      constexpr int R = first_factor(N);
      constexpr int M = N / R;
      static_assert(R * M == N && R > 1 && R <= 5, "register DFT length must be 2,3,5-smooth");
      constexpr unsigned long long ZG = group_mask(Z, N, R, 1, R, M);
      T sub[R][M];
      static_for<0, R>([&](auto j) {
        static_for<0, M>([&](auto i) { sub[j][i] = v[R * i + j]; });
        constexpr unsigned long long ZS = sub_mask(Z, N, decltype(j)::value, R, M);
        if constexpr (ZS != 0) RegDFT<P, M, INV, ZS>::run(sub[j]);
      });
      static_for<0, M>([&](auto k2) {
        T t[R];
        static_for<0, R>([&](auto j) {
          if constexpr (has(ZG, decltype(j)::value))
            t[j] = twiddle_c<P, N, decltype(j)::value * decltype(k2)::value, INV>(sub[j][k2]);
          else
            t[j] = P::zero();
        });
        RegDFT<P, R, INV, ZG>::run(t);
        static_for<0, R>([&](auto q) { v[k2 + M * q] = t[q]; });
      });
    }
  }
};

}  // namespace aim
