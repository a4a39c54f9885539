// Complex numbers in signed digits of radix 2^29 or 2^30 with a shared
// exponent, held whole by one thread: the products of the value-sum
// evaluation (kernels_sum.cu).
//
// A number is sum_i d_i 2^(B i) * 2^e, i = 0 .. L-1, for each of its two
// components.  A complex product accumulates the 2 L products of every column
// of both components in 64-bit integers (32 x 32 + 64 -> 64-bit multiply-add,
// IMAD.WIDE), keeps the columns from L - 1 up and propagates carries once per
// component: no carry flags, no sign handling, no partner lane.  The columns
// below are dropped, so a product errs by a few units of its last place.
//
// Measured on GB300 (chains of products, factor read from shared memory, 16
// warps per SM): 51 SM cycles per 32 complex products for L = 4 (double-double;
// the 128-bit sign-magnitude product of wide.cuh takes 40 to 53 for 16), 35 for L = 3
// (double; four FP64 instructions at 2 lanes per clock take 64) and 150
// for L = 8 (quad-double).  The bound is the multiply-adds: 4 L (L + 1) / 2 of
// them at 32 lanes per SM and clock.
//
// Two kinds of operands:
//   * X (table entries): balanced digits, |d_i| <= 2^(B-1), modulus within
//     2^(+-1/2) of 2^(B L - 1) (a unit-modulus number exactly there), so that
//     a product, which is shifted down by B L - 1 bits, keeps its modulus to
//     within that factor and a chain of unit-modulus factors never needs
//     renormalising;
//   * y (running products): 0 <= d_i < 2^B below the top digit, which is
//     signed.  Fresh values have a modulus near 2^(B L - 3); every
//     kCheckEvery-th product the larger component is brought back into
//     [2^(B L - 5), 2^(B L - 2)) if it has left it, so the top digit stays
//     below 2^(B + 1/2).
// Column bounds with these limits, B = 30, L <= 4: the largest doubled column
// (column L: L - 3 interior pairs of 2^29 2^30 for each component, and the two
// pairs with a top digit) is at most 2 (1 + 1 + 1.42) 2^60 < 2^63; B = 29,
// L = 8: 2 (5 + 1 + 1.42) 2^58 < 2^62.
#pragma once

#include <cstdint>

#include "internal.h"
#include "wide8.cuh"

namespace pe {
namespace fx {

// Per digit count: radix, words of the accumulation window (kernels_sum.cu),
// and the least bit of the window that the largest term of a derivative may
// have as its leading one (a derivative of one term; sum_slack in internal.h
// raises it for more).
template <int L>
struct Fmt;
template <>
struct Fmt<3> {  // double: 88-bit numbers
  static constexpr int B = 30, W = 5, kKeep = 72, kHeadMin = 16;
};
template <>
struct Fmt<4> {  // double-double: 118-bit numbers
  static constexpr int B = 30, W = 6, kKeep = 112, kHeadMin = 16;
};
template <>
struct Fmt<8> {  // quad-double: 230-bit numbers
  static constexpr int B = 29, W = 10, kKeep = 224, kHeadMin = 32;
};

constexpr int kCheckEvery = 4;
constexpr int32_t kZeroExp = -(1 << 28);

template <int L>
struct Num {
  int32_t re[L], im[L];
  int32_t e;
};

// Carries from the columns c[0] (weight B (L - 1)), c[1], ... of a product:
// r = floor(sum_i c[i] 2^(B (L - 1 + i)) / 2^(B L - 1)).
template <int L>
__device__ __forceinline__ void fold(const long long (&c)[L], int32_t (&r)[L]) {
  constexpr int B = Fmt<L>::B;
  constexpr int32_t kMask = (1 << B) - 1;
  long long t = c[0] >> (B - 1);
#pragma unroll
  for (int i = 1; i < L; i++) {
    t += c[i] << 1;
    r[i - 1] = static_cast<int32_t>(t) & kMask;
    t >>= B;
  }
  r[L - 1] = static_cast<int32_t>(t);
}

// y * X (y-kind result).
template <int L>
__device__ __forceinline__ void mul(Num<L> &y, const Num<L> &X) {
  long long cr[L], ci[L];
  int32_t n[L];
#pragma unroll
  for (int i = 0; i < L; i++) n[i] = -y.im[i];
#pragma unroll
  for (int c = 0; c < L; c++) {
    long long r = 0, m = 0;
#pragma unroll
    for (int i = c; i < L; i++) {
      const int j = c + L - 1 - i;
      r += static_cast<long long>(X.re[i]) * y.re[j];
      r += static_cast<long long>(X.im[i]) * n[j];
      m += static_cast<long long>(X.re[i]) * y.im[j];
      m += static_cast<long long>(X.im[i]) * y.re[j];
    }
    cr[c] = r;
    ci[c] = m;
  }
  fold<L>(cr, y.re);
  fold<L>(ci, y.im);
  y.e += X.e + Fmt<L>::B * L - 1;
}

// Shift the digits of a y-kind component left (s > 0) or right, |s| < B.
template <int L>
__device__ __forceinline__ void shift_digits(int32_t (&d)[L], int s) {
  constexpr int B = Fmt<L>::B;
  constexpr int32_t kMask = (1 << B) - 1;
  if (s > 0) {
    int32_t low = 0;
#pragma unroll
    for (int i = 0; i < L; i++) {
      const int32_t x = d[i];
      d[i] = i == L - 1 ? static_cast<int32_t>(static_cast<uint32_t>(x) << s) | low
                        : ((static_cast<int32_t>(static_cast<uint32_t>(x) << s) & kMask) | low);
      low = x >> (B - s);
    }
  } else if (s < 0) {
    const int r = -s;
#pragma unroll
    for (int i = 0; i < L - 1; i++)
      d[i] = (d[i] >> r) | (static_cast<int32_t>(static_cast<uint32_t>(d[i + 1]) << (B - r)) & kMask);
    d[L - 1] >>= r;
  }
}

template <int L>
__device__ __forceinline__ uint32_t top_magnitude(const Num<L> &y) {
  const int32_t a = y.re[L - 1], b = y.im[L - 1];
  return max(static_cast<uint32_t>(a ^ (a >> 31)), static_cast<uint32_t>(b ^ (b >> 31)));
}

// Bring the larger component of a running product back to the middle of its
// band when it has left it (never for factors of unit modulus).
template <int L>
__device__ __forceinline__ void check(Num<L> &y) {
  constexpr int B = Fmt<L>::B;
  constexpr uint32_t lo = 1u << (B - 5), hi = 1u << (B - 2);
  const uint32_t m = top_magnitude(y);
  if (m - lo >= hi - lo) {
    const int s = m == 0u ? 0 : __clz(static_cast<int>(m)) - (32 - (B - 3));
    shift_digits<L>(y.re, s);
    shift_digits<L>(y.im, s);
    y.e -= s;
  }
}

// ---------------------------------------------------------------------------
// conversions
// ---------------------------------------------------------------------------

// Digits of an N-word magnitude below 2^(B L + 1), negated when neg.
template <int L, int N>
__device__ __forceinline__ void digits_of(const uint32_t (&x)[N], bool neg, int32_t (&d)[L]) {
  constexpr int B = Fmt<L>::B;
  constexpr int32_t kMask = (1 << B) - 1;
  int32_t t = 0;
#pragma unroll
  for (int i = 0; i < L; i++) {
    const int w = (B * i) >> 5, b = (B * i) & 31;
    uint32_t v = x[w] >> b;
    if (b != 0 && w + 1 < N) v |= x[w + 1] << (32 - b);
    int32_t u = i == L - 1 ? static_cast<int32_t>(v) : static_cast<int32_t>(v) & kMask;
    if (neg) u = -u;
    t += u;
    if (i == L - 1) {
      d[i] = t;
    } else {
      d[i] = t & kMask;
      t >>= B;
    }
  }
}

// A sum of NP doubles as sign and magnitude times 2^e (its leading bit found,
// -1: zero).  Up to two parts take 128 bits, which hold more than the digits
// of L <= 4; more take 256.
template <int NP>
struct Component {
  static constexpr int N = NP <= 2 ? 4 : 8;
  uint32_t m[N];
  bool neg;
  int32_t e;
  int lead;
  __device__ __forceinline__ explicit Component(const double *v) {
    if constexpr (NP <= 2) {
      double h = v[0], l = 0.0;
      if constexpr (NP == 2) two_sum(v[0], v[1], h, l);
      const wide::Comp c = wide::comp_from_dd(h, l);
      m[0] = c.m.w0, m[1] = c.m.w1, m[2] = c.m.w2, m[3] = c.m.w3;
      neg = c.s != 0u;
      e = c.e;
      lead = 127 - wide::clz128(c.m);
    } else {
      const qd::Comp c = qd::comp_from_parts<NP>(v);
#pragma unroll
      for (int i = 0; i < N; i++) m[i] = c.m.w[i];
      neg = c.s != 0u;
      e = c.e;
      lead = 255 - qd::clz256(c.m);
    }
  }
  // m 2^-s
  __device__ __forceinline__ void shift(int s) {
    if constexpr (NP <= 2) {
      const wide::Mag a{m[0], m[1], m[2], m[3]}, r = s >= 0 ? wide::shr(a, s) : wide::shl(a, -s);
      m[0] = r.w0, m[1] = r.w1, m[2] = r.w2, m[3] = r.w3;
    } else {
      qd::Mag a;
#pragma unroll
      for (int i = 0; i < N; i++) a.w[i] = m[i];
      a = s >= 0 ? qd::shr(a, s) : qd::shl(a, -s);
#pragma unroll
      for (int i = 0; i < N; i++) m[i] = a.w[i];
    }
  }
};

// y-kind digits to balanced ones (X kind): |d_i| <= 2^(B-1) below the top.
template <int L>
__device__ __forceinline__ void balance(int32_t (&d)[L]) {
  constexpr int B = Fmt<L>::B;
  constexpr int32_t kHalf = 1 << (B - 1), kMask = (1 << B) - 1;
  int32_t t = 0;
#pragma unroll
  for (int i = 0; i < L - 1; i++) {
    t += d[i] + kHalf;
    d[i] = (t & kMask) - kHalf;
    t >>= B;
  }
  d[L - 1] += t;
}

// Shift a y-kind number so that its modulus is within 2^(+-1/2) (up to the
// rounding of a single-precision estimate) of 2^(B (L - 1) + t); returns the
// base-2 logarithm of its modulus.
template <int L>
__device__ __forceinline__ float scale_modulus(Num<L> &y, int t) {
  const float r = static_cast<float>(y.re[L - 1]), i = static_cast<float>(y.im[L - 1]);
  const float lg = 0.5f * log2f(fmaf(r, r, i * i));
  const int s = t - __float2int_rn(lg);
  shift_digits<L>(y.re, s);
  shift_digits<L>(y.im, s);
  y.e -= s;
  return lg + static_cast<float>(y.e + s + Fmt<L>::B * (L - 1));
}

// What a conversion found out about a number.
struct Seen {
  bool bad;      // not finite, zero, or its components too far apart
  float log2m;   // base-2 logarithm of the modulus
  bool near_axis = false;  // components more than kSumNearAxis bits apart, or one zero
  bool real = false;       // no imaginary component
};

// Components further apart than this many bits are left to the general
// kernels, which hold each component to its own relative precision.
constexpr int kMaxSkew = 24;

// A complex number given as two sums of NP doubles, as a y-kind number of
// modulus near 2^(B (L - 1) + t).  Zero and non-finite numbers give 1 (bad).
template <int L, int NP>
__device__ __forceinline__ Num<L> from_parts(const double *v, int t, Seen &seen) {
  constexpr int B = Fmt<L>::B;
  bool finite = true;
#pragma unroll
  for (int i = 0; i < 2 * NP; i++)
    finite = finite && ((static_cast<unsigned long long>(__double_as_longlong(v[i])) >> 52) & 0x7ff) != 0x7ff;
  Num<L> y;
  if (!finite) {
    seen = Seen{true, 0.0f};
  } else {
    Component<NP> r(v), i(v + NP);
    if (r.lead >= 0 || i.lead >= 0) {
      // exponents of the leading bits
      const int tr = r.e + r.lead, ti = i.e + i.lead;
      const int top = r.lead < 0 ? ti : i.lead < 0 ? tr : max(tr, ti);
      const bool both = r.lead >= 0 && i.lead >= 0;
      seen.bad = both && (tr - ti > kMaxSkew || ti - tr > kMaxSkew);
      seen.near_axis = !both || tr - ti > kSumNearAxis || ti - tr > kSumNearAxis;
      seen.real = i.lead < 0;
      // leading bit of the larger component to bit B - 2 of the top digit
      y.e = top - (B * L - 2);
      if (r.lead >= 0) r.shift(y.e - r.e);
      if (i.lead >= 0) i.shift(y.e - i.e);
      digits_of<L>(r.m, r.neg, y.re);
      digits_of<L>(i.m, i.neg, y.im);
      seen.log2m = scale_modulus<L>(y, t);
      return y;
    }
    seen = Seen{true, 0.0f};
  }
#pragma unroll
  for (int i = 0; i < L; i++) y.re[i] = y.im[i] = 0;
  y.re[L - 1] = 1 << t;
  y.e = -(B * (L - 1) + t);
  return y;
}

// A y-kind number as a table entry.
template <int L>
__device__ __forceinline__ Num<L> as_factor(Num<L> y) {
  scale_modulus<L>(y, Fmt<L>::B - 1);
  balance<L>(y.re);
  balance<L>(y.im);
  return y;
}

// The product of real numbers y and X (digits as above), y's scale kept.
template <int L>
__device__ __forceinline__ void mul_real(const int32_t (&y)[L], const int32_t (&X)[L], int32_t (&r)[L]) {
  long long c[L];
#pragma unroll
  for (int k = 0; k < L; k++) {
    c[k] = 0;
#pragma unroll
    for (int i = k; i < L; i++) c[k] += static_cast<long long>(X[i]) * y[k + L - 1 - i];
  }
  fold<L>(c, r);
}

// 1 / x for a table entry x = (a + ib) 2^(B L - 1 + e), a^2 + b^2 within a
// factor 2 of 1: conj(x) / (a^2 + b^2), the real reciprocal by Newton's
// iteration r <- r (2 - n r) from single precision; each step doubles the
// correct bits (21, 42, 84, 168, 336).  y kind.  (A complex iteration takes
// four times the multiply-adds; a double-precision start saves one step but
// takes some 25 instructions of the FP64 pipe, 400 cycles of an SM each time.)
template <int L>
__device__ __forceinline__ Num<L> reciprocal(const Num<L> &X) {
  constexpr int B = Fmt<L>::B;
  constexpr int32_t kMask = (1 << B) - 1;
  int32_t n[L], r[L];
  {
    long long c[L];
#pragma unroll
    for (int k = 0; k < L; k++) {
      c[k] = 0;
#pragma unroll
      for (int i = k; i < L; i++) {
        c[k] += static_cast<long long>(X.re[i]) * X.re[k + L - 1 - i];
        c[k] += static_cast<long long>(X.im[i]) * X.im[k + L - 1 - i];
      }
    }
    fold<L>(c, n);  // scale 2^(B L - 1)
  }
  const float f = static_cast<float>(n[L - 1]) * (1.0f / static_cast<float>(1 << (B - 1)));
#pragma unroll
  for (int i = 0; i < L - 1; i++) r[i] = 0;
  r[L - 1] = __float2int_rn(__fdividef(static_cast<float>(1 << (B - 3)), f));  // scale 2^(B L - 3)
  balance<L>(n);
  constexpr int kSteps = L == 3 ? 2 : L == 4 ? 3 : 4;
#pragma unroll 1
  for (int k = 0; k < kSteps; k++) {
    int32_t u[L], w[L];
    mul_real<L>(r, n, u);  // 1 + d at scale 2^(B L - 3)
    int32_t t = 0;         // 2 - u, then shifted up to scale 2^(B L - 1)
#pragma unroll
    for (int i = 0; i < L; i++) {
      t += (i == L - 1 ? 1 << (B - 2) : 0) - u[i];
      if (i < L - 1) {
        w[i] = t & kMask;
        t >>= B;
      } else {
        w[i] = t;
      }
    }
    shift_digits<L>(w, 2);
    balance<L>(w);
    mul_real<L>(r, w, u);
#pragma unroll
    for (int i = 0; i < L; i++) r[i] = u[i];
  }
  Num<L> y;
  int32_t minus[L];
#pragma unroll
  for (int i = 0; i < L; i++) minus[i] = -X.im[i];
  mul_real<L>(r, X.re, y.re);
  mul_real<L>(r, minus, y.im);
  y.e = -(B * L - 1) - (B * L - 3) - X.e;
  return y;
}

}  // namespace fx
}  // namespace pe
