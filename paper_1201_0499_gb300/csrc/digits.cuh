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

#include "wide8.cuh"

namespace pe {
namespace fx {

// Per digit count: radix, words of the accumulation window (kernels_sum.cu),
// and the least bit of the window that a derivative's largest term may have
// as its leading one.
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

// Digits of floor(m / 2^sh) for a 256-bit magnitude, 0 <= sh, the quotient
// below 2^(B L + 1).
template <int L>
__device__ __forceinline__ void digits_of(const qd::Mag &m, int sh, bool neg, int32_t (&d)[L]) {
  constexpr int B = Fmt<L>::B;
  constexpr int32_t kMask = (1 << B) - 1;
  const qd::Mag x = qd::shr(m, sh);
  int32_t t = 0;
#pragma unroll
  for (int i = 0; i < L; i++) {
    const int w = (B * i) >> 5, b = (B * i) & 31;
    uint32_t v = x.w[w] >> b;
    if (b != 0 && w + 1 < qd::L) v |= x.w[w + 1] << (32 - b);
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
    const qd::Comp r = qd::comp_from_parts<NP>(v), i = qd::comp_from_parts<NP>(v + NP);
    const int zr = qd::clz256(r.m), zi = qd::clz256(i.m);
    if (zr < 256 || zi < 256) {
      // exponents of the leading bits
      const int tr = r.e + 255 - zr, ti = i.e + 255 - zi;
      const int top = zr == 256 ? ti : zi == 256 ? tr : max(tr, ti);
      seen.bad = zr < 256 && zi < 256 && (tr - ti > kMaxSkew || ti - tr > kMaxSkew);
      // leading bit of the larger component to bit B - 2 of the top digit
      y.e = top - (B * L - 2);
      // (a shift of the magnitude at all: its leading bit is at 250 or below,
      // and cancelling parts may leave it lower; then the low digits are short)
      const int sr = zr == 256 ? 0 : y.e - r.e, si = zi == 256 ? 0 : y.e - i.e;
      const qd::Mag rm = sr < 0 ? qd::shl(r.m, -sr) : r.m, im = si < 0 ? qd::shl(i.m, -si) : i.m;
      digits_of<L>(rm, max(sr, 0), r.s != 0u, y.re);
      digits_of<L>(im, max(si, 0), i.s != 0u, y.im);
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

// 1 / x for a table entry x, by Newton's iteration r <- r (2 - x r) from the
// double-precision reciprocal; each step doubles the correct bits (51, 102,
// 204).  y kind.
template <int L>
__device__ __forceinline__ Num<L> reciprocal(const Num<L> &X) {
  constexpr int B = Fmt<L>::B;
  // modulus of (a + ib) within 2^(+-1/2) of 2^(B-1)
  const double s = 1.0 / static_cast<double>(1 << B);
  const double a = fma(static_cast<double>(X.re[L - 2]), s, static_cast<double>(X.re[L - 1]));
  const double b = fma(static_cast<double>(X.im[L - 2]), s, static_cast<double>(X.im[L - 1]));
  const double q = 1.0 / fma(a, a, b * b);
  const double v[2] = {a * q, -(b * q)};
  Seen unused;
  // v ~ 1 / (a + ib), X = (a + ib) 2^(B (L - 1) + e)
  Num<L> r = from_parts<L, 1>(v, B - 3, unused);
  r.e -= B * (L - 1) + X.e;
  constexpr int kSteps = L == 3 ? 1 : L == 4 ? 2 : 3;
#pragma unroll 1
  for (int k = 0; k < kSteps; k++) {
    Num<L> u = r;
    mul<L>(u, X);  // 1 + d, modulus near 2^(B L - 3 + ...)
    // 2 - u: the unit sits at bit -e
    const int bit = -u.e;
    const int w = (bit + 1) / B, p = (bit + 1) - w * B;
    int32_t t = 0, m = 0;
#pragma unroll
    for (int i = 0; i < L; i++) {
      t += (i == w ? (1 << p) : 0) - u.re[i];
      m -= u.im[i];
      if (i < L - 1) {
        u.re[i] = t & ((1 << B) - 1);
        t >>= B;
        u.im[i] = m & ((1 << B) - 1);
        m >>= B;
      } else {
        u.re[i] = t;
        u.im[i] = m;
      }
    }
    const Num<L> U = as_factor<L>(u);
    mul<L>(r, U);
  }
  return r;
}

}  // namespace fx
}  // namespace pe
