// Evaluation of f and its Jacobian from the monomials' values alone (all
// precisions).
//
// Method.  With V_t = c_t x^(a_t) the value of monomial t (power table of
// Section 3.1, one product per variable, coefficient included),
//   f_p = sum_t V_t,      x_i df_p/dx_i = sum_t a_{t,i} V_t,
// so the derivatives of a monomial cost integer additions instead of the
// forward and backward products of Section 3.2: k complex products per
// monomial instead of #(a >= 2) + 3k - 3, and one product with 1 / x_i for
// each entry of J at the end.  The error of an entry of J is relative to
// sum_t a_{t,i} |V_t| / |x_i|, the normwise measure of the accuracy target.
// It needs x_i != 0; points for which that fails, and those with non-finite
// coordinates, exponents near the range of a double or a coordinate whose
// components are more than 2^24 apart, are flagged by the power table's kernel,
// and the general kernels (kernels.cu, kernels_wide.cu, kernels_qd.cu)
// evaluate them.
//
// Near-axis points (double-double).  A number's components share its exponent
// here, so the smaller one errs like the larger.  That shows where a term's
// smaller component comes from smaller components alone, (a + ib)(c + id) with
// b << a, d << c: not with one factor off the axes, whose components then
// reach both.  The general kernels compute components apart; so a point whose
// every coordinate lies near an axis (components more than 2^kSumNearAxis apart)
// is left to them, where the coefficients of a polynomial or of a derivative
// lie near one too (`axial`, by the sums of their parts).  Real points of real
// systems stay: their imaginary parts are exact zeros.  Double and quad-double
// need no such rule: 88 bits hold 53 down to 2^-24, and the general
// quad-double kernels share exponents in the same way.  (Worst error of a
// component over its terms' parts, real coefficients, components of the points
// 2^-8, 2^-16, 2^-22 apart: general 2^-103.5, 2^-103.3, 2^-103.6, from values
// 2^-97, 2^-89, 2^-82.5; on the unit circle 2^-104.4 and 2^-105.9.  Points on
// the circle: (2 2^-kSumNearAxis)^n of them lie near an axis in n coordinates.)
//
// Layout.  One block works on one tile of 1, 2 or 4 points of a system and
// a run of polynomials.  The tile's power table (digits.cuh) is copied to
// shared memory once.  For each polynomial, chunks of monomials:
//   A  one thread per (monomial, point) multiplies its k factors in
//      registers (two monomials where shared memory has room for the values);
//   -  the block agrees on the largest exponent per point, and every value is
//      stored as a W-word two's complement integer below it (the window);
//      (the leading bit of a sum's terms is kept beside it and falls with the
//      sum when a later chunk raises the window: below kKeep, the terms were
//      too small for the window, see own_windows)
//   B  one thread per (variable, component, point) adds the values of the
//      monomials that hold its variable, times the exponent, from a list made
//      at create; four list entries at a time, without branches.  (Additions
//      alone, over lists ordered by exponent with a second running sum, ran
//      slower: a warp holds several lists, whose steps differ.)
// Integer sums are exact, so they depend on the order only through the values'
// truncation to the window.  No lane pairs, no shuffles in the products, no
// read-modify-write of J.
//
// Bound: the 64-bit multiply-adds of the products (digits.cuh).
#include <cuda_runtime.h>

#include <cstdint>

#include "digits.cuh"
#include "internal.h"
#include "words.cuh"

namespace pe {

using fx::Fmt;
using fx::Num;

namespace {

template <int L>
constexpr int kParts = L == 8 ? 4 : 2;  // 16-byte parts of a table entry

// Table entries: digits in 16-byte parts, part-major over the points of the
// tile; the exponent in the last part (L = 3) or in an array of its own.
// Neighbouring parts are exchanged in every second 128 bytes, so that the
// lanes of different monomials, which read the same part of different
// entries, meet in the same banks half as often.
__device__ __forceinline__ int part_swap(unsigned idx, int lg) { return static_cast<int>(idx >> (2 - lg)) & 1; }

template <int L>
__device__ __forceinline__ Num<L> load_factor(const int4 *tab, const int32_t *exps, unsigned idx, int lg, int q) {
  const int4 *p = tab + (static_cast<size_t>(idx * kParts<L>) << lg) + q;
  const int sw = part_swap(idx, lg);
  Num<L> x;
  if constexpr (L == 3) {
    const int4 a = p[sw << lg], b = p[(1 ^ sw) << lg];
    x.re[0] = a.x, x.re[1] = a.y, x.re[2] = a.z;
    x.im[0] = a.w, x.im[1] = b.x, x.im[2] = b.y;
    x.e = b.z;
  } else {
#pragma unroll
    for (int h = 0; h < L / 4; h++) {
      const int4 a = p[(h ^ sw) << lg], b = p[((L / 4 + h) ^ sw) << lg];
      x.re[4 * h] = a.x, x.re[4 * h + 1] = a.y, x.re[4 * h + 2] = a.z, x.re[4 * h + 3] = a.w;
      x.im[4 * h] = b.x, x.im[4 * h + 1] = b.y, x.im[4 * h + 2] = b.z, x.im[4 * h + 3] = b.w;
    }
    x.e = exps[(static_cast<size_t>(idx) << lg) + q];
  }
  return x;
}

template <int L>
__device__ __forceinline__ void store_factor(int4 *tab, int32_t *exps, unsigned idx, int lg, int q, const Num<L> &x) {
  int4 *p = tab + (static_cast<size_t>(idx * kParts<L>) << lg) + q;
  const int sw = part_swap(idx, lg);
  if constexpr (L == 3) {
    p[sw << lg] = make_int4(x.re[0], x.re[1], x.re[2], x.im[0]);
    p[(1 ^ sw) << lg] = make_int4(x.im[1], x.im[2], x.e, 0);
  } else {
#pragma unroll
    for (int h = 0; h < L / 4; h++) {
      p[(h ^ sw) << lg] = make_int4(x.re[4 * h], x.re[4 * h + 1], x.re[4 * h + 2], x.re[4 * h + 3]);
      p[((L / 4 + h) ^ sw) << lg] = make_int4(x.im[4 * h], x.im[4 * h + 1], x.im[4 * h + 2], x.im[4 * h + 3]);
    }
    exps[(static_cast<size_t>(idx) << lg) + q] = x.e;
  }
}

// a += b over W words.
template <int W>
__device__ __forceinline__ void add_words(uint32_t (&a)[W], const uint32_t (&b)[W]) {
  static_assert(W == 5 || W == 6 || W == 10, "window sizes of Fmt");
  if constexpr (W == 5) {
    asm("add.cc.u32 %0, %0, %5;\n\taddc.cc.u32 %1, %1, %6;\n\taddc.cc.u32 %2, %2, %7;\n\t"
        "addc.cc.u32 %3, %3, %8;\n\taddc.u32 %4, %4, %9;"
        : "+r"(a[0]), "+r"(a[1]), "+r"(a[2]), "+r"(a[3]), "+r"(a[4])
        : "r"(b[0]), "r"(b[1]), "r"(b[2]), "r"(b[3]), "r"(b[4]));
  } else if constexpr (W == 6) {
    asm("add.cc.u32 %0, %0, %6;\n\taddc.cc.u32 %1, %1, %7;\n\taddc.cc.u32 %2, %2, %8;\n\t"
        "addc.cc.u32 %3, %3, %9;\n\taddc.cc.u32 %4, %4, %10;\n\taddc.u32 %5, %5, %11;"
        : "+r"(a[0]), "+r"(a[1]), "+r"(a[2]), "+r"(a[3]), "+r"(a[4]), "+r"(a[5])
        : "r"(b[0]), "r"(b[1]), "r"(b[2]), "r"(b[3]), "r"(b[4]), "r"(b[5]));
  } else {
    asm("add.cc.u32 %0, %0, %10;\n\taddc.cc.u32 %1, %1, %11;\n\taddc.cc.u32 %2, %2, %12;\n\t"
        "addc.cc.u32 %3, %3, %13;\n\taddc.cc.u32 %4, %4, %14;\n\taddc.cc.u32 %5, %5, %15;\n\t"
        "addc.cc.u32 %6, %6, %16;\n\taddc.cc.u32 %7, %7, %17;\n\taddc.cc.u32 %8, %8, %18;\n\t"
        "addc.u32 %9, %9, %19;"
        : "+r"(a[0]), "+r"(a[1]), "+r"(a[2]), "+r"(a[3]), "+r"(a[4]), "+r"(a[5]), "+r"(a[6]), "+r"(a[7]), "+r"(a[8]),
          "+r"(a[9])
        : "r"(b[0]), "r"(b[1]), "r"(b[2]), "r"(b[3]), "r"(b[4]), "r"(b[5]), "r"(b[6]), "r"(b[7]), "r"(b[8]),
          "r"(b[9]));
  }
}

// (e + 2^32 o) += k z (mod 2^(32 W): two's complement): the products of the
// even words of z in e, those of the odd words in o, so that every 64-bit
// product adds into one aligned register pair.  (One accumulator for both
// costs a dozen register moves a call, on the pipe of the multiply-adds.)
template <int W>
__device__ __forceinline__ void add_times(uint32_t (&e)[W], uint32_t (&o)[W - 1], const uint32_t (&z)[W], uint32_t k) {
  if constexpr (W == 5) {
    asm(
        "mad.lo.cc.u32 %0, %9, %14, %0;\n\tmadc.hi.cc.u32 %1, %9, %14, %1;\n\t"
        "madc.lo.cc.u32 %2, %11, %14, %2;\n\tmadc.hi.cc.u32 %3, %11, %14, %3;\n\t"
        "madc.lo.u32 %4, %13, %14, %4;\n\tmad.lo.cc.u32 %5, %10, %14, %5;\n\t"
        "madc.hi.cc.u32 %6, %10, %14, %6;\n\tmadc.lo.cc.u32 %7, %12, %14, %7;\n\t"
        "madc.hi.u32 %8, %12, %14, %8;"
        : "+r"(e[0]), "+r"(e[1]), "+r"(e[2]), "+r"(e[3]), "+r"(e[4]),
          "+r"(o[0]), "+r"(o[1]), "+r"(o[2]), "+r"(o[3])
        : "r"(z[0]), "r"(z[1]), "r"(z[2]), "r"(z[3]), "r"(z[4]), "r"(k));
  } else if constexpr (W == 6) {
    asm(
        "mad.lo.cc.u32 %0, %11, %17, %0;\n\tmadc.hi.cc.u32 %1, %11, %17, %1;\n\t"
        "madc.lo.cc.u32 %2, %13, %17, %2;\n\tmadc.hi.cc.u32 %3, %13, %17, %3;\n\t"
        "madc.lo.cc.u32 %4, %15, %17, %4;\n\tmadc.hi.u32 %5, %15, %17, %5;\n\t"
        "mad.lo.cc.u32 %6, %12, %17, %6;\n\tmadc.hi.cc.u32 %7, %12, %17, %7;\n\t"
        "madc.lo.cc.u32 %8, %14, %17, %8;\n\tmadc.hi.cc.u32 %9, %14, %17, %9;\n\t"
        "madc.lo.u32 %10, %16, %17, %10;"
        : "+r"(e[0]), "+r"(e[1]), "+r"(e[2]), "+r"(e[3]), "+r"(e[4]), "+r"(e[5]),
          "+r"(o[0]), "+r"(o[1]), "+r"(o[2]), "+r"(o[3]), "+r"(o[4])
        : "r"(z[0]), "r"(z[1]), "r"(z[2]), "r"(z[3]), "r"(z[4]), "r"(z[5]), "r"(k));
  } else {
    asm(
        "mad.lo.cc.u32 %0, %19, %29, %0;\n\tmadc.hi.cc.u32 %1, %19, %29, %1;\n\t"
        "madc.lo.cc.u32 %2, %21, %29, %2;\n\tmadc.hi.cc.u32 %3, %21, %29, %3;\n\t"
        "madc.lo.cc.u32 %4, %23, %29, %4;\n\tmadc.hi.cc.u32 %5, %23, %29, %5;\n\t"
        "madc.lo.cc.u32 %6, %25, %29, %6;\n\tmadc.hi.cc.u32 %7, %25, %29, %7;\n\t"
        "madc.lo.cc.u32 %8, %27, %29, %8;\n\tmadc.hi.u32 %9, %27, %29, %9;\n\t"
        "mad.lo.cc.u32 %10, %20, %29, %10;\n\tmadc.hi.cc.u32 %11, %20, %29, %11;\n\t"
        "madc.lo.cc.u32 %12, %22, %29, %12;\n\tmadc.hi.cc.u32 %13, %22, %29, %13;\n\t"
        "madc.lo.cc.u32 %14, %24, %29, %14;\n\tmadc.hi.cc.u32 %15, %24, %29, %15;\n\t"
        "madc.lo.cc.u32 %16, %26, %29, %16;\n\tmadc.hi.cc.u32 %17, %26, %29, %17;\n\t"
        "madc.lo.u32 %18, %28, %29, %18;"
        : "+r"(e[0]), "+r"(e[1]), "+r"(e[2]), "+r"(e[3]), "+r"(e[4]), "+r"(e[5]), "+r"(e[6]), "+r"(e[7]), "+r"(e[8]), "+r"(e[9]),
          "+r"(o[0]), "+r"(o[1]), "+r"(o[2]), "+r"(o[3]), "+r"(o[4]), "+r"(o[5]), "+r"(o[6]), "+r"(o[7]), "+r"(o[8])
        : "r"(z[0]), "r"(z[1]), "r"(z[2]), "r"(z[3]), "r"(z[4]), "r"(z[5]), "r"(z[6]), "r"(z[7]), "r"(z[8]), "r"(z[9]), "r"(k));
  }
}

// ---------------------------------------------------------------------------
// outputs
// ---------------------------------------------------------------------------

// A sum (window words, exponent of bit 0) to the doubles of one output component.
template <int L>
__device__ __forceinline__ void store_sum(double *p, uint32_t (&z)[Fmt<L>::W], int32_t e0) {
  constexpr int W = Fmt<L>::W;
  const int lead = lead_words<W>(z);
  const int s = 32 * W - 3 - lead;  // the headroom keeps lead below 32 W - 2
  if (lead >= 0 || z[W - 1]) shl_words<W>(z, min(s, 32 * W - 1));
  const int32_t e = e0 - min(s, 32 * W - 1);
  if constexpr (L == 8) {
    qd::Acc a;
#pragma unroll
    for (int i = 0; i < qd::LA; i++) a.w[i] = z[W - qd::LA + i];
    a.e = e + 32 * (W - qd::LA);
    double o[4];
    qd::acc_to_qd(a, o);
    reinterpret_cast<double2 *>(p)[0] = make_double2(o[0], o[1]);
    reinterpret_cast<double2 *>(p)[1] = make_double2(o[2], o[3]);
  } else {
    const dd r = words_to_dd(z[W - 4], z[W - 3], z[W - 2], z[W - 1], e + 32 * (W - 4));
    if constexpr (L == 4)
      *reinterpret_cast<double2 *>(p) = make_double2(r.h, r.l);
    else
      *p = r.h;  // normalised: the value rounded to nearest
  }
}

// One component of a product to the output: rounded at bit kRound of the
// digits, which is above the product's error, so that exact results come out
// exact.
template <int L>
__device__ __forceinline__ void store_product(double *p, const int32_t (&d)[L], int32_t e) {
  constexpr int NW = kPackWords<L>;
  constexpr int kRound = L == 8 ? 10 : 8;
  uint32_t w[NW];
  pack_digits<L, NW>(d, w);
  uint32_t carry = 1u << (kRound - 1);
#pragma unroll
  for (int i = 0; i < NW; i++) {
    const uint32_t s = w[i] + carry;
    carry = s < carry ? 1u : 0u;
    w[i] = s;
  }
  w[0] &= ~((1u << kRound) - 1u);
  if constexpr (L == 8) {
    qd::Acc a;
#pragma unroll
    for (int i = 0; i < qd::LA; i++) a.w[i] = __funnelshift_r(w[i], w[i + 1], kRound);
    a.e = e + kRound;
    double o[4];
    qd::acc_to_qd(a, o);
    reinterpret_cast<double2 *>(p)[0] = make_double2(o[0], o[1]);
    reinterpret_cast<double2 *>(p)[1] = make_double2(o[2], o[3]);
  } else if constexpr (L == 4) {
    const dd r = words_to_dd(w[0], w[1], w[2], w[3], e);
    *reinterpret_cast<double2 *>(p) = make_double2(r.h, r.l);
  } else {
    *p = words_to_dd(0u, w[0], w[1], w[2], e - 32).h;
  }
}

template <int L>
__device__ __forceinline__ void store_zero(double *p) {
  if constexpr (L == 3) {
    *p = 0.0;
  } else {
    reinterpret_cast<double2 *>(p)[0] = make_double2(0.0, 0.0);
    if constexpr (L == 8) reinterpret_cast<double2 *>(p)[1] = make_double2(0.0, 0.0);
  }
}

template <int L>
constexpr int kComp = L == 3 ? 1 : L == 4 ? 2 : 4;  // doubles per output component

// ---------------------------------------------------------------------------
// tables and coefficients
// ---------------------------------------------------------------------------

template <int L>
__device__ __forceinline__ Num<L> read_number(const double *p, int t, fx::Seen &seen) {
  constexpr int NP = kComp<L>;
  double v[2 * NP];
#pragma unroll
  for (int i = 0; i < 2 * NP; i++) v[i] = p[i];
  return fx::from_parts<L, NP>(v, t, seen);
}

template <int L>
__global__ void sum_coef_kernel(const double *coef, const int32_t *order, const int32_t *fac_ptr, const uint32_t *fac,
                                int32_t *out, int64_t M) {
  constexpr int CW = kSumCoefWords<L>;
  const int64_t stride = static_cast<int64_t>(gridDim.x) * blockDim.x;
  for (int64_t t = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x; t < M; t += stride) {
    fx::Seen seen;
    Num<L> y = read_number<L>(coef + static_cast<int64_t>(order[t]) * 2 * kComp<L>, Fmt<L>::B - 3, seen);
    bool zero = true;
    for (int i = 0; i < 2 * kComp<L>; i++) zero = zero && coef[static_cast<int64_t>(order[t]) * 2 * kComp<L> + i] == 0.0;
    if (zero) {
#pragma unroll
      for (int i = 0; i < L; i++) y.re[i] = y.im[i] = 0;
      y.e = fx::kZeroExp;
    }
    int32_t *o = out + t * CW;
#pragma unroll
    for (int i = 0; i < L; i++) o[i] = y.re[i], o[L + i] = y.im[i];
    o[2 * L] = y.e;
    o[2 * L + 1] = fac_ptr[t];
    o[2 * L + 2] = fac_ptr[t + 1] - fac_ptr[t];
    o[2 * L + 3] = fac_ptr[t + 1] > fac_ptr[t] ? static_cast<int32_t>(fac[fac_ptr[t]]) : 0;
  }
}

// One thread per (point, variable) and role: role 0 writes x, x^2, ..,
// x^emax, role 1 writes 1 / x.  Points past the last repeat it.
template <int L>
__global__ void __launch_bounds__(128) sum_powers(const SumParams sp) {
  let_next_start();
  const int64_t stride = static_cast<int64_t>(gridDim.x) * blockDim.x;
  for (int64_t i = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x; i < 2 * sp.power_total; i += stride) {
    const bool inverse = i >= sp.power_total;
    int64_t local = inverse ? i - sp.power_total : i;
    int s = 0;
    if (sp.single_P < 0) {
      int lo = 0, hi = sp.count;
      while (hi - lo > 1) {
        const int mid = (lo + hi) >> 1;
        if (sp.prefix[mid] <= local) lo = mid; else hi = mid;
      }
      s = lo;
      local -= sp.prefix[lo];
    }
    const SumSys ss = sp.sum_sys[s];
    const SysDesc sd = sp.sys[s];
    const int P = sp.single_P >= 0 ? sp.single_P : sd.P;
    const int lg = sp.lg;
    const int n = sd.n;
    const int tile_entries = n << lg;
    const int tile = static_cast<int>(local / tile_entries);
    const int r = static_cast<int>(local - static_cast<int64_t>(tile) * tile_entries);
    const int v = r >> lg, q = r & ((1 << lg) - 1);
    const int qg = (tile << lg) + q;
    const int qc = min(qg, P - 1);
    fx::Seen seen;
    Num<L> y = read_number<L>(sp.points + (sd.pt_off + static_cast<int64_t>(v) * P + qc) * 2 * kComp<L>, Fmt<L>::B - 1, seen);
    const bool bad = seen.bad || fabsf(seen.log2m) > ss.most_log2;
    if constexpr (L == 4) {
      if (seen.near_axis && ss.axial && !inverse && qg < P) {
        const unsigned one = seen.real ? 1u : 0x10001u;
        const unsigned c = atomicAdd(sp.near + ss.flag_off + qg, one) + one;
        if ((c & 0xffffu) == static_cast<unsigned>(n) && (ss.axial == kAxial || c >> 16)) {  // the last one sees it
          sp.flags[ss.flag_off + qg] = 1;
          *sp.any = 1;
        }
      }
    }
    if (bad) {
      if (!inverse) {
        sp.flags[ss.flag_off + qc] = 1;
        *sp.any = 1;
      }
#pragma unroll
      for (int k = 0; k < L; k++) y.re[k] = y.im[k] = 0;
      y.re[L - 1] = 1 << (Fmt<L>::B - 1);
      y.e = -(Fmt<L>::B * L - 1);
    }
    fx::balance<L>(y.re);
    fx::balance<L>(y.im);
    const Num<L> x = y;
    const int levels = sd.emax;
    const unsigned entries = static_cast<unsigned>(levels) * n;
    unsigned char *blob = sp.table + ss.tab_off + static_cast<size_t>(tile) * sum_blob_bytes(L, n, levels, lg);
    int4 *tab = reinterpret_cast<int4 *>(blob);
    int32_t *exps = reinterpret_cast<int32_t *>(blob + (static_cast<size_t>(entries) * kParts<L> * 16 << lg));
    if (inverse) {
      unsigned char *ib = blob + sum_tab_bytes(L, n, levels, lg);
      const Num<L> r1 = fx::as_factor<L>(fx::reciprocal<L>(x));
      store_factor<L>(reinterpret_cast<int4 *>(ib),
                      reinterpret_cast<int32_t *>(ib + (static_cast<size_t>(n) * kParts<L> * 16 << lg)), v, lg, q, r1);
      continue;
    }
    store_factor<L>(tab, exps, v, lg, q, x);
    // x^a = x^(a - h) x^h with h = floor(a/2): error depth O(log a)
    for (int a = 2; a <= levels; a++) {
      const int h = a >> 1, g = a - h;
      Num<L> u = g == 1 ? x : load_factor<L>(tab, exps, (g - 1) * n + v, lg, q);
      fx::mul<L>(u, h == 1 ? x : load_factor<L>(tab, exps, (h - 1) * n + v, lg, q));
      store_factor<L>(tab, exps, (a - 1) * n + v, lg, q, fx::as_factor<L>(u));
    }
  }
}

// ---------------------------------------------------------------------------
// the evaluation
// ---------------------------------------------------------------------------

// Shared memory of a block (bytes from its start): the tile's table, the
// values of a chunk, the sums.
template <int L>
struct Win {  // a window integer in memory: 16-byte parts and the rest
  static constexpr int W = Fmt<L>::W, Q = W / 4, R = W % 4;
};

template <int L>
__device__ __forceinline__ void load_window(const int4 *quads, const int32_t *rest, int rows, int row, uint32_t (&z)[Fmt<L>::W]) {
  constexpr int Q = Win<L>::Q, R = Win<L>::R;
#pragma unroll
  for (int h = 0; h < Q; h++) {
    const int4 a = quads[h * rows + row];
    z[4 * h] = a.x, z[4 * h + 1] = a.y, z[4 * h + 2] = a.z, z[4 * h + 3] = a.w;
  }
  if constexpr (R == 1) {
    z[4 * Q] = rest[row];
  } else {
    const int2 a = reinterpret_cast<const int2 *>(rest)[row];
    z[4 * Q] = a.x, z[4 * Q + 1] = a.y;
  }
}

template <int L>
__device__ __forceinline__ void store_window(int4 *quads, int32_t *rest, int rows, int row, const uint32_t (&z)[Fmt<L>::W]) {
  constexpr int Q = Win<L>::Q, R = Win<L>::R;
#pragma unroll
  for (int h = 0; h < Q; h++) quads[h * rows + row] = make_int4(z[4 * h], z[4 * h + 1], z[4 * h + 2], z[4 * h + 3]);
  if constexpr (R == 1)
    rest[row] = z[4 * Q];
  else
    reinterpret_cast<int2 *>(rest)[row] = make_int2(z[4 * Q], z[4 * Q + 1]);
}

// The value of monomial t at point q of the tile.  Its record holds the
// coefficient's digits and exponent, the place and number of its factors and
// the first of them, so that one load leads to the first product.
template <int L>
__device__ __forceinline__ Num<L> monomial_value(const SumParams &sp, int t, const int4 *tab, const int32_t *exps, int lg,
                                                 int q) {
  constexpr int CW = kSumCoefWords<L>;
  int32_t r[CW];
  const int4 *co = reinterpret_cast<const int4 *>(sp.coef + static_cast<size_t>(t) * CW);
#pragma unroll
  for (int i = 0; i < CW / 4; i++) {
    const int4 x = __ldg(co + i);
    r[4 * i] = x.x, r[4 * i + 1] = x.y, r[4 * i + 2] = x.z, r[4 * i + 3] = x.w;
  }
  Num<L> y;
#pragma unroll
  for (int i = 0; i < L; i++) y.re[i] = r[i], y.im[i] = r[L + i];
  y.e = r[2 * L];
  const int fb = r[2 * L + 1], fe = fb + r[2 * L + 2];
  unsigned idx = static_cast<unsigned>(r[2 * L + 3]);
#pragma unroll 1
  for (int j = fb; j < fe; j++) {
    const Num<L> x = load_factor<L>(tab, exps, idx, lg, q);
    if (j + 1 < fe) idx = __ldg(sp.fac + j + 1);
    fx::mul<L>(y, x);
    if (((j - fb) & (fx::kCheckEvery - 1)) == fx::kCheckEvery - 1) fx::check<L>(y);
  }
  return y;
}

// The exponent bound of a value: |y| < 2^value_top.
template <int L>
__device__ __forceinline__ int value_top(const Num<L> &y) {
  const int e = y.e + Fmt<L>::B * (L - 1) + 32 - __clz(static_cast<int>(fx::top_magnitude<L>(y)));
  return max(e, fx::kZeroExp);
}

// A component's digits (exponent e) as a window integer below 2^E: bit 0 at
// exponent E - (32 W - 1 - hb).
template <int L>
__device__ __forceinline__ void to_window(const int32_t (&d)[L], int32_t e, int E, int hb, uint32_t (&z)[Fmt<L>::W]) {
  constexpr int W = Fmt<L>::W, NW = kPackWords<L>;
  uint32_t p[NW];
  pack_digits<L, NW>(d, p);
#pragma unroll
  for (int i = 0; i < W; i++) z[i] = i < W - NW ? 0u : p[i - (W - NW)];
  sar_words<W>(z, max(E - e - 32 * NW + 1 + hb, 0));
}

// The top B L - 1 bits of a window integer (exponent of bit 0: e0), counted
// from two above bit `lead`, as y-kind digits, and their exponent.
template <int L>
__device__ __forceinline__ void top_digits(uint32_t (&z)[Fmt<L>::W], int lead, int32_t e0, int32_t (&d)[L], int32_t &e) {
  constexpr int B = Fmt<L>::B, W = Fmt<L>::W, o0 = 32 * W + 1 - B * L;
  const int sh = min(32 * W - 3 - lead, 32 * W - 1);
  shl_words<W>(z, sh);
#pragma unroll
  for (int i = 0; i < L; i++) {
    const int w = (o0 + B * i) >> 5, b = (o0 + B * i) & 31;
    d[i] = i == L - 1 ? static_cast<int32_t>(z[W - 1]) >> (33 - B)
                      : static_cast<int32_t>(__funnelshift_r(z[w], z[w + 1], b)) & ((1 << B) - 1);
  }
  e = e0 - sh + o0;
}

// The lanes that hold the parts of f: eight tasks of 2^lg points, aligned.
__device__ __forceinline__ unsigned lanes_of_parts(int lane, int lg) {
  const int count = 2 * kSumParts << lg;  // 8, 16 or 32
  return count == 32 ? 0xffffffffu : ((1u << count) - 1u) << (lane & ~(count - 1));
}

// One entry of J: the sums of its components (window integers, exponent of
// bit 0) times 1 / x_v.
template <int L>
__device__ __forceinline__ void finish_entry(uint32_t (&zr)[Fmt<L>::W], uint32_t (&zi)[Fmt<L>::W], int32_t e0,
                                             const Num<L> &inv, double *o) {
  constexpr int W = Fmt<L>::W;
  const int lead = max(lead_words<W>(zr), lead_words<W>(zi));
  Num<L> y;
  top_digits<L>(zr, lead, e0, y.re, y.e);
  top_digits<L>(zi, lead, e0, y.im, y.e);
  fx::mul<L>(y, inv);
  store_product<L>(o, y.re, y.e);
  store_product<L>(o + kComp<L>, y.im, y.e);
}

// The entries of J at point q (of the tile) whose every term lies so far
// below the polynomial's largest monomial that the shared window cut them
// short (not set in `kept`): their monomials' values once more, each sum in a
// window of its own.  Variables sub, sub + subs, ...; o: the entry of variable 0.
template <int L>
__device__ __forceinline__ void own_windows(const SumParams &sp, int gp, const int32_t *kept, const int4 *tab,
                                         const int32_t *exps, const int4 *inv4, const int32_t *inve, int lg, int q, int hb,
                                         int sub, int subs, double *Jp, int P) {
  constexpr int W = Fmt<L>::W;
  const SumPoly sy = sp.polys[gp];
  const int t0 = sp.poly_ptr[gp], blocks = (sp.poly_ptr[gp + 1] - t0 + kSumBlock - 1) / kSumBlock;
  for (int i = sub; i < sy.act_n; i += subs) {
    const int row = ((2 * i) << lg) + q;
    if (kept[row]) continue;
    int E = fx::kZeroExp;
    uint32_t zr[W], zi[W];
#pragma unroll
    for (int k = 0; k < W; k++) zr[k] = zi[k] = 0u;
    for (int b = 0; b < blocks; b++) {
      const int32_t *hq = sp.hit_ptr + sy.hit_off + static_cast<int64_t>(b) * (sy.act_n + 1) + i;
      for (int k = 4 * hq[0]; k < 4 * hq[1]; k++) {
        const unsigned h = reinterpret_cast<const uint16_t *>(sp.hits)[k];
        if (h / kSumBlock == 0u) continue;
        const Num<L> y = monomial_value<L>(sp, t0 + b * kSumBlock + static_cast<int>(h & (kSumBlock - 1)), tab, exps, lg, q);
        const int e = value_top<L>(y);
        if (e > E) {
          sar_words<W>(zr, min(e - E, 32 * W));
          sar_words<W>(zi, min(e - E, 32 * W));
          E = e;
        }
        uint32_t z[W];
        to_window<L>(y.re, y.e, E, hb, z);
        for (unsigned a = h / kSumBlock; a > 0; a--) add_words<W>(zr, z);
        to_window<L>(y.im, y.e, E, hb, z);
        for (unsigned a = h / kSumBlock; a > 0; a--) add_words<W>(zi, z);
      }
    }
    const int v = static_cast<int>(sp.act[sy.act_off + i] & 0xffffu);
    finish_entry<L>(zr, zi, E - (32 * W - 1 - hb), load_factor<L>(inv4, inve, v, lg, q),
                    Jp + static_cast<size_t>(v) * P * 2 * kComp<L>);
  }
}

// kBatch: a batch handle (systems and items from tables in global memory);
// else one system, whose description comes with the parameters.
// kOne: every polynomial's monomials fit in one chunk; the sums then stay in
// registers from the first term to the output.
//
// Three blocks (24 warps) per SM, 80 registers: with two blocks double-double
// at n = 32 took 15 % longer.  Quad-double with several chunks spills at 80
// registers and keeps two blocks (n = 64: 3.65 ms, with three 3.83); with one
// chunk (n = 32: 533 -> 490 us) and in batches three are faster all the same.
template <int L, bool kTabShared, bool kBatch, bool kOne>
__global__ void __launch_bounds__(kSumThreadsMax, L == 8 && !kOne && !kBatch ? 2 : 3) sum_kernel(const SumParams sp) {
  constexpr int B = Fmt<L>::B, W = Fmt<L>::W, KC = kComp<L>;
  constexpr int kw = Fmt<L>::kKeep / 32, kb = Fmt<L>::kKeep % 32;
  extern __shared__ __align__(16) unsigned char smem[];
  __shared__ int32_t ebuf[2][kSumPointsMax];
  __shared__ unsigned next_item;
  const int tid = threadIdx.x, NT = blockDim.x, lane = tid & 31;
  int64_t held = -1;  // the tile whose table is in shared memory
  int eb = 0;         // ebuf of the current chunk: the largest exponent per point
  if (tid < kSumPointsMax) ebuf[0][tid] = fx::kZeroExp;
  let_next_start();
  wait_for_previous();
  for (unsigned item = blockIdx.x; item < static_cast<unsigned>(sp.n_items);) {
    int gp0, gp1, tile, s = 0;
    if constexpr (kBatch) {
      const int4 it = sp.items[item];
      gp0 = it.x, gp1 = it.x + it.y, tile = it.z, s = it.w;
    } else {
      tile = item / sp.groups;
      gp0 = (item - tile * sp.groups) * sp.group_polys;
      gp1 = min(gp0 + sp.group_polys, sp.n_polys_total);
    }
    const SysDesc &sd = kBatch ? sp.sys[s] : sp.sys0;
    const SumSys &ss = kBatch ? sp.sum_sys[s] : sp.sum_sys0;
    const int P = kBatch ? sd.P : sp.single_P;
    const int lg = sp.lg;
    const int TP = 1 << lg, q = tid & (TP - 1), sub = tid >> lg, subs = NT >> lg;
    const int n = sd.n, levels = sd.emax;
    const int qg = (tile << lg) + q;
    const bool valid = qg < P;
    const bool left = sp.flags[ss.flag_off + min(qg, P - 1)] != 0;  // to the general kernels
    const unsigned char *blob = sp.table + ss.tab_off + static_cast<size_t>(tile) * sum_blob_bytes(L, n, levels, lg);
    const size_t tab_bytes = sum_tab_bytes(L, n, levels, lg);
    const size_t exp_off = static_cast<size_t>(levels) * n * kParts<L> * 16 << lg;
    // shared memory: values first (their place does not depend on the system),
    // sums, their leading bits, table
    const int vrows = 2 * NT * sp.values;
    int4 *vq = reinterpret_cast<int4 *>(smem);
    int32_t *vr = reinterpret_cast<int32_t *>(vq + Win<L>::Q * vrows);
    const int arows = sum_rows(ss.act_max) << lg;
    unsigned char *at = smem + static_cast<size_t>(vrows) * W * 4;
    int4 *aq = reinterpret_cast<int4 *>(at);
    int32_t *ar = reinterpret_cast<int32_t *>(aq + Win<L>::Q * arows);
    if (!kOne) at += static_cast<size_t>(arows) * W * 4;
    int32_t *am = reinterpret_cast<int32_t *>(at);
    unsigned char *stab = at + static_cast<size_t>(arows) * 4;
    const int64_t tile_id = (static_cast<int64_t>(s) << 32) | tile;
    if (kTabShared && held != tile_id) {
      const int4 *src = reinterpret_cast<const int4 *>(blob);
      int4 *dst = reinterpret_cast<int4 *>(stab);
      const int words = static_cast<int>(tab_bytes / 16);
      // (a plain load: sum_powers may still have been writing the table when
      // this kernel started, which non-coherent loads do not allow)
      for (int i = tid; i < words; i += NT) dst[i] = src[i];
      held = tile_id;
    }
    const int4 *tab = reinterpret_cast<const int4 *>(kTabShared ? stab : blob);
    const int32_t *exps = reinterpret_cast<const int32_t *>((kTabShared ? stab : blob) + exp_off);
    const unsigned char *ib = blob + tab_bytes;
    const int4 *inv4 = reinterpret_cast<const int4 *>(ib);
    const int32_t *inve = reinterpret_cast<const int32_t *>(ib + (static_cast<size_t>(n) * kParts<L> * 16 << lg));
    const int hb = ss.head_bits;
    // a tile whose every point is left to the general kernels is not evaluated
    if (__syncthreads_and(left)) gp0 = gp1;
    for (int gp = gp0; gp < gp1; gp++) {
      const int t0 = __ldg(sp.poly_ptr + gp), t1 = __ldg(sp.poly_ptr + gp + 1);
      const int pl = gp - sd.poly0;
      const SumPoly sy = sp.polys[gp];
      // tasks of phase B: (active variable, component), then from a multiple
      // of eight the parts of f
      const int tasks = 2 * sy.act_n, fb = (tasks + 7) & ~7, all = fb + 2 * kSumParts;
      double *Jp = sp.out_J + (static_cast<size_t>(sd.J_off) + static_cast<size_t>(pl) * n * P + qg) * 2 * KC;
      double *fp = sp.out_f + (static_cast<size_t>(sd.f_off) + static_cast<size_t>(pl) * P + qg) * 2 * KC;
      // entries of variables that do not occur in the polynomial
      if (sy.act_n + sy.const_n < n && valid) {
        for (int v = sub; v < n; v += subs) {
          if (__ldg(sp.act_bits + sy.bits_off + (v >> 5)) >> (v & 31) & 1u) continue;
          double *o = Jp + static_cast<size_t>(v) * P * 2 * KC;
          store_zero<L>(o);
          store_zero<L>(o + KC);
        }
      }
      // entries that are one coefficient
      for (int i = sub; i < sy.const_n && valid; i += subs) {
        const double *c = sp.const_val + static_cast<size_t>(sy.const_off + i) * 2 * KC;
        double *o = Jp + static_cast<size_t>(sp.const_var[sy.const_off + i]) * P * 2 * KC;
#pragma unroll
        for (int k = 0; k < 2 * KC; k++) o[k] = c[k];
      }
      if (t0 == t1) {  // no monomials
        if (valid && sub < 2) store_zero<L>(fp + sub * KC);
        continue;
      }
      const int chunk = subs * sp.values;
      bool again = false;
      int32_t e0 = 0;  // exponent of the window's bit 0
      // The sum into f (its parts are 2 TP lanes apart, in one warp).
      auto finish_f = [&](int u, uint32_t (&a)[W]) {
        const unsigned mask = lanes_of_parts(lane, lg);
#pragma unroll
        for (int d = 2; d < 2 * kSumParts; d <<= 1) {
          uint32_t z[W];
#pragma unroll
          for (int i = 0; i < W; i++) z[i] = __shfl_xor_sync(mask, a[i], d << lg);
          add_words<W>(a, z);
        }
        if (valid && u - fb < 2) store_sum<L>(fp + (u & 1) * KC, a, e0);
      };
      // An entry of J: the sum times 1 / x_v, where the window kept enough of
      // its terms (`seen`: the or of their bits from kKeep + sp.slack up with
      // one chunk, which leaves the window as it is; else their leading bit).
      // (The slack of every entry by itself, in a register through the loop
      // below, cost n = 32 in double-double 2 % with one chunk.)  The other
      // component's sum is in lane ^ TP; each lane forms its own component of
      // the product.
      auto finish_J = [&](int u, uint32_t (&a)[W], int32_t seen) {
        const int c = u & 1;
        const unsigned pair = (1u << lane) | (1u << (lane ^ TP));
        const uint32_t entry = __ldg(sp.act + sy.act_off + (u >> 1));
        const int v = static_cast<int>(entry & 0xffffu);
        const Num<L> inv = load_factor<L>(inv4, inve, v, lg, q);
        const int32_t other_seen = __shfl_xor_sync(pair, seen, TP);
        const bool kept = kOne ? (seen | other_seen) != 0 : max(seen, other_seen) >= Fmt<L>::kKeep + static_cast<int>(entry >> 16);
        am[(u << lg) + q] = kept;
        again = again || (!kept && valid);
        int lead = lead_words<W>(a);
        lead = max(lead, __shfl_xor_sync(pair, lead, TP));
        int32_t own[L], other[L], r[L];
        int32_t ey;
        top_digits<L>(a, lead, e0, own, ey);
#pragma unroll
        for (int i = 0; i < L; i++) other[i] = __shfl_xor_sync(pair, own[i], TP);
        const int32_t flip = c ? 0 : -1;  // real lanes subtract the product of the imaginary parts
        long long col[L];
#pragma unroll
        for (int k = 0; k < L; k++) {
          col[k] = 0;
#pragma unroll
          for (int i = k; i < L; i++) {
            col[k] += static_cast<long long>(inv.re[i]) * own[k + L - 1 - i];
            col[k] += static_cast<long long>((inv.im[i] ^ flip) - flip) * other[k + L - 1 - i];
          }
        }
        fx::fold<L>(col, r);
        if (valid && kept)
          store_product<L>(Jp + static_cast<size_t>(v) * P * 2 * KC + c * KC, r, ey + inv.e + B * L - 1);
      };
      int Eprev = 0;
      if constexpr (!kOne) {  // sums to zero
        for (int u = sub; u < all; u += subs) {
          uint32_t z[W];
#pragma unroll
          for (int i = 0; i < W; i++) z[i] = 0u;
          const int row = (u << lg) + q;
          store_window<L>(aq, ar, arows, row, z);
          am[row] = -1;
        }
      }
      for (int tb = t0; kOne ? tb == t0 : tb < t1; tb += chunk) {
        const bool last = kOne || tb + chunk >= t1;
        // A: the values of monomials tb + sub, tb + sub + subs at point q, their
        // digits to the places of their window integers
        int em = fx::kZeroExp;
        for (int x = 0; x < sp.values; x++) {
          const int tl = x * subs + sub;
          if (tb + tl >= t1) break;
          const Num<L> y = monomial_value<L>(sp, tb + tl, tab, exps, lg, q);
          em = max(em, value_top<L>(y));
          uint32_t z[W];
#pragma unroll
          for (int i = 0; i < W; i++) z[i] = i < L ? static_cast<uint32_t>(y.re[i]) : static_cast<uint32_t>(y.e);
          store_window<L>(vq, vr, vrows, ((2 * tl) << lg) + q, z);
#pragma unroll
          for (int i = 0; i < L; i++) z[i] = static_cast<uint32_t>(y.im[i]);
          store_window<L>(vq, vr, vrows, ((2 * tl + 1) << lg) + q, z);
        }
        for (int d = TP; d < 32; d <<= 1) em = max(em, __shfl_xor_sync(0xffffffffu, em, d));
        if (lane < TP) atomicMax(&ebuf[eb][q], em);
        __syncthreads();
        const int E = ebuf[eb][q];
        const int grown = kOne || tb == t0 ? 0 : E - Eprev;
        for (int x = 0; x < sp.values; x++) {
          const int tl = x * subs + sub;
          if (tb + tl >= t1) break;
#pragma unroll
          for (int c = 0; c < 2; c++) {
            uint32_t z[W];
            int32_t d[L];
            load_window<L>(vq, vr, vrows, ((2 * tl + c) << lg) + q, z);
#pragma unroll
            for (int i = 0; i < L; i++) d[i] = static_cast<int32_t>(z[i]);
            to_window<L>(d, static_cast<int32_t>(z[L]), E, hb, z);
            store_window<L>(vq, vr, vrows, ((2 * tl + c) << lg) + q, z);
          }
        }
        if (tid < TP) ebuf[eb ^ 1][q] = last ? fx::kZeroExp : E;  // of the next chunk
        __syncthreads();
        // B: the sums of active variable u >> 1, component u & 1 at point q, and
        // the parts of f
        const int b0 = kOne ? 0 : (tb - t0) / kSumBlock;
        const int b1 = min((tb - t0 + chunk) / kSumBlock, (t1 - t0 + kSumBlock - 1) / kSumBlock);
        e0 = E - (32 * W - 1 - hb);
        for (int u = sub; u < all; u += subs) {
          if (u >= tasks && u < fb) continue;
          const int row = (u << lg) + q, c = u & 1;
          uint32_t a[W];
          uint32_t m = 0u, low = 0u;  // the or of the terms' words above kw, of their words kw
          if constexpr (kOne) {
#pragma unroll
            for (int i = 0; i < W; i++) a[i] = 0u;
          } else {
            load_window<L>(aq, ar, arows, row, a);
            if (grown > 0) sar_words<W>(a, grown);
          }
          if (u >= fb) {
            constexpr int len = kSumBlock / kSumParts;
            for (int b = b0; b < b1; b++) {
              const int tl = (b - b0) * kSumBlock + ((u - fb) >> 1) * len;
              const int count = min(len, t1 - tb - tl);
#pragma unroll 4
              for (int k = 0; k < count; k++) {
                uint32_t z[W];
                load_window<L>(vq, vr, vrows, ((2 * (tl + k) + c) << lg) + q, z);
                add_words<W>(a, z);
              }
            }
            if constexpr (kOne)
              finish_f(u, a);
            else
              store_window<L>(aq, ar, arows, row, a);
            continue;
          }
          uint32_t odd[W - 1];
#pragma unroll
          for (int i = 0; i < W - 1; i++) odd[i] = 0u;
          for (int b = b0; b < b1; b++) {
            const int32_t *hq = sp.hit_ptr + sy.hit_off + static_cast<int64_t>(b) * (sy.act_n + 1) + (u >> 1);
            const int h0 = __ldg(hq), h1 = __ldg(hq + 1);
            if (h0 == h1) continue;
            uint32_t mk = 0u;
            const int base = ((2 * (b - b0) * kSumBlock + c) << lg) + q;
            uint2 hw = __ldg(sp.hits + h0);
#pragma unroll 1
            for (int k = h0; k < h1; k++) {  // four list entries, their values read together
              const unsigned h[4] = {hw.x & 0xffffu, hw.x >> 16, hw.y & 0xffffu, hw.y >> 16};
              if (k + 1 < h1) hw = __ldg(sp.hits + k + 1);
              uint32_t z[4][W];
#pragma unroll
              for (int x = 0; x < 4; x++)
                load_window<L>(vq, vr, vrows, base + (static_cast<int>(h[x] & (kSumBlock - 1)) << (lg + 1)), z[x]);
#pragma unroll
              for (int x = 0; x < 4; x++) {
                add_times<W>(a, odd, z[x], h[x] / kSumBlock);
                const uint32_t sg = static_cast<uint32_t>(static_cast<int32_t>(z[x][W - 1]) >> 31);
#pragma unroll
                for (int i = kw + 1; i < W; i++) m |= z[x][i] ^ sg;
                mk |= z[x][kw] ^ sg;
              }
            }
            if constexpr (kOne)
              m |= __funnelshift_rc(mk, 0u, kb + sp.slack);
            else
              low |= mk;
          }
          uint32_t up[W];
          up[0] = 0u;
#pragma unroll
          for (int i = 0; i < W - 1; i++) up[i + 1] = odd[i];
          add_words<W>(a, up);
          if constexpr (kOne) {
            finish_J(u, a, static_cast<int32_t>(m));
          } else {
            store_window<L>(aq, ar, arows, row, a);
            // (exact but for bits above word kw + 1, which count as of that word)
            int32_t top = max(am[row] - grown, -1);
            if (m | low) top = max(top, (m ? 32 * kw + 63 : 32 * kw + 31) - __clz(static_cast<int>(m ? m : low)));
            am[row] = top;
          }
        }
        eb ^= 1;
        Eprev = E;
        if (!last) __syncthreads();
      }
      if constexpr (!kOne) {  // every thread finishes the sums that it stored
        for (int u = sub; u < all; u += subs) {
          if (u >= tasks && u < fb) continue;
          const int row = (u << lg) + q;
          uint32_t a[W];
          load_window<L>(aq, ar, arows, row, a);
          if (u >= fb)
            finish_f(u, a);
          else
            finish_J(u, a, am[row]);
        }
      }
      if (__syncthreads_or(again)) {
        if (valid) own_windows<L>(sp, gp, am, tab, exps, inv4, inve, lg, q, hb, sub, subs, Jp, P);
        __syncthreads();
      }
    }
    // (Items come from a counter: equal shares of them in order, without one,
    // took 8 % longer at n = 128, since the SMs are not equally fast; taking the
    // next item while this one runs took 3 % longer there.)
    if (tid == 0) next_item = atomicAdd(sp.counter, 1u) + gridDim.x;
    __syncthreads();
    item = next_item;
  }
}

// The kernel of a launch.
using SumKernel = void (*)(const SumParams);

template <int L>
SumKernel kernel_of(bool tab_shared, bool batch, bool one) {
  if (one)
    return tab_shared ? (batch ? sum_kernel<L, true, true, true> : sum_kernel<L, true, false, true>)
                      : (batch ? sum_kernel<L, false, true, true> : sum_kernel<L, false, false, true>);
  return tab_shared ? (batch ? sum_kernel<L, true, true, false> : sum_kernel<L, true, false, false>)
                    : (batch ? sum_kernel<L, false, true, false> : sum_kernel<L, false, false, false>);
}

SumKernel kernel_of(int L, bool tab_shared, bool batch, bool one) {
  return L == 3 ? kernel_of<3>(tab_shared, batch, one) : L == 4 ? kernel_of<4>(tab_shared, batch, one)
                                                                : kernel_of<8>(tab_shared, batch, one);
}

}  // namespace

size_t sum_smem_bytes(int L, int n, int act_max, int levels, int lg, int threads, int values, bool one, bool tab_shared) {
  const size_t W = L == 3 ? Fmt<3>::W : L == 4 ? Fmt<4>::W : Fmt<8>::W;
  return static_cast<size_t>(2) * threads * values * W * 4 +
         (static_cast<size_t>(sum_rows(act_max)) << lg) * (one ? 4 : W * 4 + 4) +
         (tab_shared ? sum_tab_bytes(L, n, levels, lg) : 0);
}

int sum_one_slack(int L) {
  return 32 - (L == 3 ? Fmt<3>::kKeep : L == 4 ? Fmt<4>::kKeep : Fmt<8>::kKeep) % 32;
}

int sum_head_bits_min(int L) { return L == 3 ? Fmt<3>::kHeadMin : L == 4 ? Fmt<4>::kHeadMin : Fmt<8>::kHeadMin; }

cudaError_t prepare_sum(int L, bool batch, size_t smem) {
  for (int k = 0; k < 4; k++) {
    const cudaError_t e = cudaFuncSetAttribute(kernel_of(L, k & 1, batch, k >> 1),
                                               cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(smem));
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

cudaError_t sum_occupancy(int L, bool batch, bool one, bool tab_shared, int threads, size_t smem, int *blocks) {
  return cudaOccupancyMaxActiveBlocksPerMultiprocessor(blocks, kernel_of(L, tab_shared, batch, one), threads, smem);
}

cudaError_t launch_sum_powers(int L, const SumParams &p, cudaStream_t s) {
  const int64_t work = 2 * p.power_total;
  if (work <= 0) return cudaSuccess;
  int64_t blocks = (work + 127) / 128;
  if (blocks > kSms * 64) blocks = kSms * 64;
  const unsigned b = static_cast<unsigned>(blocks);
  if (L == 3)
    sum_powers<3><<<b, 128, 0, s>>>(p);
  else if (L == 4)
    sum_powers<4><<<b, 128, 0, s>>>(p);
  else
    sum_powers<8><<<b, 128, 0, s>>>(p);
  return cudaGetLastError();
}

cudaError_t launch_sum(int L, const SumParams &p, bool one, bool tab_shared, int threads, size_t smem, int grid,
                       cudaStream_t s) {
  return launch_next(kernel_of(L, tab_shared, p.single_P < 0, one), dim3(grid), dim3(threads), smem, s, p);
}

cudaError_t convert_coef_sum(int L, const double *coef, const int32_t *order, const int32_t *fac_ptr, const uint32_t *fac,
                             int32_t *out, int64_t M, cudaStream_t s) {
  if (M <= 0) return cudaSuccess;
  int64_t blocks = (M + 127) / 128;
  if (blocks > kSms * 64) blocks = kSms * 64;
  const unsigned b = static_cast<unsigned>(blocks);
  if (L == 3)
    sum_coef_kernel<3><<<b, 128, 0, s>>>(coef, order, fac_ptr, fac, out, M);
  else if (L == 4)
    sum_coef_kernel<4><<<b, 128, 0, s>>>(coef, order, fac_ptr, fac, out, M);
  else
    sum_coef_kernel<8><<<b, 128, 0, s>>>(coef, order, fac_ptr, fac, out, M);
  return cudaGetLastError();
}

}  // namespace pe
