// The Newton step's linear systems in double-double, on the integer pipes.
//
// A double-double elimination step of one entry (a - l u, complex) takes 42
// FP64 instructions, which a GB300 SM issues at 16 cycles per warp: the LU of a
// 32 x 32 system at 1024 points took 1.45 ms, bound by the FP64 pipe.  Here an
// entry is a pair of 128-bit two's complement integers with one exponent
// (El); a product l u is the digit product of digits.cuh (118 bits), aligned
// and subtracted in words.  Errors are relative to the larger of the operands'
// magnitudes at 2^-115, against 2^-104 for the double-double operations.
//
// One block per point, the augmented system [J | -f] in shared memory, rows
// exchanged by index.  Step k: the multipliers, and the pivot row as table-kind
// factors; then the trailing entries, the right-hand side as one more column,
// while the first warp, which takes column k + 1, goes on to the next pivot (as
// lu.cuh: largest modulus by the leading parts, smallest row on ties) and its
// reciprocal.  The other warps write the multipliers out, by position: an
// exchange does not move those of earlier steps.  The reciprocals are kept for
// the back substitution.  Points with entries that are not finite or beyond
// 2^(+-kMaxExp) are solved by the double-double code of lu.cuh, whose
// overflows and NaN they keep; so are systems all of whose entries lie near an
// axis (components more than 2^kElApart apart) unless all are real, whose
// smaller parts come from smaller parts alone and would take the error of the
// larger ones (118 bits for both, 106 each there).
#include <cuda_runtime.h>

#include <cmath>
#include <cstdint>

#include "cplx.cuh"
#include "internal.h"
#include "lu.cuh"
#include "words.cuh"

namespace pe {

namespace {

using fx::Num;

constexpr int kMaxExp = 200;
constexpr int kElApart = 10;
constexpr int kZeroEl = -(1 << 20);  // exponent of an exactly zero entry

struct El {
  uint32_t r[4], i[4];  // |value| < 2^126
  int32_t e;
};

// Arrays of entries in shared memory.
struct Els {
  int4 *re, *im;
  int32_t *e;
  __device__ El load(int k) const {
    const int4 a = re[k], b = im[k];
    return El{{static_cast<uint32_t>(a.x), static_cast<uint32_t>(a.y), static_cast<uint32_t>(a.z), static_cast<uint32_t>(a.w)},
              {static_cast<uint32_t>(b.x), static_cast<uint32_t>(b.y), static_cast<uint32_t>(b.z), static_cast<uint32_t>(b.w)},
              e[k]};
  }
  __device__ void store(int k, const El &x) const {
    re[k] = make_int4(x.r[0], x.r[1], x.r[2], x.r[3]);
    im[k] = make_int4(x.i[0], x.i[1], x.i[2], x.i[3]);
    e[k] = x.e;
  }
  __device__ Num<4> load_num(int k) const {
    const int4 a = re[k], b = im[k];
    return Num<4>{{a.x, a.y, a.z, a.w}, {b.x, b.y, b.z, b.w}, e[k]};
  }
  __device__ void store_num(int k, const Num<4> &x) const {
    re[k] = make_int4(x.re[0], x.re[1], x.re[2], x.re[3]);
    im[k] = make_int4(x.im[0], x.im[1], x.im[2], x.im[3]);
    e[k] = x.e;
  }
};

// A normalised double-double component as a two's complement integer with its
// leading bit at 124.
__device__ __forceinline__ void component_words(double h, double l, uint32_t (&w)[4], int32_t &e) {
  const wide::Comp c = wide::comp_from_dd(h, l);
  const uint32_t neg = c.s ? 0xffffffffu : 0u, one = neg & 1u;
  w[0] = c.m.w0 ^ neg, w[1] = c.m.w1 ^ neg, w[2] = c.m.w2 ^ neg, w[3] = c.m.w3 ^ neg;
  asm("add.cc.u32 %0, %0, %4;\n\taddc.cc.u32 %1, %1, 0;\n\taddc.cc.u32 %2, %2, 0;\n\taddc.u32 %3, %3, 0;"
      : "+r"(w[0]), "+r"(w[1]), "+r"(w[2]), "+r"(w[3])
      : "r"(one));
  e = wide::is_zero(c.m) ? kZeroEl : c.e;
}

// What the entries of a system are: usual, or values that the integer
// elimination is not meant for; some not real; some away from the axes.
struct Kinds {
  bool usual = true, complex = false, off_axis = false;
};

// An entry from the evaluator's (normalised) double-doubles.  No FP64
// arithmetic: 1000 entries of 5 blocks would queue for its pipe.
__device__ __forceinline__ El el_from(const CDD &v, Kinds &kinds) {
  auto exponent = [](double x) { return static_cast<int>(static_cast<unsigned long long>(__double_as_longlong(x)) >> 52) & 0x7ff; };
  auto zero = [](double x) { return (__double_as_longlong(x) << 1) == 0; };
  const int xr = exponent(v.re.h), xi = exponent(v.im.h), top = max(xr, xi);
  const bool zr = zero(v.re.h), zi = zero(v.im.h);
  if (!(zr && zi) && (top > 1023 + kMaxExp || top < 1023 - kMaxExp)) kinds.usual = false;
  kinds.complex = kinds.complex || !zi;
  kinds.off_axis = kinds.off_axis || (!zr && !zi && xr - xi <= kElApart && xi - xr <= kElApart);
  El x;
  if (!kinds.usual) {
    for (int k = 0; k < 4; k++) x.r[k] = x.i[k] = 0u;
    x.e = kZeroEl;
    return x;
  }
  int32_t er, ei;
  component_words(v.re.h, v.re.l, x.r, er);
  component_words(v.im.h, v.im.l, x.i, ei);
  x.e = max(er, ei);
  sar_words<4>(x.r, x.e - er);
  sar_words<4>(x.i, x.e - ei);
  return x;
}

__device__ __forceinline__ CDD to_cdd(const El &x) {
  return CDD{words_to_dd(x.r[0], x.r[1], x.r[2], x.r[3], x.e), words_to_dd(x.i[0], x.i[1], x.i[2], x.i[3], x.e)};
}

// An entry as a y-kind number (digits.cuh), its larger component's leading bit
// three below the top of the digits; zero stays zero.
__device__ __forceinline__ Num<4> el_digits(El x) {
  const int lead = max(lead_words<4>(x.r), lead_words<4>(x.i));
  Num<4> y;
  if (lead < 0 && !(x.r[3] | x.i[3])) {
#pragma unroll
    for (int k = 0; k < 4; k++) y.re[k] = y.im[k] = 0;
    y.e = kZeroEl;
    return y;
  }
  const int sh = min(125 - lead, 127);
  shl_words<4>(x.r, sh);
  shl_words<4>(x.i, sh);
  constexpr int o0 = 128 + 1 - 120;
#pragma unroll
  for (int k = 0; k < 4; k++) {
    const int w = (o0 + 30 * k) >> 5, b = (o0 + 30 * k) & 31;
    if (k == 3) {
      y.re[k] = static_cast<int32_t>(x.r[3]) >> 3;
      y.im[k] = static_cast<int32_t>(x.i[3]) >> 3;
    } else {
      y.re[k] = static_cast<int32_t>(__funnelshift_r(x.r[w], x.r[w + 1], b)) & 0x3fffffff;
      y.im[k] = static_cast<int32_t>(__funnelshift_r(x.i[w], x.i[w + 1], b)) & 0x3fffffff;
    }
  }
  y.e = x.e - sh + o0;
  return y;
}

__device__ __forceinline__ bool is_zero(const Num<4> &y) { return fx::top_magnitude<4>(y) == 0u && y.e <= kZeroEl; }

// The same as a factor (X kind) of modulus near 2^(B L - 1).
__device__ __forceinline__ Num<4> el_factor(const El &x) {
  Num<4> y = el_digits(x);
  if (!is_zero(y)) y = fx::as_factor<4>(y);
  return y;
}

__device__ __forceinline__ El el_of(const Num<4> &y) {
  El x;
  pack_digits<4, 4>(y.re, x.r);
  pack_digits<4, 4>(y.im, x.i);
  x.e = y.e;
  return x;
}

// A factor's balanced digits back in words.
__device__ __forceinline__ El el_of_factor(Num<4> x) {
  int32_t t = 0, m = 0;
#pragma unroll
  for (int k = 0; k < 3; k++) {
    t += x.re[k];
    x.re[k] = t & 0x3fffffff;
    t >>= 30;
    m += x.im[k];
    x.im[k] = m & 0x3fffffff;
    m >>= 30;
  }
  x.re[3] += t;
  x.im[3] += m;
  return el_of(x);
}

__device__ __forceinline__ void sub_words(uint32_t (&a)[4], const uint32_t (&b)[4]) {
  asm("sub.cc.u32 %0, %0, %4;\n\tsubc.cc.u32 %1, %1, %5;\n\tsubc.cc.u32 %2, %2, %6;\n\tsubc.u32 %3, %3, %7;"
      : "+r"(a[0]), "+r"(a[1]), "+r"(a[2]), "+r"(a[3])
      : "r"(b[0]), "r"(b[1]), "r"(b[2]), "r"(b[3]));
}

// a - p
__device__ __forceinline__ El el_sub(El a, El p) {
  const int d = p.e - a.e;
  if (d > 0) {
    sar_words<4>(a.r, d);
    sar_words<4>(a.i, d);
    a.e = p.e;
  } else {
    sar_words<4>(p.r, -d);
    sar_words<4>(p.i, -d);
  }
  sub_words(a.r, p.r);
  sub_words(a.i, p.i);
  const int32_t tr = static_cast<int32_t>(a.r[3]), ti = static_cast<int32_t>(a.i[3]);
  if ((tr >> 30) != (tr >> 31) || (ti >> 30) != (ti >> 31)) {  // 2^126 reached
    sar_words<4>(a.r, 1);
    sar_words<4>(a.i, 1);
    a.e += 1;
  }
  return a;
}

// The squared modulus from the components' 62 leading bits, as an integer
// that orders like it: exponent, then 48 bits of the mantissa; 0 for zero.
// (By integers: every pivot search would queue for the FP64 pipe.)
__device__ __forceinline__ unsigned long long order_by_modulus(El x) {
  const int lead = max(lead_words<4>(x.r), lead_words<4>(x.i));
  if (lead < 0 && !(x.r[3] | x.i[3])) return 0ULL;
  const int sh = min(125 - lead, 127);
  shl_words<4>(x.r, sh);
  shl_words<4>(x.i, sh);
  const long long r = static_cast<long long>((static_cast<unsigned long long>(x.r[3]) << 32) | x.r[2]);
  const long long i = static_cast<long long>((static_cast<unsigned long long>(x.i[3]) << 32) | x.i[2]);
  const unsigned long long ur = static_cast<unsigned long long>(r < 0 ? -r : r), ui = static_cast<unsigned long long>(i < 0 ? -i : i);
  // the larger component leads at bit 61: the sum of the squares' upper halves is in [2^58, 2^60]
  const unsigned long long m = __umul64hi(ur, ur) + __umul64hi(ui, ui);
  const int z = __clzll(static_cast<long long>(m));
  const int e = 2 * (x.e - sh) + 63 - z + (1 << 14);  // > 0 for every exponent an entry can have
  return (static_cast<unsigned long long>(e) << 48) | ((m << (z + 1)) >> 16);
}

// Shared memory of a block: the entries [n][n + 1], the pivot row's factors
// [n + 1], the multipliers [n], the reciprocals [n], the row order twice.
__host__ __device__ constexpr size_t int_lu_entries(int n) {
  return static_cast<size_t>(n) * (n + 1) + (n + 1) + n + n;
}
__host__ __device__ constexpr size_t int_lu_bytes(int n) { return int_lu_entries(n) * 36 + static_cast<size_t>(n) * 8 + 64; }

__global__ void __launch_bounds__(256, 2) newton_int(const NewtonParams p) {
  extern __shared__ __align__(16) unsigned char smem[];
  __shared__ int pivot, is_singular;
  __shared__ double red[2][8];
  const int64_t q = blockIdx.x;
  const int n = p.n, cols = n + 1, tid = threadIdx.x, T = blockDim.x, lane = tid & 31, warp = tid >> 5;
  const size_t P = static_cast<size_t>(p.P);
  const size_t entries = int_lu_entries(n);
  int4 *quads = reinterpret_cast<int4 *>(smem);
  int32_t *exps = reinterpret_cast<int32_t *>(quads + 2 * entries);
  const Els A{quads, quads + entries, exps};
  const int off_u = n * cols, off_l = off_u + cols, off_v = off_l + n;
  int32_t *row = exps + entries;
  const PointView<CDD> gv{p.J, p.f, n, P, q};
  auto Xel = [&](int i) { return p.x + (static_cast<size_t>(i) * P + q) * 4; };
  auto block_max = [&](double v, double *slot) {  // every thread gets the maximum
    for (int d = 16; d > 0; d >>= 1) v = nan_max(v, __shfl_xor_sync(0xffffffffu, v, d));
    if (lane == 0) slot[warp] = v;
    __syncthreads();
    v = slot[0];
    for (int w = 1; w < T / 32; w++) v = nan_max(v, slot[w]);
    return v;
  };

  Kinds kinds;
  double fnorm = 0.0;
  for (int i = tid; i < n; i += T) {
    const CDD v = CDD::load(gv.bel(i));
    fnorm = nan_max(fnorm, v.abs_hi());
    A.store(i * cols + n, el_from(v.neg(), kinds));
  }
  for (int k0 = tid; k0 < n * n; k0 += 4 * T) {  // four loads in flight
    CDD v[4];
#pragma unroll
    for (int x = 0; x < 4; x++)
      if (k0 + x * T < n * n) v[x] = CDD::load(gv.Jel((k0 + x * T) / n, (k0 + x * T) % n));
#pragma unroll
    for (int x = 0; x < 4; x++)
      if (k0 + x * T < n * n) A.store((k0 + x * T) / n * cols + (k0 + x * T) % n, el_from(v[x], kinds));
  }
  for (int i = tid; i < n; i += T) row[i] = i;
  if (tid == 0) is_singular = 0;
  fnorm = block_max(fnorm, red[0]);
  bool singular = false;
  const bool usual = __syncthreads_and(kinds.usual);
  const bool near_axis = !__syncthreads_or(kinds.off_axis) && __syncthreads_or(kinds.complex);
  if (!usual || near_axis) {
    // the double-double elimination in place, by the first warp
    if (warp == 0) {
      for (int i = lane; i < n; i += 32) CDD::load(gv.bel(i)).neg().store(gv.bel(i));
      __syncwarp();
      const bool s = lu_solve<CDD>(gv, Lanes<32>::of_thread());
      if (lane == 0) is_singular = s;
    }
    __syncthreads();
    singular = is_singular != 0;
  } else {
    // Warp 0: the pivot of column k (of modulus-largest entry, the smallest row
    // on ties) among rows k .. n-1, and its reciprocal.  Reads the row order `r`.
    auto find_pivot = [&](int k, const int32_t *r) {
      unsigned long long best = 0;
      int piv = n;
      for (int i = k + lane; i < n; i += 32) {
        const unsigned long long m = order_by_modulus(A.load(r[i] * cols + k));
        if (m > best) {
          best = m;
          piv = i;
        }
      }
      for (int d = 16; d > 0; d >>= 1) {
        const unsigned long long ob = __shfl_xor_sync(0xffffffffu, best, d);
        const int op = __shfl_xor_sync(0xffffffffu, piv, d);
        if (ob > best || (ob == best && op < piv)) {
          best = ob;
          piv = op;
        }
      }
      if (lane == 0) {
        if (best != 0) {
          pivot = piv;
          A.store_num(off_v + k, fx::as_factor<4>(fx::reciprocal<4>(el_factor(A.load(r[piv] * cols + k)))));
        } else {
          is_singular = 1;
        }
      }
    };
    int32_t *was = row, *now = row + n;  // row order before and after the exchange of this step
    int done = n;                        // columns eliminated
    if (warp == 0) find_pivot(0, was);
    __syncthreads();
    for (int k = 0; k < n; k++) {
      singular = is_singular != 0;  // uniform
      if (singular) {
        now = was;
        done = k;
        break;
      }
      const int piv = pivot, pr = was[piv] * cols;
      const Num<4> inv = A.load_num(off_v + k);
      // the exchange, the multipliers (first warps), the pivot row's factors (the others)
      for (int i = tid; i < n; i += T) now[i] = i == k ? was[piv] : i == piv ? was[k] : was[i];
      const int split = ((n - k - 1 + 31) & ~31) < T ? (n - k - 1 + 31) & ~31 : 0;
      for (int i = k + 1 + tid; i < n; i += T) {
        const int at = (i == piv ? was[k] : was[i]) * cols + k;
        Num<4> l = el_digits(A.load(at));
        if (!is_zero(l)) fx::mul<4>(l, inv);
        A.store_num(off_l + i, l);
      }
      if (tid >= split)
        for (int j = k + 1 + tid - split; j < cols; j += T - split) A.store_num(off_u + j, el_factor(A.load(pr + j)));
      __syncthreads();
      // trailing entries and right-hand side; the first warp takes the next
      // column, its pivot and its reciprocal, whose chains the others hide
      const int w = n - k - 1;
      auto update = [&](int i, int j) {
        Num<4> l = A.load_num(off_l + i);
        fx::mul<4>(l, A.load_num(off_u + j));
        const int at = now[i] * cols + j;
        A.store(at, el_sub(A.load(at), el_of(l)));
      };
      if (w > 0) {
        if (warp == 0) {
          for (int i = k + 1 + lane; i < n; i += 32) update(i, k + 1);
          __syncwarp();
          find_pivot(k + 1, now);
        } else {
          const int wc = w, T1 = T - 32, t1 = tid - 32;  // columns k + 2 .. n
          int i = k + 1 + t1 / wc, j = k + 2 + t1 % wc;
          const int di = T1 / wc, dj = T1 % wc;
          for (int e = t1; e < w * wc; e += T1) {
            update(i, j);
            i += di;
            j += dj;
            if (j >= cols) {
              j -= wc;
              i++;
            }
          }
          // the multipliers stay where step k put them (later exchanges move
          // the columns after k only), so they go out by position, now
          for (int r = k + 1 + t1; r < n; r += T1) to_cdd(el_of(A.load_num(off_l + r))).store(gv.Jel(r, k));
        }
      }
      __syncthreads();
      int32_t *swap = was;
      was = now;
      now = swap;
    }
    row = was;
    // back substitution by columns: every thread forms x_i, then the threads
    // over the rows above take it out of them.  The entries above the diagonal
    // are turned into factors beforehand (and back when they are written out).
    for (int k = tid; k < n * n && !singular; k += T) {
      const int i = k / n, j = k - i * n;
      if (j > i) A.store_num(row[i] * cols + j, el_factor(A.load(row[i] * cols + j)));
    }
    __syncthreads();
    for (int i = n - 1; i >= 0 && !singular; i--) {
      Num<4> x = el_digits(A.load(row[i] * cols + n));
      if (!is_zero(x)) fx::mul<4>(x, A.load_num(off_v + i));
      __syncthreads();
      if (tid == 0) A.store(row[i] * cols + n, el_of(x));
      for (int r = tid; r < i; r += T) {
        Num<4> y = x;
        fx::mul<4>(y, A.load_num(row[r] * cols + i));
        const int at = row[r] * cols + n;
        A.store(at, el_sub(A.load(at), el_of(y)));
      }
      __syncthreads();
    }
    // factors and solution out (a singular point keeps what was eliminated)
    for (int k = tid; k < n * cols; k += T) {
      const int i = k / cols, j = k - i * cols;
      if (j < min(i, done)) continue;  // a multiplier, written in step j
      const bool digits = !singular && j > i && j < n;
      const CDD v = to_cdd(digits ? el_of_factor(A.load_num(row[i] * cols + j)) : A.load(row[i] * cols + j));
      v.store(j < n ? gv.Jel(i, j) : gv.bel(i));
    }
    __syncthreads();
  }
  double dxnorm = 0.0;
  for (int i = tid; i < n; i += T) {
    if (singular) {
      CDD::zero().store(gv.bel(i));
      continue;
    }
    const CDD dx = CDD::load(gv.bel(i));
    dxnorm = nan_max(dxnorm, dx.abs_hi());
    CDD::add2(CDD::load(Xel(i)), dx).finish().store(Xel(i));
  }
  dxnorm = block_max(dxnorm, red[1]);
  if (tid == 0 && p.norms) {
    p.norms[q * 2] = fnorm;
    p.norms[q * 2 + 1] = singular ? nan("") : dxnorm;
  }
}

}  // namespace

// The integer elimination takes a block per point; its shared memory bounds n.
constexpr size_t kIntLuBytesMax = 220 * 1024;
bool newton_int_fits(int n) { return n >= kIntLuMin && int_lu_bytes(n) <= kIntLuBytesMax; }

cudaError_t launch_newton_int(const NewtonParams &p, cudaStream_t s) {
  const size_t bytes = int_lu_bytes(p.n);
  if (bytes > 48 * 1024) {
    // the same limit on every call: it belongs to the kernel, not to this call,
    // and another thread may be about to launch a larger system
    const cudaError_t e =
        cudaFuncSetAttribute(newton_int, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(kIntLuBytesMax));
    if (e != cudaSuccess) return e;
  }
  // threads as the trailing updates need (the first warp also finds the pivots and their reciprocals)
  const int threads = p.n <= 16 ? 64 : p.n <= 40 ? 128 : 256;
  newton_int<<<static_cast<unsigned>(p.P), threads, bytes, s>>>(p);
  return cudaGetLastError();
}

}  // namespace pe
