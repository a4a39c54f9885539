// Two's complement integers of W 32-bit words (word 0 least significant): the
// shifts and conversions of the kernels that sum or eliminate with them
// (kernels_sum.cu, newton_int.cu).
#pragma once

#include <cstdint>

#include "digits.cuh"

namespace pe {

// Arithmetic right shift of W words by s >= 0.
template <int W>
__device__ __forceinline__ void sar_words(uint32_t (&z)[W], int s) {
  s = min(s, 32 * W - 1);
  const uint32_t fill = static_cast<uint32_t>(static_cast<int32_t>(z[W - 1]) >> 31);
  if (s >= 32) {
#pragma unroll
    for (int st = 8; st >= 1; st >>= 1) {
      if (st >= W) continue;
      const bool on = ((s >> 5) & st) != 0;
#pragma unroll
      for (int i = 0; i < W; i++) z[i] = on ? (i + st < W ? z[i + st] : fill) : z[i];
    }
  }
  const int b = s & 31;
#pragma unroll
  for (int i = 0; i < W - 1; i++) z[i] = __funnelshift_r(z[i], z[i + 1], b);
  z[W - 1] = static_cast<uint32_t>(static_cast<int32_t>(z[W - 1]) >> b);
}

// Left shift of W words by 0 <= s < 32 W.
template <int W>
__device__ __forceinline__ void shl_words(uint32_t (&z)[W], int s) {
#pragma unroll
  for (int st = 8; st >= 1; st >>= 1) {
    if (st >= W) continue;
    const bool on = ((s >> 5) & st) != 0;
#pragma unroll
    for (int i = W - 1; i >= 0; i--) z[i] = on ? (i >= st ? z[i - st] : 0u) : z[i];
  }
  const int b = s & 31;
#pragma unroll
  for (int i = W - 1; i > 0; i--) z[i] = __funnelshift_l(z[i - 1], z[i], b);
  z[0] <<= b;
}

// Position of the leading bit of |z| (of |z| - 1 for a negative z); -1 if none.
template <int W>
__device__ __forceinline__ int lead_words(const uint32_t (&z)[W]) {
  const uint32_t fill = static_cast<uint32_t>(static_cast<int32_t>(z[W - 1]) >> 31);
  int p = -1;
#pragma unroll
  for (int i = 0; i < W; i++) {
    const uint32_t x = z[i] ^ fill;
    if (x) p = 32 * i + 31 - __clz(static_cast<int>(x));
  }
  return p;
}

// The two's complement integer of a y-kind component in NW words (the top
// digit may hold B + 1 bits and its sign).
template <int L, int NW>
__device__ __forceinline__ void pack_digits(const int32_t (&d)[L], uint32_t (&w)[NW]) {
  constexpr int B = fx::Fmt<L>::B;
#pragma unroll
  for (int i = 0; i < NW; i++) w[i] = 0u;
#pragma unroll
  for (int i = 0; i < L; i++) {
    const int at = (B * i) >> 5, b = (B * i) & 31;
    w[at] |= static_cast<uint32_t>(d[i]) << b;
    if (at + 1 < NW) {
      const uint32_t high = b == 0 ? static_cast<uint32_t>(i == L - 1 ? d[i] >> 31 : 0)
                                   : static_cast<uint32_t>(i == L - 1 ? d[i] >> (32 - b)
                                                                      : static_cast<int32_t>(static_cast<uint32_t>(d[i]) >> (32 - b)));
      w[at + 1] |= high;
      if (i == L - 1)
        for (int k = at + 2; k < NW; k++) w[k] = static_cast<uint32_t>(d[i] >> 31);
    }
  }
}

template <int L>
constexpr int kPackWords = L == 3 ? 3 : L == 4 ? 4 : 8;

// A 128-bit two's complement integer times 2^e as a normalised double-double.
__device__ __forceinline__ dd words_to_dd(uint32_t w0, uint32_t w1, uint32_t w2, uint32_t w3, int32_t e) {
  const uint32_t neg = static_cast<uint32_t>(static_cast<int32_t>(w3) >> 31);
  wide::Mag m{w0 ^ neg, w1 ^ neg, w2 ^ neg, w3 ^ neg};
  const uint32_t one = neg & 1u;
  asm("add.cc.u32 %0, %0, %4;\n\taddc.cc.u32 %1, %1, 0;\n\taddc.cc.u32 %2, %2, 0;\n\taddc.u32 %3, %3, 0;"
      : "+r"(m.w0), "+r"(m.w1), "+r"(m.w2), "+r"(m.w3)
      : "r"(one));
  if (wide::is_zero(m)) return dd{0.0, 0.0};
  const int z = wide::clz128(m);
  const dd r = wide::to_dd(wide::WV{wide::shl(m, z), neg & wide::kSignBit, e - z});
  return normalize(r);
}

}  // namespace pe
