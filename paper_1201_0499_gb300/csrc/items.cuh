// Decoding of a work item of the main kernels (kernels.cu, kernels_wide.cu).
//
// A single-system call has T x N x C items: tile of 16 points, polynomial
// rank r (in decreasing cost order within the tile), and chunk of the
// polynomial's monomials (C = 1 unless the call has too few (polynomial,
// tile) pairs to fill the GPU).  Tile-major order keeps the warps that run at
// the same time on few tiles, so their points and power-table entries are
// read from L2 rather than DRAM (n = 128, k = 32: 5 % less DRAM traffic in
// double-double, 3 % faster with integer-pipe products).  Chunk 0 writes f and J into the outputs; chunk c > 0 into scratch
// copy c-1 of the same layout, which a combine kernel adds afterwards.  A
// batch handle has C items per (polynomial, tile) entry of its item table,
// chunked the same way.
#pragma once

#include <cstdint>

#include "internal.h"

namespace pe {

struct Item {
  int gp, tile, s, P;  // global polynomial, tile (of 16 / groups points), system, points of the system
  int groups;          // monomial groups per warp
  int t0, t1;          // monomial range
  double *f_base;      // output (or scratch) base for f
  double *J_base;      // output (or scratch) base for J
};

// kSome: a launch that evaluates only flagged points (kernels of its own: the
// code for it would take registers from the others).
// Returns false for an item to skip: one without a flagged point in such a
// launch, or an inconsistent one (flags the status word).
template <bool kSome>
__device__ __forceinline__ bool decode_item(const MainParams &kp, unsigned item, int lane, Item &it) {
  int chunk = 0;
  if (kp.single_P >= 0) {
    const unsigned C = static_cast<unsigned>(kp.n_chunks);
    const unsigned rest = item / C;
    chunk = static_cast<int>(item - rest * C);
    it.tile = static_cast<int>(rest) / kp.n_polys_total;  // tile-major: the warps resident at once share tiles
    const int r = static_cast<int>(rest) - it.tile * kp.n_polys_total;
    it.gp = kp.perm[r];
    it.s = 0;
    it.P = kp.single_P;
    it.groups = kp.groups;
  } else {
    const unsigned C = static_cast<unsigned>(kp.n_chunks);
    const unsigned rest = item / C;
    chunk = static_cast<int>(item - rest * C);
    const int2 x = kp.items[rest];
    it.gp = x.x;
    it.groups = 1 << ((x.y >> kTileBits) & 7);
    it.tile = (x.y & ((1 << kTileBits) - 1)) * it.groups;  // in tiles of 16 / groups points
    it.s = (x.x >= 0 && x.x < kp.n_polys_total) ? kp.poly_sys[x.x] : 0;
    it.P = kp.sys[it.s].P;
  }
  if (it.gp < 0 || it.gp >= kp.n_polys_total || it.groups > kPointsPerWarp ||
      it.tile * (kPointsPerWarp / it.groups) >= it.P) {
    if (lane == 0) atomicOr(kp.status, 1);
    return false;
  }
  if constexpr (kSome) {
    // flagged points only; few of them spread over the warp's monomial
    // groups: the most groups whose sub-tile holds them all
    const int tp = kPointsPerWarp / it.groups, q = it.tile * tp + lane;
    const unsigned set = __ballot_sync(0xffffffffu, lane < tp && q < it.P && kp.flags[kp.sys[it.s].fl_off + q] != 0);
    if (set == 0u) return false;
    if (kp.regroup) {
      int first = __ffs(static_cast<int>(set)) - 1, last = 31 - __clz(static_cast<int>(set)), sub = tp;
      while (sub > 1 && first / (sub / 2) == last / (sub / 2)) {
        sub /= 2;
        it.groups *= 2;
      }
      it.tile = (it.tile * tp + first) / sub;
    }
  }
  int t0 = kp.poly_ptr[it.gp], t1 = kp.poly_ptr[it.gp + 1];
  if (kp.n_chunks > 1) {
    const long long m = t1 - t0;
    const int a = t0 + static_cast<int>(m * chunk / kp.n_chunks);
    const int b = t0 + static_cast<int>(m * (chunk + 1) / kp.n_chunks);
    t0 = a;
    t1 = b;
  }
  it.t0 = t0;
  it.t1 = t1;
  it.f_base = chunk == 0 ? kp.out_f : kp.scratch_f + static_cast<size_t>(chunk - 1) * kp.chunk_f_stride;
  it.J_base = chunk == 0 ? kp.out_J : kp.scratch_J + static_cast<size_t>(chunk - 1) * kp.chunk_J_stride;
  return true;
}

}  // namespace pe
