// Tile and cell indexing shared by the tiled reductions (one CTA per tile).
#pragma once

#include "smcx_bcc_tile.cuh"

namespace smcx {

namespace bccfast {

// Origin t0 and extent ts of tile t (tiles numbered x fastest).
__device__ __forceinline__ void tile_of_index(const LatDesc& D, int t, int t0[3], int ts[3]) {
  const int ntx = D.nt[0], nty = D.nt[1];
  const int ti[3] = {t % ntx, (t / ntx) % nty, t / (ntx * nty)};
#pragma unroll
  for (int a = 0; a < 3; a++) {
    const int base = D.n[a] / D.nt[a], rem = D.n[a] % D.nt[a];
    ts[a] = base + (ti[a] < rem ? 1 : 0);
    t0[a] = ti[a] * base + min(ti[a], rem);
  }
}

// Exact division of 0 <= c < 2^16 by 2 <= d < 2^10 with a 32-bit multiply-high
// by m = ceil(2^32 / d): c m / 2^32 = c / d + c e / 2^32 with 0 <= e < 1, and
// c e / 2^32 < 2^-16 < 1 / d, so the floor is c / d (d = 1 passes c through).
struct FastDiv {
  uint32_t d, m;
  __device__ __forceinline__ explicit FastDiv(uint32_t dd)
      : d(dd), m(dd > 1 ? (uint32_t)((0xFFFFFFFFull) / dd + 1) : 0u) {}
  __device__ __forceinline__ uint32_t div(uint32_t c) const { return d > 1 ? __umulhi(c, m) : c; }
};

// Cell c of a tile of ts[0] x ts[1] x ts[2] cells (x fastest).
struct CellIndex {
  FastDiv dx, dxy;
  __device__ __forceinline__ CellIndex(const int ts[3]) : dx((uint32_t)ts[0]), dxy((uint32_t)(ts[0] * ts[1])) {}
  __device__ __forceinline__ void at(int c, int& xr, int& yr, int& zr) const {
    const uint32_t z = dxy.div((uint32_t)c);
    const uint32_t r = (uint32_t)c - z * dxy.d;
    const uint32_t y = dx.div(r);
    zr = (int)z;
    yr = (int)y;
    xr = (int)(r - y * dx.d);
  }
};

// Tile counts nt of a reduction that stages each tile with its 2-cell halo, and the
// number of tiles.  Lattices of at least two tiles per SM take the largest tiles, of
// `most` or 12 cells.  Smaller ones take the largest edge that gives 100 tiles: below
// that SMs idle, above it the halo costs more than the SMs gain.  Wall time of FCC pair
// counts against tiles for two per SM throughout: 44^3 cells, 4 species, 2 shells 42 -> 30
// us, 36^3, 8 species, 3 shells 58 -> 36; local energies of 36^3 BCC cells, 4 shells 16
// -> 8 us.  (Gathers from global memory take 32, 47 and 18.)
inline long long reduction_tiles(const int n[3], int most, int nt[3]) {
  auto tiles = [&](int edge) {
    long long g = 1;
    for (int a = 0; a < 3; a++) g *= nt[a] = (n[a] + edge - 1) / edge;
    return g;
  };
  long long g = 0;
  for (int edge : {most, 12})
    if ((g = tiles(edge)) >= 2 * kSMs) return g;
  for (int edge : {12, 10, 8, 7, 6})
    if ((g = tiles(edge)) >= 100) return g;
  return tiles(4);
}

// acc += x * one (one: 0 or 1), without the branch that the compiler makes of a test of
// the lane's species: where lanes differ, it runs every branch in turn.
__device__ __forceinline__ void add_if(uint32_t& acc, uint32_t x, uint32_t one) {
  asm("mad.lo.u32 %0, %1, %2, %0;" : "+r"(acc) : "r"(x), "r"(one));
}

}  // namespace bccfast

}  // namespace smcx
