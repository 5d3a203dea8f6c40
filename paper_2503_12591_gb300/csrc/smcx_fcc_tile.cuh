// Shared-memory box of an FCC tile (tiles of at most 15 cells, 2-cell halo) and
// its staging, used by the FCC tile sweep and the tiled FCC reductions.
//
// FCC sites are the even points (x + y + z even) of the half-unit cubic grid.
// The box stores the site at half-unit box position (x, y, z) in byte (x + y
// PXF + z PPF) / 2; PXF and PPF are odd, so the numerator of every site is even
// and no byte is wasted.  A neighbour along the lattice vector v is then at the
// constant offset (vx + vy PXF + vz PPF) / 2 from any site, whatever its
// sublattice.
#pragma once

#include "smcx_bcc_tile.cuh"

namespace smcx {

namespace fccfast {

using bccfast::LatDesc;
using bccfast::Planes;

constexpr int H = 2;                     // halo cells
constexpr int TMAX = 15;                 // largest tile edge (cells)
constexpr int EXT = 2 * (TMAX + 2 * H);  // box edge in half units (38)
// Odd pitches (>= EXT and >= EXT * PXF) chosen by simulating the banks of a
// warp's 32 slot origins (link cell 3, 5^3 slots): every centre-environment
// load is one wavefront; the partner loads, scattered by the per-lane
// directions, are not.  No odd row pitch from 39 to 47 has such a plane
// pitch within 3000 bytes of the minimum; 49 / 1867 is the smallest box.
constexpr int PXF = 49;
constexpr int PPF = 1867;
static_assert(PXF % 2 == 1 && PPF % 2 == 1 && PXF > EXT - 1 && PPF >= EXT * PXF, "FCC box pitches");
constexpr int BOXB = ((EXT - 1) + (EXT - 1) * PXF + (EXT - 1) * PPF) / 2 + 1;  // bytes used
constexpr int BOX_BYTES = (BOXB + 15) / 16 * 16;

__host__ __device__ constexpr int hoff(int x, int y, int z) { return (x + y * PXF + z * PPF) / 2; }
// FCC basis (0,0,0), (1,1,0), (1,0,1), (0,1,1) in half units: offset of site b in its cell
__host__ __device__ constexpr int boff(int b) {
  return hoff((b == 1 || b == 2) ? 1 : 0, (b == 1 || b == 3) ? 1 : 0, (b == 2 || b == 3) ? 1 : 0);
}

// FCC lattice vectors of shells 1..3 (|v|^2 = 2, 4, 6 half units squared),
// shell-major, lexicographic inside a shell: the canonical order of the
// library and the oracle (shell-1 index = partner direction).
struct FVec {
  int x, y, z, k;
};
struct FTable {
  FVec v[42];
  int n;
};
__host__ __device__ constexpr FTable make_fvecs() {
  FTable t{};
  t.n = 0;
  for (int k = 0; k < 3; k++)
    for (int x = -2; x <= 2; x++)
      for (int y = -2; y <= 2; y++)
        for (int z = -2; z <= 2; z++) {
          if ((x + y + z) & 1) continue;
          if (x * x + y * y + z * z == 2 * (k + 1)) {
            t.v[t.n] = FVec{x, y, z, k};
            t.n++;
          }
        }
  return t;
}

// Stage the tile and its 2-cell halo from 32-bit words of the site store,
// CPW cells per word (2: 16-bit cells of four 4-bit ids; 1: four int8 ids).
// Box column c of a row holds the cell at global x = t0x - 2 + c (periodic);
// the NWR words of a box row start at the multiple of CPW at or below
// t0x - 2, and with nx a multiple of CPW no word straddles the wrap.  Lane l
// of a warp takes word l % NWR of row l / NWR of each group of RPS rows; warp
// w stages the planes w, w + nwarp, ..., and issues the loads of PLB planes
// (PLB * RS words per lane) before it unpacks them.  The box holds SC times the
// species.
template <int SC, int CPW>
__device__ __forceinline__ void stage_words(const LatDesc& D, uint8_t* box, const int (&t0)[3], int ex, int ey,
                                            int ez, int lane, int warp, int nwarp) {
  constexpr int BE = TMAX + 2 * H;               // box edge (cells)
  constexpr int NWR = CPW == 2 ? BE / 2 + 1 : BE;  // words per box row (10 or 19)
  constexpr int RPS = 32 / NWR;                  // rows per warp step (3 or 1)
  constexpr int RS = (BE + RPS - 1) / RPS;       // steps per plane (7 or 19)
  constexpr int PLB = CPW == 2 ? 2 : 1;          // planes per batch of loads
  const int nx = D.n[0], ny = D.n[1], nz = D.n[2];
  const int xs = t0[0] - H;
  const int r = xs & (CPW - 1);
  const int m = lane % NWR, ry = lane / NWR;
  const bool lane_ok = ry < RPS && CPW * m - r < ex;
  int gw = (xs - r + CPW * m) % nx;  // first cell of this lane's word
  gw += gw < 0 ? nx : 0;
  const uint32_t* words = reinterpret_cast<const uint32_t*>(D.sites);
  const long long nword = (long long)nx * ny * nz / CPW;
  for (int zb = warp; zb < ez; zb += nwarp * PLB) {
    uint32_t v[PLB][RS];
#pragma unroll
    for (int p = 0; p < PLB; p++) {
      const int zs = zb + p * nwarp;
      const long long zrow = zs < ez ? (long long)wrap_add(t0[2] - H, zs, nz) * ny : 0;
#pragma unroll
      for (int q = 0; q < RS; q++) {
        const int ys = RPS * q + ry;
        v[p][q] = 0;
        if (zs < ez && ys < ey && lane_ok) {
          const long long cell = (zrow + wrap_add(t0[1] - H, ys, ny)) * nx + gw;
          v[p][q] = ld_chk(words, cell / CPW, nword, kDbgSite);
        }
      }
    }
#pragma unroll
    for (int p = 0; p < PLB; p++) {
      const int zs = zb + p * nwarp;
#pragma unroll
      for (int q = 0; q < RS; q++) {
        const int ys = RPS * q + ry;
        if (zs < ez && ys < ey && lane_ok) {
#pragma unroll
          for (int j = 0; j < CPW; j++) {
            const int c = CPW * m + j - r;
            if (c >= 0 && c < ex) {
              const uint32_t cv = CPW == 2 ? (v[p][q] >> (16 * j)) & 0xFFFFu : v[p][q];
              const int base = hoff(2 * c, 2 * ys, 2 * zs);
#pragma unroll
              for (int b = 0; b < 4; b++) {
                const uint32_t sp = CPW == 2 ? (cv >> (4 * b)) & 15u : (cv >> (8 * b)) & 0xFFu;
                st_chk(box, base + boff(b), BOX_BYTES, kDbgFccBox, (uint8_t)(sp * SC));
              }
            }
          }
        }
      }
    }
  }
}

// Stage a tile (origin t0, extent ts) and its 2-cell halo: from 32-bit words
// when the rows allow it, else cell by cell.  Every thread of the CTA takes part.
template <int SC>
__device__ __forceinline__ void stage_box(const LatDesc& D, uint8_t* box, const int (&t0)[3], const int (&ts)[3],
                                          int lane, int warp, int nwarp) {
  const int ex = ts[0] + 2 * H, ey = ts[1] + 2 * H, ez = ts[2] + 2 * H;
  const int nx = D.n[0], ny = D.n[1], nz = D.n[2];
  if (D.storage == SMCX_INT8)
    stage_words<SC, 1>(D, box, t0, ex, ey, ez, lane, warp, nwarp);
  else if ((nx & 1) == 0)
    stage_words<SC, 2>(D, box, t0, ex, ey, ez, lane, warp, nwarp);
  else {
    // odd x extent, 16-bit cells: one box column (cell x) per lane, warp w
    // the planes w, w + nwarp, ..., 8 rows of global loads in flight per lane
    constexpr int U = 8;
    const int gx = lane < ex ? wrap_add(t0[0] - H, lane, nx) : 0;
    for (int zs = warp; zs < ez; zs += nwarp) {
      const long long zrow = (long long)wrap_add(t0[2] - H, zs, nz) * ny;
      for (int ys0 = 0; ys0 < ey; ys0 += U) {
        uint32_t v[U];
#pragma unroll
        for (int u = 0; u < U; u++) {
          const int ys = ys0 + u;
          v[u] = 0;
          if (ys < ey && lane < ex) {
            const long long cell = (zrow + wrap_add(t0[1] - H, ys, ny)) * nx + gx;
            v[u] = (uint32_t)(*reinterpret_cast<const uint16_t*>(D.sites + 2 * cell));
          }
        }
#pragma unroll
        for (int u = 0; u < U; u++) {
          const int ys = ys0 + u;
          if (ys < ey && lane < ex) {
            const int base = hoff(2 * lane, 2 * ys, 2 * zs);
#pragma unroll
            for (int b = 0; b < 4; b++) {
              const uint32_t sp = (v[u] >> (4 * b)) & 15u;
              st_chk(box, base + boff(b), BOX_BYTES, kDbgFccBox, (uint8_t)(sp * SC));
            }
          }
        }
      }
    }
  }
}

}  // namespace fccfast
}  // namespace smcx
