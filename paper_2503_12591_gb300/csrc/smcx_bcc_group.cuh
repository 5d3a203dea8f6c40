// BCC tile pass with two or four lanes per trial, for sweeps that leave most of the
// GPU idle.
//
// Same trials, same order of phases, same Philox words and the same integer arithmetic
// as bcc_tile_pass (smcx_bcc_tile.cuh): bit-identical.  A tile pass is a chain of 2 L^3
// phases; with a tile or two on an SM a phase lasts as long as its one thread needs
// for a trial, some 480 instructions at 3.5 cycles each.  Here the lanes of a trial
// share its 100 neighbour loads: with two, lane 0 takes the environment of s and lane
// 1 that of s'; with four, every lane takes one half shell +w or its mirror image -w
// around s or s'.  The shells are symmetric, so all lanes run the same loads at
// c + sigma off(w), sigma = +-1: the offset of -w from one sublattice is minus the
// offset of w from the other, and for odd w the two sublattices' offsets differ by a
// constant.  Exchanges between lanes add the byte counters up.  The Philox block of
// the next phase is drawn between the loads and the exchanges, which it fills.
//
// ms per sweep with one, two and four lanes per trial (4 shells, M <= 4, L = 4):
// 24^3 cells 0.870, 0.665, 0.612; 48^3 0.879, 0.673, 0.621 (3^3 slots); 64^3 0.823,
// 0.799, 0.833 (4^3 slots; shared directions 0.816, 0.705, 0.772); 80^3 0.902, 1.101,
// 1.245 (5^3 slots: the SM has warps enough with one).
#pragma once

#include "smcx_bcc_tile.cuh"

namespace smcx {
namespace bccfast {

constexpr int kMaxGroupNQ = 4;  // link-cell slots per axis at most
// lanes per trial, threads of a CTA
__host__ __device__ constexpr int group_lanes(int nq) { return nq <= 3 ? 4 : 2; }
__host__ __device__ constexpr int group_threads(int nq) {
  return (group_lanes(nq) * nq * nq * nq + 31) / 32 * 32;
}
constexpr int kGroupThreads = 128;  // 4 lanes x 3^3 slots or 2 lanes x 4^3

__host__ __device__ constexpr bool plus_half(const Vec& v) {
  return v.x > 0 || (v.x == 0 && (v.y > 0 || (v.y == 0 && v.z > 0)));
}
// off_1(w) - off_0(w) for odd w (nb_offset of the two sublattices)
constexpr int kOddShift = PP + PX + 1 - 2 * SUB;
__host__ __device__ constexpr bool odd_shift_ok() {
  constexpr VecTable T = make_vecs();
  for (int j = 0; j < T.n; j++) {
    const Vec v = T.v[j];
    const int d = nb_offset(1, v.x, v.y, v.z) - nb_offset(0, v.x, v.y, v.z);
    if (d != ((v.x & 1) ? kOddShift : 0)) return false;
    if (nb_offset(0, -v.x, -v.y, -v.z) != -nb_offset(1, v.x, v.y, v.z)) return false;
  }
  return true;
}
static_assert(odd_shift_ok(), "mirror images of the neighbour offsets");

struct GroupMem {
  uint32_t rows[128];  // V-difference rows (Planes::R)
  uint8_t dir[512];    // phase directions (shared-direction proposals)
  unsigned long long stat[3];
};

// Every thread of the CTA (a multiple of 32, at least LN per slot of any tile) must
// call it.  Shared directions: 2 L^3 <= 512.
template <int LN, int K, int NW, int PL>
__device__ __forceinline__ void group_pass(const LatDesc& D, const Planes& Q, int tc, int jt, unsigned long long sweep,
                                           uint8_t* box, uint32_t* sA, uint32_t* sB, GroupMem& M) {
  const int tid = threadIdx.x, nth = blockDim.x;
  const int lane = tid & 31, warp = tid >> 5, nwarp = nth >> 5;
  const int ntc0 = D.nt[0] / 2, ntc1 = D.nt[1] / 2;
  const int jx = jt % ntc0, jy = (jt / ntc0) % ntc1, jz = jt / (ntc0 * ntc1);
  const int ti[3] = {2 * jx + (tc & 1), 2 * jy + ((tc >> 1) & 1), 2 * jz + ((tc >> 2) & 1)};
  int t0[3], ts[3];
#pragma unroll
  for (int a = 0; a < 3; a++) {
    const int base = D.n[a] / D.nt[a], rem = D.n[a] % D.nt[a];
    ts[a] = base + (ti[a] < rem ? 1 : 0);
    t0[a] = ti[a] * base + min(ti[a], rem);
  }
  const bool shared_dir = D.proposal != 0;
  const bool use_rows = K == 4 && NW == 1 && PL == 2 && Q.rows;
  const int NQ = D.NQ, L = D.L, nx = D.n[0], ny = D.n[1];
  __syncthreads();  // the previous pass of this CTA is done with the box and the tables
  if (tid < 3) M.stat[tid] = 0;
  for (int i = tid; i < D.nA; i += nth) sA[i] = D.thr[i];
  for (int i = tid; i < kNB; i += nth) sB[i] = D.thr[kNA + i];
  if (use_rows)
    for (int i = tid; i < 128; i += nth) M.rows[i] = Q.R[i >> 3][i & 7];
  if (shared_dir) {
    const unsigned tile = (unsigned)((ti[2] * D.nt[1] + ti[1]) * D.nt[0] + ti[0]);
    for (int pr = tid; pr < L * L * L; pr += nth) {
      const uint4 r = D.proposal == 2 ? block_direction_block(D.seed_lo, D.seed_hi, sweep, D.replica, tc,
                                                              (unsigned)jt >> 1, pr)
                                      : phase_direction_block(D.seed_lo, D.seed_hi, sweep, D.replica, tile, pr);
      st_chk(M.dir, 2 * pr, 512, kDbgBccDir, (uint8_t)(r.x >> 29));
      st_chk(M.dir, 2 * pr + 1, 512, kDbgBccDir, (uint8_t)(r.z >> 29));
    }
  }
  stage_box(D, box, t0, ts, lane, warp, nwarp);
  __syncthreads();

  const int g = tid % LN;
  int q = tid / LN;
  // the bank-spreading order of 4^3 slots (two lanes)
  if (NQ >= kOrderMinNQ && L >= kOrderMinL && L <= kOrderMaxL && nth >= LN * order_lanes(NQ))
    q = q < order_lanes(NQ) ? (int)d_slot_orders.q[NQ - kOrderMinNQ][L - kOrderMinL][q] : 255;
  const int qx = q % NQ, qy = (q / NQ) % NQ, qz = q / (NQ * NQ);
  const bool slot = q < NQ * NQ * NQ;
  const bool part = (g & 1) != 0;  // around s'
  const int sigma = LN == 4 && g >= 2 ? -1 : 1;
  unsigned acc = 0, same = 0;
  long long dsum = 0;
  int cx = 0, cy = 0, cz = 0;
  auto draw = [&](int x, int y, int z) {
    const unsigned long long cell =
        ((unsigned long long)(t0[2] + z + L * qz) * ny + (t0[1] + y + L * qy)) * nx + (t0[0] + x + L * qx);
    return attempt_block(cell * 2, sweep, D.replica, D.seed_lo, D.seed_hi);
  };
  uint4 rw = draw(0, 0, 0);
  for (int ph = 0; ph < L * L * L; ph++) {
    const int xr = cx + L * qx, yr = cy + L * qy, zr = cz + L * qz;
    const bool live = slot && xr < ts[0] && yr < ts[1] && zr < ts[2];
    // lanes without a trial follow at some valid place of the box
    const int s0 = live ? (zr + 2) * PP + (yr + 2) * PX + (xr + 2) : 4 * PP + 4 * PX + 4;
    if (++cx == L) {
      cx = 0;
      if (++cy == L) {
        cy = 0;
        cz++;
      }
    }
    uint4 next;
#pragma unroll
    for (int B = 0; B < 2; B++) {
      const int dir = shared_dir ? (int)ld_chk(M.dir, 2 * ph + B, 512, kDbgBccDir) : (int)((B ? rw.z : rw.x) >> 29);
      const uint32_t ru = B ? rw.w : rw.y;
      const int dx = ((dir >> 2) & 1) - 1 + B, dy = ((dir >> 1) & 1) - 1 + B, dz = (dir & 1) - 1 + B;
      const int s = s0 + B * SUB;
      const int sp = s + (1 - 2 * B) * SUB + dz * PP + dy * PX + dx;
      const uint32_t a8 = ld_chk(box, s, 2 * SUB, kDbgBccBox), b8 = ld_chk(box, sp, 2 * SUB, kDbgBccBox);
      // this lane's centre, on sublattice B (s) or 1 - B (s')
      const int c = part ? sp : s;
      const bool sub = part != (B == 1);
      const int codd = c + (sigma > 0 ? (sub ? kOddShift : 0) : (sub ? 0 : -kOddShift));
      uint32_t h[kMaxShells][2];
#pragma unroll
      for (int k = 0; k < K; k++) h[k][0] = h[k][1] = 0;
      constexpr VecTable T = make_vecs();
#pragma unroll
      for (int j = 0; j < T.n; j++) {
        const Vec w = T.v[j];
        if (w.k >= K || (LN == 4 && !plus_half(w))) continue;
        const int off = (LN == 4 ? sigma : 1) * nb_offset(0, w.x, w.y, w.z);
        add_one<NW>(h[w.k], ld_chk(box, ((w.x & 1) ? codd : c) + off, 2 * SUB, kDbgBccBox), +1);
      }
      if (B == 1) next = draw(cx, cy, cz);  // one phase ahead: independent of the box
#pragma unroll
      for (int k = 0; k < K; k++)
#pragma unroll
        for (int w = 0; w < NW; w++) {
          uint32_t x = part ? 0u - h[k][w] : h[k][w];
          x += __shfl_xor_sync(0xffffffffu, x, 1);
          if (LN == 4) x += __shfl_xor_sync(0xffffffffu, x, 2);
          h[k][w] = 0x80808080u + x;
        }
      if (live && g == 0) {
        if (a8 == b8) {
          same++;
        } else {
          // the s-s' bond is not part of either environment after the swap
          add_one<NW>(h[0], b8, -1);
          add_one<NW>(h[0], a8, +1);
          if (use_rows) finish_trial_rows<K>(box, s, sp, a8, b8, h, ru, M.rows, D.nA, sA, sB, acc, dsum);
          else finish_trial<K, NW, PL>(box, s, sp, a8, b8, h, ru, Q, D.nA, sA, sB, acc, dsum);
        }
      }
      __syncthreads();
    }
    rw = next;
  }

  // write back tile + 1-cell partner ring: one lane per column, warp w the planes w,
  // w + nwarp, ...
  const int wx = ts[0] + 2, wy = ts[1] + 2, wz = ts[2] + 2;
  const int nz = D.n[2];
  const long long ncell = (long long)nx * ny * nz;
  const int gxw = lane < wx ? wrap_add(t0[0] - 1, lane, nx) : 0;
  for (int zw = warp; zw < wz; zw += nwarp) {
    const long long zrow = (long long)wrap_add(t0[2] - 1, zw, nz) * ny;
#pragma unroll 4
    for (int yw = 0; yw < wy; yw++) {
      if (lane < wx) {
        const long long cell = (zrow + wrap_add(t0[1] - 1, yw, ny)) * nx + gxw;
        const int bi = (zw + 1) * PP + (yw + 1) * PX + (lane + 1);
        const uint32_t s0 = ld_chk(box, bi, 2 * SUB, kDbgBccWrite) >> 3;
        const uint32_t s1 = ld_chk(box, SUB + bi, 2 * SUB, kDbgBccWrite) >> 3;
        if (D.storage == SMCX_INT8) {
          st_chk(D.sites, 2 * cell, 2 * ncell, kDbgSite, (uint8_t)s0);
          st_chk(D.sites, 2 * cell + 1, 2 * ncell, kDbgSite, (uint8_t)s1);
        } else {
          st_chk(D.sites, cell, ncell, kDbgSite, (uint8_t)(s0 | (s1 << 4)));
        }
      }
    }
  }
  add_stats_warp(M.stat, acc, same, dsum);
  __syncthreads();
  if (tid == 0) {
    atomicAdd(&D.stats[0], (unsigned long long)ts[0] * ts[1] * ts[2] * 2);
    atomicAdd(&D.stats[1], M.stat[0]);
    atomicAdd(&D.stats[2], M.stat[1]);
    atomicAdd(&D.stats[3], M.stat[2]);
  }
}

// Single-lattice sweep kernel: one CTA per tile of colour `tc`.
template <int LN, int K, int NW, int PL>
__global__ void __launch_bounds__(kGroupThreads, 4) k_bcc_group_sweep(const LatDesc D, const Planes Q, int tc) {
  extern __shared__ __align__(16) unsigned char smem[];
  __shared__ __align__(16) GroupMem M;
  uint32_t* sA = reinterpret_cast<uint32_t*>(smem + 2 * SUB);
  group_pass<LN, K, NW, PL>(D, Q, tc, blockIdx.x, D.sweep, smem, sA, sA + D.nA, M);
}

}  // namespace bccfast
}  // namespace smcx
