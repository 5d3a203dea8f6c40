// Local-energy field and clusters (Results, FeCoNiAlTi one-billion-atom
// section; Method "MC simulation": the local energy of every site is
// computed, an energy threshold decides which neighbouring sites belong to
// one set, and union-find collects the sets).
//
//  * e2[i] = 2 E_i = sum_k sum_{v in shell k} V_k[s_i][s_{i+v}] (Eq.
//    Linear_EPI without the bias terms, each bond counted at both ends, so
//    sum_i e2[i] = 2 E), plus 2 sum_k W_k[s_i] n_k(i)^2 under the qSRO model
//    (Eq. quadratic_local_SRO).  FCC lattices and BCC lattices of at most four
//    species are read in shared-memory tiles (k_local_tile: a shared load, a
//    shift and an addition per neighbour, then dp4a against the byte planes of
//    V); other shapes gather from the lattice store, a thread per cell.
//  * class(i) = e2[i] < thr2.  Two shell-1 neighbours of one class are in
//    one cluster.  Concurrent union-find over int32 parents: a root is only
//    ever linked below a smaller root with a compare-and-swap, so parents
//    decrease along every path, paths can be halved with plain stores, and
//    the final root of a cluster is its smallest site id (a unique label).
//    Parents are read with volatile loads (L2, coherent across SMs).  Every
//    find and union loop has an iteration limit that raises an error flag.
//    On the tiled path a CTA first joins the sites of its own tile in shared
//    memory (k_label_tile), so that only pairs across tile faces go through
//    global memory (k_label_faces).
//  * Summary: cluster sizes and species counts by atomics that are gathered per
//    CTA in shared memory first (a percolating cluster would otherwise take an
//    atomic of every warp), the clusters of at least min_size sites listed on the
//    device and the largest selected on the host.
#include <algorithm>
#include <vector>

#include "smcx_fcc_tile.cuh"
#include "smcx_tiles.cuh"

namespace smcx {

void fill_offsets_global(const smcx_lattice* hd, SweepParams& P);

namespace {

constexpr int kFindLimit = 1 << 22;
constexpr int kUnionLimit = 1 << 20;

// Half of shell 1 (first nonzero half-unit component positive), per centre
// sublattice: global (dx, dy, dz, b').
struct HalfShell {
  signed char d[4][8][4];
  int n;
};

__device__ __forceinline__ long long nb_gid(const SweepParams& P, int x, int y, int z, const signed char* d, int m) {
  return (((long long)wrap_add(z, d[2], P.n[2]) * P.n[1] + wrap_add(y, d[1], P.n[1])) * P.n[0] +
          wrap_add(x, d[0], P.n[0])) * m + d[3];
}

// qSRO weights W[k][c] (on = 0: pair model)
struct QsroWeights {
  int32_t w[kMaxShells * kMaxSweepM];
  int on;
};

template <int KIND, int K>
__global__ void __launch_bounds__(256) k_local_energy2(const SweepParams P, const int32_t* __restrict__ dV,
                                                       const QsroWeights QW, int32_t* e2, uint8_t* cls,
                                                       long long thr2) {
  constexpr int m = cell_sites(KIND);
  __shared__ int32_t sV[kMaxShells * kMaxSweepM * kMaxSweepM];
  __shared__ int32_t sW[kMaxShells * kMaxSweepM];
  const int M = P.M;
  for (int i = threadIdx.x; i < K * M * M; i += blockDim.x) sV[i] = dV[i];
  for (int i = threadIdx.x; i < K * M; i += blockDim.x) sW[i] = QW.on ? QW.w[i] : 0;
  __syncthreads();
  const long long ncell = (long long)P.n[0] * P.n[1] * P.n[2];
  for (long long c = (long long)blockIdx.x * blockDim.x + threadIdx.x; c < ncell;
       c += (long long)gridDim.x * blockDim.x) {
    const int x = (int)(c % P.n[0]);
    const long long r = c / P.n[0];
    const int y = (int)(r % P.n[1]), z = (int)(r / P.n[1]);
    for (int b = 0; b < m; b++) {
      const int p = load_site(P.sites, c * m + b, P.storage);
      int acc = 0;
      int j = 0;
#pragma unroll
      for (int k = 0; k < K; k++) {
        const int32_t* row = sV + (k * M + p) * M;
        int n = 0;
#pragma unroll 4
        for (int q = 0; q < shell_size(KIND, k); q++, j++) {
          const int c = load_site(P.sites, nb_gid(P, x, y, z, P.gd[b][j], m), P.storage);
          acc += row[c];
          n += (c == p);
        }
        acc += 2 * sW[k * M + p] * n * n;  // qSRO term (W = 0 for the pair model)
      }
      if (e2) e2[c * m + b] = acc;
      if (cls) cls[c * m + b] = (uint8_t)((long long)acc < thr2);
    }
  }
}

__global__ void k_label_init(int32_t* lab, long long N) {
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < N; i += (long long)gridDim.x * blockDim.x)
    lab[i] = (int32_t)i;
}

__device__ __forceinline__ int find_root(int32_t* lab, int x, int* flag) {
  volatile int32_t* p = lab;
  for (int it = 0; it < kFindLimit; it++) {
    const int px = p[x];
    if (px == x) return x;
    const int gx = p[px];
    if (gx != px) p[x] = gx;  // halving: gx < px < x, still an ancestor
    x = gx;
  }
  atomicOr(flag, 1);
  return x;
}

__device__ __forceinline__ void unite(int32_t* lab, int a, int b, int* flag) {
  for (int it = 0; it < kUnionLimit; it++) {
    a = find_root(lab, a, flag);
    b = find_root(lab, b, flag);
    if (a == b) return;
    if (a < b) {
      const int t = a;
      a = b;
      b = t;
    }
    if (atomicCAS(&lab[a], a, b) == a) return;  // a was a root: now below b
  }
  atomicOr(flag, 2);
}

template <int KIND>
__global__ void __launch_bounds__(256) k_hook(const SweepParams P, const HalfShell H, const uint8_t* cls, int32_t* lab,
                                              int* flag) {
  constexpr int m = cell_sites(KIND);
  const long long ncell = (long long)P.n[0] * P.n[1] * P.n[2];
  for (long long c = (long long)blockIdx.x * blockDim.x + threadIdx.x; c < ncell;
       c += (long long)gridDim.x * blockDim.x) {
    const int x = (int)(c % P.n[0]);
    const long long r = c / P.n[0];
    const int y = (int)(r % P.n[1]), z = (int)(r / P.n[1]);
#pragma unroll
    for (int b = 0; b < m; b++) {
      const long long i = c * m + b;
      const uint8_t ci = cls[i];
      for (int j = 0; j < H.n; j++) {
        const long long t = nb_gid(P, x, y, z, H.d[b][j], m);
        if (cls[t] == ci && t != i) unite(lab, (int)i, (int)t, flag);
      }
    }
    if (*(volatile int*)flag) return;
  }
}

// ---- tiles -----------------------------------------------------------------
// Byte planes of V for dp4a against neighbour counts: P[j][k][p] holds bytes j of
// V_k[p][c]: BCC word 0 for c = 0..3; FCC word 0 for c = 0, 2, 4, 6 and word 1
// for c = 1, 3, 5, 7 (planes 0 and 1 unsigned, 2 signed); W: qSRO weights.
struct LocalTab {
  uint32_t P[3][kMaxShells][kMaxSweepM][2];
  int32_t W[kMaxShells][kMaxSweepM];
};
constexpr int kTabWords = sizeof(LocalTab) / 4;

// The lattice kinds as the tile kernels see them: box scale, sites of a cell,
// offset of site b of a cell, half of shell 1.
template <int KIND>
struct TileGeom;
template <>
struct TileGeom<kBCC> {
  static constexpr int m = 2, kBoxBytes = 2 * bccfast::SUB, kEdge = 20, kLabelEdge = 16;
  static __device__ __forceinline__ int cell(int x, int y, int z) {
    return (z + 2) * bccfast::PP + (y + 2) * bccfast::PX + (x + 2);
  }
  static __device__ __forceinline__ int site(int b) { return b * bccfast::SUB; }
  static __device__ __forceinline__ void stage(const bccfast::LatDesc& D, uint8_t* box, const int (&t0)[3],
                                               const int (&ts)[3]) {
    bccfast::stage_box(D, box, t0, ts, threadIdx.x & 31, threadIdx.x >> 5, blockDim.x >> 5);
  }
};
template <>
struct TileGeom<kFCC> {
  static constexpr int m = 4, kBoxBytes = fccfast::BOX_BYTES, kEdge = fccfast::TMAX, kLabelEdge = 12;
  static __device__ __forceinline__ int cell(int x, int y, int z) {
    return fccfast::hoff(2 * (x + fccfast::H), 2 * (y + fccfast::H), 2 * (z + fccfast::H));
  }
  static __device__ __forceinline__ int site(int b) { return fccfast::boff(b); }
  static __device__ __forceinline__ void stage(const bccfast::LatDesc& D, uint8_t* box, const int (&t0)[3],
                                               const int (&ts)[3]) {
    fccfast::stage_box<4>(D, box, t0, ts, threadIdx.x & 31, threadIdx.x >> 5, blockDim.x >> 5);
  }
};

// 2 E of BCC sublattice B at box index s.  The box holds 8 sigma: a neighbour
// adds 1 << (8 sigma) to the byte counters of its shell (at most 24).
template <int B, int K>
__device__ __forceinline__ int local2_bcc(const uint8_t* box, int s, const LocalTab& T, bool qsro) {
  using namespace bccfast;
  constexpr VecTable V = make_vecs();
  const int p = (ld_chk(box, s, 2 * SUB, kDbgBccBox) >> 3) & 3;
  uint32_t h[K];
#pragma unroll
  for (int k = 0; k < K; k++) h[k] = 0;
#pragma unroll
  for (int j = 0; j < V.n; j++)
    if (V.v[j].k < K) h[V.v[j].k] += 1u << (ld_chk(box, s + nb_offset(B, V.v[j].x, V.v[j].y, V.v[j].z), 2 * SUB, kDbgBccBox) & 31);
  int a0 = 0, a1 = 0, a2 = 0, q = 0;
#pragma unroll
  for (int k = 0; k < K; k++) {
    a0 = dp4a_su((int)h[k], T.P[0][k][p][0], a0);
    a1 = dp4a_su((int)h[k], T.P[1][k][p][0], a1);
    a2 = dp4a_ss((int)h[k], T.P[2][k][p][0], a2);
    if (qsro) {
      const int n = (int)((h[k] >> (8 * p)) & 255u);
      q += 2 * T.W[k][p] * n * n;
    }
  }
  return a0 + (a1 << 8) + (a2 << 16) + q;
}

// 2 E of the FCC site at box index s.  The box holds 4 sigma: the two halves of
// a shell count in nibbles (at most 12 each), whose sum is taken in bytes, even
// and odd species apart.
template <int K>
__device__ __forceinline__ int local2_fcc(const uint8_t* box, int s, const LocalTab& T, bool qsro) {
  using namespace fccfast;
  constexpr FTable V = make_fvecs();
  const int p = (ld_chk(box, s, BOX_BYTES, kDbgFccBox) >> 2) & 7;
  uint32_t hp[K], hm[K];
#pragma unroll
  for (int k = 0; k < K; k++) hp[k] = hm[k] = 0;
#pragma unroll
  for (int j = 0; j < V.n; j++)
    if (V.v[j].k < K) {
      const uint32_t one = 1u << (ld_chk(box, s + hoff(V.v[j].x, V.v[j].y, V.v[j].z), BOX_BYTES, kDbgFccBox) & 31);
      const bool half = V.v[j].x > 0 || (V.v[j].x == 0 && (V.v[j].y > 0 || (V.v[j].y == 0 && V.v[j].z > 0)));
      if (half) hp[V.v[j].k] += one;
      else hm[V.v[j].k] += one;
    }
  int a0 = 0, a1 = 0, a2 = 0, q = 0;
#pragma unroll
  for (int k = 0; k < K; k++) {
    const uint32_t e = (hp[k] & 0x0F0F0F0Fu) + (hm[k] & 0x0F0F0F0Fu);
    const uint32_t o = ((hp[k] >> 4) & 0x0F0F0F0Fu) + ((hm[k] >> 4) & 0x0F0F0F0Fu);
    a0 = bccfast::dp4a_su((int)o, T.P[0][k][p][1], bccfast::dp4a_su((int)e, T.P[0][k][p][0], a0));
    a1 = bccfast::dp4a_su((int)o, T.P[1][k][p][1], bccfast::dp4a_su((int)e, T.P[1][k][p][0], a1));
    a2 = bccfast::dp4a_ss((int)o, T.P[2][k][p][1], bccfast::dp4a_ss((int)e, T.P[2][k][p][0], a2));
    if (qsro) {
      const int n = (int)((((p & 1) ? o : e) >> (8 * (p >> 1))) & 255u);
      q += 2 * T.W[k][p] * n * n;
    }
  }
  return a0 + (a1 << 8) + (a2 << 16) + q;
}

template <int KIND, int K>
__device__ __forceinline__ int local2(const uint8_t* box, int cbase, int b, const LocalTab& T, bool qsro) {
  if constexpr (KIND == kBCC)
    return b == 0 ? local2_bcc<0, K>(box, cbase, T, qsro) : local2_bcc<1, K>(box, cbase + bccfast::SUB, T, qsro);
  else
    return local2_fcc<K>(box, cbase + fccfast::boff(b), T, qsro);
}

__device__ __forceinline__ void load_tab(LocalTab& sT, const LocalTab& T) {
  for (int i = threadIdx.x; i < kTabWords; i += blockDim.x)
    reinterpret_cast<uint32_t*>(&sT)[i] = reinterpret_cast<const uint32_t*>(&T)[i];
}

// 2 E_i of every site of the tile.
template <int KIND, int K>
__global__ void __launch_bounds__(256) k_local_tile(const bccfast::LatDesc D, const LocalTab T, int qsro, int32_t* e2) {
  using G = TileGeom<KIND>;
  extern __shared__ __align__(16) unsigned char smem[];
  __shared__ LocalTab sT;
  int t0[3], ts[3];
  bccfast::tile_of_index(D, blockIdx.x, t0, ts);
  load_tab(sT, T);
  G::stage(D, smem, t0, ts);
  __syncthreads();
  const bccfast::CellIndex ci(ts);
  const int ncell = ts[0] * ts[1] * ts[2];
  for (int c = threadIdx.x; c < ncell; c += blockDim.x) {
    int x, y, z;
    ci.at(c, x, y, z);
    const int cb = G::cell(x, y, z);
    const long long cell = ((long long)(t0[2] + z) * D.n[1] + (t0[1] + y)) * D.n[0] + (t0[0] + x);
#pragma unroll(KIND == kBCC ? 2 : 1)
    for (int b = 0; b < G::m; b++) e2[cell * G::m + b] = local2<KIND, K>(smem, cb, b, sT, qsro != 0);
  }
}

// Union-find in shared memory: as find_root and unite, on local site indices
// (cell of the tile * m + b, in the order of the global ids).
__device__ __forceinline__ int find_local(int* lab, int x, int* flag) {
  volatile int* p = lab;
  for (int it = 0; it < kFindLimit; it++) {
    const int px = p[x];
    if (px == x) return x;
    const int gx = p[px];
    if (gx != px) p[x] = gx;
    x = gx;
  }
  atomicOr(flag, 1);
  return x;
}
__device__ __forceinline__ void unite_local(int* lab, int a, int b, int* flag) {
  for (int it = 0; it < kUnionLimit; it++) {
    a = find_local(lab, a, flag);
    b = find_local(lab, b, flag);
    if (a == b) return;
    if (a < b) {
      const int t = a;
      a = b;
      b = t;
    }
    if (atomicCAS(&lab[a], a, b) == a) return;
  }
  atomicOr(flag, 2);
}

// Classes of the tile's sites and their clusters inside the tile: lab[i] = the
// smallest id of i's cluster within the tile, cls[i] = class, bit 1 set where i
// is that smallest id.  Tiles of at most kLabelEdge cells; pairs that leave the
// tile's own range of cells (periodic images too) are left to k_label_faces.  16.4M
// FCC sites, 3 shells, 20% of them below the threshold: 614 us (shared-memory
// latency of the finds) against 1428 for the energies and 2364 for the unions of
// every pair through global memory.
template <int KIND, int K>
__global__ void __launch_bounds__(256, 3) k_label_tile(const bccfast::LatDesc D, const LocalTab T, int qsro,
                                                    long long thr2, const HalfShell H, uint8_t* cls, int32_t* lab,
                                                    int* flag) {
  using G = TileGeom<KIND>;
  constexpr int m = G::m;
  extern __shared__ __align__(16) unsigned char smem[];
  __shared__ LocalTab sT;
  int* s_lab = reinterpret_cast<int*>(smem + (G::kBoxBytes + 15) / 16 * 16);
  uint8_t* s_cls = reinterpret_cast<uint8_t*>(s_lab + G::kLabelEdge * G::kLabelEdge * G::kLabelEdge * m);
  int t0[3], ts[3];
  bccfast::tile_of_index(D, blockIdx.x, t0, ts);
  load_tab(sT, T);
  G::stage(D, smem, t0, ts);
  __syncthreads();
  const bccfast::CellIndex ci(ts);
  const int ncell = ts[0] * ts[1] * ts[2];
  for (int c = threadIdx.x; c < ncell; c += blockDim.x) {
    int x, y, z;
    ci.at(c, x, y, z);
    const int cb = G::cell(x, y, z);
#pragma unroll(KIND == kBCC ? 2 : 1)
    for (int b = 0; b < m; b++) {
      s_cls[c * m + b] = (uint8_t)((long long)local2<KIND, K>(smem, cb, b, sT, qsro != 0) < thr2);
      s_lab[c * m + b] = c * m + b;
    }
  }
  __syncthreads();
  for (int c = threadIdx.x; c < ncell; c += blockDim.x) {
    int x, y, z;
    ci.at(c, x, y, z);
    for (int b = 0; b < m; b++) {
      const int i = c * m + b;
      const uint8_t cc = s_cls[i];
      for (int j = 0; j < H.n; j++) {
        const signed char* d = H.d[b][j];
        const int nx = x + d[0], ny = y + d[1], nz = z + d[2];
        if ((unsigned)nx >= (unsigned)ts[0] || (unsigned)ny >= (unsigned)ts[1] || (unsigned)nz >= (unsigned)ts[2]) continue;
        const int t = ((nz * ts[1] + ny) * ts[0] + nx) * m + d[3];
        if (s_cls[t] == cc) unite_local(s_lab, i, t, flag);
      }
    }
  }
  __syncthreads();
  for (int c = threadIdx.x; c < ncell; c += blockDim.x) {
    int x, y, z;
    ci.at(c, x, y, z);
    const long long cell = ((long long)(t0[2] + z) * D.n[1] + (t0[1] + y)) * D.n[0] + (t0[0] + x);
    for (int b = 0; b < m; b++) {
      const int i = c * m + b;
      int r = i;
      for (int it = 0; it < kFindLimit; it++) {  // parents decrease: ends at the root
        const int pr = s_lab[r];
        if (pr == r) break;
        r = pr;
      }
      int rx, ry, rz;
      ci.at(r / m, rx, ry, rz);
      const long long root = ((long long)(t0[2] + rz) * D.n[1] + (t0[1] + ry)) * D.n[0] + (t0[0] + rx);
      lab[cell * m + b] = (int32_t)(root * m + r % m);
      cls[cell * m + b] = (uint8_t)(s_cls[i] | (r == i ? 2 : 0));
    }
  }
}

// Joins the pairs of shell-1 neighbours whose second site lies outside the tile
// of the first.  A site's label is the root of its cluster within its tile or, for
// such a root, something below it; two tiles meet in many pairs of the same two
// clusters, so the CTA remembers the pairs of labels it has joined in a
// direct-mapped table (an exchange tells whether the last user of the slot was the
// same pair) and joins each pair about once: 385 us for 16.4M FCC sites with a
// percolating class, 1457 us with a union per pair of sites.  Bound by the latency
// of the label reads.
constexpr int kSeenSlots = 2048;
template <int KIND>
__global__ void __launch_bounds__(256) k_label_faces(const bccfast::LatDesc D, const HalfShell H,
                                                     const uint8_t* __restrict__ cls, int32_t* lab, int* flag) {
  constexpr int m = TileGeom<KIND>::m;
  __shared__ unsigned long long s_seen[kSeenSlots];
  __shared__ signed char s_d[4 * 8 * 4];
  for (int i = threadIdx.x; i < kSeenSlots; i += blockDim.x) s_seen[i] = ~0ull;
  for (int i = threadIdx.x; i < 4 * 8 * 4; i += blockDim.x) s_d[i] = H.d[i >> 5][(i >> 2) & 7][i & 3];
  __syncthreads();
  int t0[3], ts[3];
  bccfast::tile_of_index(D, blockIdx.x, t0, ts);
  const bccfast::CellIndex ci(ts);
  const int ncell = ts[0] * ts[1] * ts[2];
  for (int c = threadIdx.x; c < ncell; c += blockDim.x) {
    int x, y, z;
    ci.at(c, x, y, z);
    if (x > 0 && x < ts[0] - 1 && y > 0 && y < ts[1] - 1 && z > 0 && z < ts[2] - 1) continue;
    const int gx = t0[0] + x, gy = t0[1] + y, gz = t0[2] + z;
    const long long cell = ((long long)gz * D.n[1] + gy) * D.n[0] + gx;
    for (int b = 0; b < m; b++) {
      const long long i = cell * m + b;
      const int ci_ = cls[i] & 1;
      for (int j = 0; j < H.n; j++) {
        const signed char* d = s_d + (b * 8 + j) * 4;
        const int nx = x + d[0], ny = y + d[1], nz = z + d[2];
        if ((unsigned)nx < (unsigned)ts[0] && (unsigned)ny < (unsigned)ts[1] && (unsigned)nz < (unsigned)ts[2]) continue;
        const long long t = (((long long)wrap_add(gz, d[2], D.n[2]) * D.n[1] + wrap_add(gy, d[1], D.n[1])) * D.n[0] +
                             wrap_add(gx, d[0], D.n[0])) * m + d[3];
        if ((cls[t] & 1) != ci_ || t == i) continue;
        const unsigned a = (unsigned)*(volatile int32_t*)(lab + i), e = (unsigned)*(volatile int32_t*)(lab + t);
        const unsigned long long pair = ((unsigned long long)a << 32) | e;
        const unsigned slot = (a * 2654435761u + e * 2246822519u) >> 21;
        if (atomicExch(&s_seen[slot], pair) != pair) unite(lab, (int)a, (int)e, flag);
      }
    }
    if (*(volatile int*)flag) return;
  }
}

// Shortens the paths of the tile roots (cls bit 1), which every other site
// points at.
__global__ void k_compress_roots(const uint8_t* __restrict__ cls, int32_t* lab, long long N, int* flag) {
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < N; i += (long long)gridDim.x * blockDim.x)
    if (cls[i] & 2) lab[i] = find_root(lab, (int)i, flag);
}

// Root without writing: every pointer read is an ancestor, so the walk ends
// at the root whatever other threads write meanwhile, as long as they write
// ancestors too.
__device__ __forceinline__ int find_root_ro(const int32_t* lab, int x, int* flag) {
  const volatile int32_t* p = lab;
  for (int it = 0; it < kFindLimit; it++) {
    const int px = p[x];
    if (px == x) return x;
    x = px;
  }
  atomicOr(flag, 1);
  return x;
}

// Labels to roots in two launches.  The first shortens the paths (halving)
// and points every site at its root; a concurrent halving step elsewhere can
// still overwrite such a final write with an intermediate ancestor.  The
// second walks without halving, so every write is a root and stays one, and
// counts the roots.
template <bool FINAL>
__global__ void k_compress(int32_t* lab, long long N, int* flag, unsigned long long* n_roots) {
  unsigned long long roots = 0;
  if (FINAL) {
    // four sites a thread: neighbouring sites mostly share the label they start
    // from (16.4M sites: 196 us, 287 with a walk per site)
    const long long nq = (N + 3) / 4;
    for (long long q = (long long)blockIdx.x * blockDim.x + threadIdx.x; q < nq; q += (long long)gridDim.x * blockDim.x) {
      int from = -1, r = 0;
#pragma unroll
      for (int j = 0; j < 4; j++) {
        const long long i = 4 * q + j;
        if (i >= N) break;
        const int l = *(volatile int32_t*)(lab + i);
        if (l != from) {
          from = l;
          r = find_root_ro(lab, l, flag);
        }
        if (l != r) lab[i] = r;
        roots += (r == (int)i);
      }
    }
    for (int o = 16; o > 0; o >>= 1) roots += __shfl_down_sync(0xffffffffu, roots, o);
    if ((threadIdx.x & 31) == 0 && roots) atomicAdd(n_roots, roots);
  } else {
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < N; i += (long long)gridDim.x * blockDim.x)
      lab[i] = find_root(lab, (int)i, flag);
  }
}

// size[label]++.  A warp takes one step per distinct label; counts go through a
// direct-mapped table of the CTA in shared memory, so that the label of a
// percolating cluster takes one global atomic per CTA instead of one per warp
// (16.4M sites: 51 us against 645).
constexpr int kSizeSlots = 1024;
__global__ void __launch_bounds__(256) k_sizes(const int32_t* lab, long long N, int32_t* size) {
  __shared__ int s_key[kSizeSlots];
  __shared__ int s_cnt[kSizeSlots];
  for (int i = threadIdx.x; i < kSizeSlots; i += blockDim.x) {
    s_key[i] = -1;
    s_cnt[i] = 0;
  }
  __syncthreads();
  for (long long i0 = (long long)blockIdx.x * blockDim.x; i0 < N; i0 += (long long)gridDim.x * blockDim.x) {
    const long long i = i0 + threadIdx.x;
    const bool ok = i < N;
    const int l = ok ? lab[i] : -1;
    const unsigned peers = __match_any_sync(0xffffffffu, l);
    if (ok && (threadIdx.x & 31) == __ffs(peers) - 1) {
      const int slot = (int)(((unsigned)l * 2654435761u) >> 22);
      int key = *(volatile int*)&s_key[slot];
      if (key == -1) {
        key = atomicCAS(&s_key[slot], -1, l);
        if (key == -1) key = l;
      }
      if (key == l) atomicAdd(&s_cnt[slot], __popc(peers));
      else atomicAdd(&size[l], __popc(peers));
    }
  }
  __syncthreads();
  for (int i = threadIdx.x; i < kSizeSlots; i += blockDim.x)
    if (s_key[i] >= 0 && s_cnt[i]) atomicAdd(&size[s_key[i]], s_cnt[i]);
}

// Labels and sizes of the clusters of at least min_size sites (the first cap of
// them, in no order) and their number.
__global__ void k_select(const int32_t* size, long long N, long long min_size, int32_t* out, int32_t* out_size,
                         long long cap, unsigned long long* count) {
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < N; i += (long long)gridDim.x * blockDim.x) {
    const int n = size[i];
    if (n > 0 && n >= min_size) {
      const unsigned long long k = atomicAdd(count, 1ull);
      if ((long long)k < cap) {
        out[k] = (int32_t)i;
        out_size[k] = n;
      }
    }
  }
}

__global__ void k_mark(const int32_t* roots, int n, int32_t* size) {
  const int j = blockIdx.x * blockDim.x + threadIdx.x;
  if (j < n) size[roots[j]] = -(j + 1);
}

// Species counts of the marked clusters: in shared memory when there are at most
// kSpeciesBins of them, else straight to global memory (16.4M sites, 64 clusters of
// five species: 79 us against 646 with an atomic of every warp).
constexpr int kSpeciesBins = 2048;
__global__ void __launch_bounds__(256) k_species(const int32_t* lab, const int32_t* size, const uint8_t* sites,
                                                 int storage, long long N, int M, int bins,
                                                 unsigned long long* counts) {
  __shared__ unsigned s_bin[kSpeciesBins];
  const bool local = bins <= kSpeciesBins;
  if (local)
    for (int i = threadIdx.x; i < bins; i += blockDim.x) s_bin[i] = 0;
  __syncthreads();
  for (long long i0 = (long long)blockIdx.x * blockDim.x; i0 < N; i0 += (long long)gridDim.x * blockDim.x) {
    const long long i = i0 + threadIdx.x;
    int key = -1;
    if (i < N) {
      const int v = size[lab[i]];
      if (v < 0) key = (-v - 1) * M + min(load_site(sites, i, storage), M - 1);
    }
    const unsigned peers = __match_any_sync(0xffffffffu, key);
    if (key >= 0 && (threadIdx.x & 31) == __ffs(peers) - 1) {
      if (local) atomicAdd(&s_bin[key], __popc(peers));  // < 2^31 sites in all
      else atomicAdd(&counts[key], (unsigned long long)__popc(peers));
    }
  }
  __syncthreads();
  if (local)
    for (int i = threadIdx.x; i < bins; i += blockDim.x)
      if (s_bin[i]) atomicAdd(&counts[i], (unsigned long long)s_bin[i]);
}

int grid_for(long long work) {
  int dev = 0, nsm = 0;
  check_cuda(cudaGetDevice(&dev), "cudaGetDevice");
  check_cuda(cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev), "SM count");
  return (int)std::max<long long>(1, std::min<long long>((work + 255) / 256, (long long)nsm * 16));
}

void setup_params(const smcx_lattice* hd, SweepParams& P) {
  memset(&P, 0, sizeof(P));
  P.sites = hd->d_sites;
  P.M = hd->M;
  P.storage = hd->storage;
  for (int a = 0; a < 3; a++) P.n[a] = hd->n[a];
  fill_offsets_global(hd, P);
}

void need_epi(const smcx_lattice* hd) {
  if (!hd->have_epi) fail(SMCX_E_NO_EPI, "smcx_set_epi first");
  // |2 E_i| <= sum_k z_k max |V_k|
  long long bound = 0;
  const int M = hd->M;
  for (int k = 0; k < hd->shells.K; k++) {
    long long vmax = 0;
    for (int i = 0; i < M * M; i++) vmax = std::max(vmax, std::llabs((long long)hd->V[k * M * M + i]));
    bound += vmax * hd->shells.z[k];
    if (!hd->Wq.empty()) {
      long long wmax = 0;
      for (int p = 0; p < M; p++) wmax = std::max(wmax, std::llabs((long long)hd->Wq[k * M + p]));
      bound += 2 * wmax * hd->shells.z[k] * hd->shells.z[k];
    }
  }
  if (bound > 2147483647ll) fail(SMCX_E_RANGE, "local energies do not fit int32 for this EPI table");
}

// The tile kernels: FCC, or BCC with at most four species, |V| < 2^23, edges of
// two cells at least (the staging wraps a coordinate once).
bool tiles_usable(const smcx_lattice* hd) {
  if (hd->kernel_choice == SMCX_KERNEL_GENERIC || hd->M > (hd->kind == kBCC ? 4 : kMaxSweepM)) return false;
  if (reinterpret_cast<uintptr_t>(hd->d_sites) % 4 != 0) return false;
  for (int a = 0; a < 3; a++)
    if (hd->n[a] < 2) return false;
  for (int32_t v : hd->V)
    if (v >= (1 << 23) || v <= -(1 << 23)) return false;
  return true;
}

bccfast::LatDesc tile_desc(const smcx_lattice* hd) {
  bccfast::LatDesc D;
  memset(&D, 0, sizeof(D));
  D.sites = hd->d_sites;
  D.storage = hd->storage;
  D.M = hd->M;
  for (int a = 0; a < 3; a++) D.n[a] = hd->n[a];
  return D;
}

int tile_grid(long long tiles) {
  if (tiles > 0x7FFFFFFFll) fail(SMCX_E_UNSUPPORTED, "lattice too large for the tile kernels");
  return (int)tiles;
}

// Tiles for the labels, whose unions take longer than the staging: of at most `edge`
// cells, smaller ones (down to 4) until there are two per SM.
int label_tiles(bccfast::LatDesc& D, int edge) {
  int grid = 0;
  for (int e : {edge, 12, 10, 8, 6, 4}) {
    if (e > edge) continue;
    long long g = 1;
    for (int a = 0; a < 3; a++) g *= D.nt[a] = (D.n[a] + e - 1) / e;
    grid = tile_grid(g);
    if (g >= 2 * kSMs) break;
  }
  return grid;
}

LocalTab local_tab(const smcx_lattice* hd) {
  LocalTab T;
  memset(&T, 0, sizeof(T));
  const int K = hd->shells.K, M = hd->M;
  for (int k = 0; k < K; k++)
    for (int p = 0; p < M; p++) {
      for (int c = 0; c < M; c++) {
        const uint32_t v = (uint32_t)hd->V[((size_t)k * M + p) * M + c];
        const int w = hd->kind == kBCC ? 0 : c & 1, sh = 8 * (hd->kind == kBCC ? c : c >> 1);
        for (int j = 0; j < 3; j++) T.P[j][k][p][w] |= ((v >> (8 * j)) & 0xFFu) << sh;
      }
      if (!hd->Wq.empty()) T.W[k][p] = hd->Wq[(size_t)k * M + p];
    }
  return T;
}

template <int KIND>
void launch_local_tiles(smcx_lattice* hd, int32_t* e2) {
  bccfast::LatDesc D = tile_desc(hd);
  const int grid = tile_grid(bccfast::reduction_tiles(D.n, TileGeom<KIND>::kEdge, D.nt));
  const LocalTab T = local_tab(hd);
  const size_t smem = TileGeom<KIND>::kBoxBytes;
  const int qsro = hd->Wq.empty() ? 0 : 1;
  auto go = [&](auto kern) {
    check_cuda(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem), "smem attr");
    kern<<<grid, 256, smem, hd->stream>>>(D, T, qsro, e2);
  };
  const int K = hd->shells.K;
  if (K == 1) go(k_local_tile<KIND, 1>);
  else if (K == 2) go(k_local_tile<KIND, 2>);
  else if (K == 3) go(k_local_tile<KIND, 3>);
  else if constexpr (KIND == kBCC) go(k_local_tile<KIND, 4>);
  check_cuda(cudaGetLastError(), "tiled local energy launch");
}

template <int KIND>
void launch_label_tiles(smcx_lattice* hd, long long thr2, const HalfShell& H, uint8_t* cls, int32_t* lab) {
  using G = TileGeom<KIND>;
  bccfast::LatDesc D = tile_desc(hd);
  const int grid = label_tiles(D, G::kLabelEdge);
  const LocalTab T = local_tab(hd);
  const int sites = G::kLabelEdge * G::kLabelEdge * G::kLabelEdge * G::m;
  const size_t smem = (G::kBoxBytes + 15) / 16 * 16 + (size_t)sites * 5;
  const int qsro = hd->Wq.empty() ? 0 : 1;
  auto go = [&](auto kern) {
    check_cuda(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem), "smem attr");
    kern<<<grid, 256, smem, hd->stream>>>(D, T, qsro, thr2, H, cls, lab, hd->d_flag);
  };
  const int K = hd->shells.K;
  if (K == 1) go(k_label_tile<KIND, 1>);
  else if (K == 2) go(k_label_tile<KIND, 2>);
  else if (K == 3) go(k_label_tile<KIND, 3>);
  else if constexpr (KIND == kBCC) go(k_label_tile<KIND, 4>);
  k_label_faces<KIND><<<grid, 256, 0, hd->stream>>>(D, H, cls, lab, hd->d_flag);
  check_cuda(cudaGetLastError(), "tile label launches");
}

void launch_local_energy(smcx_lattice* hd, int32_t* e2, uint8_t* cls, long long thr2) {
  need_epi(hd);
  // int8 stores of 14 neighbours at most: a gather from the caches is done before a tile is
  // staged while the lattice is small (BCC, 2 shells: 24^3 and 32^3 cells 6.2 us against
  // 8.2 in tiles, 36^3 8.2 in both)
  const bool gather = hd->kind == kBCC && hd->shells.K <= 2 && hd->storage == SMCX_INT8 && hd->N <= 65536;
  if (e2 && !cls && !gather && tiles_usable(hd)) {
    if (hd->kind == kBCC) launch_local_tiles<kBCC>(hd, e2);
    else launch_local_tiles<kFCC>(hd, e2);
    return;
  }
  SweepParams P;
  setup_params(hd, P);
  // the plain V table sits after W[a][b][k][c] and X[a][b] in the device EPI table
  const int32_t* dV = hd->d_wtab + (size_t)hd->M * hd->M * hd->shells.K * hd->M + hd->M * hd->M;
  QsroWeights QW;
  memset(&QW, 0, sizeof(QW));
  QW.on = hd->Wq.empty() ? 0 : 1;
  for (size_t i = 0; i < hd->Wq.size(); i++) QW.w[i] = hd->Wq[i];
  const long long ncell = (long long)hd->n[0] * hd->n[1] * hd->n[2];
  const int grid = grid_for(ncell);
  const int K = hd->shells.K;
  auto go = [&](auto kern) { kern<<<grid, 256, 0, hd->stream>>>(P, dV, QW, e2, cls, thr2); };
  if (hd->kind == kBCC) {
    switch (K) {
      case 1: go(k_local_energy2<kBCC, 1>); break;
      case 2: go(k_local_energy2<kBCC, 2>); break;
      case 3: go(k_local_energy2<kBCC, 3>); break;
      default: go(k_local_energy2<kBCC, 4>); break;
    }
  } else {
    switch (K) {
      case 1: go(k_local_energy2<kFCC, 1>); break;
      case 2: go(k_local_energy2<kFCC, 2>); break;
      default: go(k_local_energy2<kFCC, 3>); break;
    }
  }
  check_cuda(cudaGetLastError(), "local energy launch");
}

HalfShell half_shell(const smcx_lattice* hd) {
  HalfShell H;
  memset(&H, 0, sizeof(H));
  const Shells& S = hd->shells;
  int n = 0;
  for (int j = 0; j < S.z[0]; j++) {
    const int* v = S.v[j];
    const bool half = v[0] > 0 || (v[0] == 0 && (v[1] > 0 || (v[1] == 0 && v[2] > 0)));
    if (!half) continue;
    for (int b = 0; b < hd->m; b++) {
      int B[3], d[3], r[3];
      basis_of(hd->kind, b, B);
      for (int a = 0; a < 3; a++) {
        const int p = B[a] + v[a];
        d[a] = (p >= 0) ? p / 2 : -((-p + 1) / 2);
        r[a] = p - 2 * d[a];
      }
      H.d[b][n][0] = (signed char)d[0];
      H.d[b][n][1] = (signed char)d[1];
      H.d[b][n][2] = (signed char)d[2];
      H.d[b][n][3] = (signed char)basis_index(hd->kind, r[0], r[1], r[2]);
    }
    n++;
  }
  H.n = n;
  return H;
}

// Device scratch of one call: the handle keeps up to kKeepBytes of it from call to
// call (an allocation and its release cost more than the kernels on a lattice of
// 16M sites); larger requests are allocated and released with the call.  All work
// on it is ordered on the handle's stream.
constexpr size_t kKeepBytes = (size_t)256 << 20;
struct Scratch {
  uint8_t* p = nullptr;
  uint8_t* own = nullptr;
  Scratch(smcx_lattice* hd, size_t bytes) {
    if (bytes > kKeepBytes) {
      check_cuda(cudaMalloc(&own, bytes), "cluster scratch");
      p = own;
      return;
    }
    if (hd->scratch_bytes < bytes) {
      cudaFree(hd->d_scratch);
      hd->d_scratch = nullptr;
      hd->scratch_bytes = 0;
      check_cuda(cudaMalloc(&hd->d_scratch, bytes), "cluster scratch");
      hd->scratch_bytes = bytes;
    }
    p = hd->d_scratch;
  }
  ~Scratch() { cudaFree(own); }
  Scratch(const Scratch&) = delete;
  Scratch& operator=(const Scratch&) = delete;
};
size_t align16(size_t b) { return (b + 15) & ~(size_t)15; }

}  // namespace

void local_energy_device(smcx_lattice* hd, int32_t* d_e2) { launch_local_energy(hd, d_e2, nullptr, 0); }

void clusters_device(smcx_lattice* hd, long long thr2, int32_t* d_lab, int64_t* n_clusters) {
  if (hd->N > 2147483647ll) fail(SMCX_E_RANGE, "cluster labels are int32: at most 2^31 - 1 sites");
  need_epi(hd);
  const size_t cls_bytes = align16((size_t)hd->N);
  Scratch scr(hd, cls_bytes + sizeof(unsigned long long));
  uint8_t* cls = scr.p;
  unsigned long long* roots = reinterpret_cast<unsigned long long*>(scr.p + cls_bytes);
  const int grid = grid_for(hd->N);
  check_cuda(cudaMemsetAsync(hd->d_flag, 0, sizeof(int), hd->stream), "clear flag");
  check_cuda(cudaMemsetAsync(roots, 0, sizeof(unsigned long long), hd->stream), "clear root count");
  const HalfShell H = half_shell(hd);
  if (tiles_usable(hd)) {
    if (hd->kind == kBCC) launch_label_tiles<kBCC>(hd, thr2, H, cls, d_lab);
    else launch_label_tiles<kFCC>(hd, thr2, H, cls, d_lab);
    k_compress_roots<<<grid, 256, 0, hd->stream>>>(cls, d_lab, hd->N, hd->d_flag);
  } else {
    launch_local_energy(hd, nullptr, cls, thr2);
    k_label_init<<<grid, 256, 0, hd->stream>>>(d_lab, hd->N);
    SweepParams P;
    setup_params(hd, P);
    const long long ncell = (long long)hd->n[0] * hd->n[1] * hd->n[2];
    if (hd->kind == kBCC)
      k_hook<kBCC><<<grid_for(ncell), 256, 0, hd->stream>>>(P, H, cls, d_lab, hd->d_flag);
    else
      k_hook<kFCC><<<grid_for(ncell), 256, 0, hd->stream>>>(P, H, cls, d_lab, hd->d_flag);
    k_compress<false><<<grid, 256, 0, hd->stream>>>(d_lab, hd->N, hd->d_flag, roots);
  }
  k_compress<true><<<grid, 256, 0, hd->stream>>>(d_lab, hd->N, hd->d_flag, roots);
  check_cuda(cudaGetLastError(), "cluster launches");
  int flag = 0;
  unsigned long long nr = 0;
  check_cuda(cudaMemcpyAsync(&flag, hd->d_flag, sizeof(int), cudaMemcpyDeviceToHost, hd->stream), "flag download");
  check_cuda(cudaMemcpyAsync(&nr, roots, sizeof(nr), cudaMemcpyDeviceToHost, hd->stream), "root count download");
  check_cuda(cudaStreamSynchronize(hd->stream), "cluster sync");
  if (flag) fail(SMCX_E_TIMEOUT, "union-find exceeded its iteration limit");
  if (n_clusters) *n_clusters = (int64_t)nr;
}

void cluster_summary_device(smcx_lattice* hd, const int32_t* d_lab, long long min_size, int max_out, int64_t* roots,
                            int64_t* sizes, int64_t* counts, int* n_out) {
  if (hd->N > 2147483647ll) fail(SMCX_E_RANGE, "cluster labels are int32: at most 2^31 - 1 sites");
  const long long N = hd->N;
  const int grid = grid_for(N), M = hd->M;
  // sizes [N], the list of large clusters and their sizes (N / min_size at most; up to
  // kList entries, more in a second pass) or, in its place afterwards, the marks and
  // counts of the ones returned, the counter.  A handle's first call pays for the
  // allocation: 165,168 sites, min_size 8, labels and summary 324 us, 489 with a list
  // of N entries.
  constexpr long long kList = 1 << 20;
  const long long cap0 = std::min(N / std::max(1ll, min_size), kList);
  const size_t size_bytes = align16((size_t)N * 4), list_bytes = align16((size_t)cap0 * 4);
  auto mark_bytes = [&](long long n) { return align16((size_t)n * 4) + (size_t)n * M * sizeof(unsigned long long); };
  const size_t most_marks = counts ? mark_bytes(std::min<long long>(cap0, std::max(0, max_out))) : 0;
  const size_t room = std::max(2 * list_bytes, align16(std::min(most_marks, 8 * (size_t)kList)));
  Scratch scr(hd, size_bytes + room + 16);
  int32_t* size = reinterpret_cast<int32_t*>(scr.p);
  int32_t* list = reinterpret_cast<int32_t*>(scr.p + size_bytes);
  int32_t* lsize = reinterpret_cast<int32_t*>(scr.p + size_bytes + list_bytes);
  unsigned long long* cnt = reinterpret_cast<unsigned long long*>(scr.p + size_bytes + room);
  check_cuda(cudaMemsetAsync(size, 0, (size_t)N * sizeof(int32_t), hd->stream), "clear sizes");
  check_cuda(cudaMemsetAsync(cnt, 0, sizeof(unsigned long long), hd->stream), "clear count");
  k_sizes<<<grid, 256, 0, hd->stream>>>(d_lab, N, size);
  k_select<<<grid, 256, 0, hd->stream>>>(size, N, std::max(1ll, min_size), list, lsize, cap0, cnt);
  check_cuda(cudaGetLastError(), "summary launches");
  unsigned long long n_big = 0;
  check_cuda(cudaMemcpyAsync(&n_big, cnt, sizeof(n_big), cudaMemcpyDeviceToHost, hd->stream), "count download");
  check_cuda(cudaStreamSynchronize(hd->stream), "summary sync");
  if (n_big > (1ull << 26)) fail(SMCX_E_RANGE, "more than 2^26 clusters of min_size sites: raise min_size");
  struct More {
    int32_t* p = nullptr;
    ~More() { cudaFree(p); }
  } more;
  if ((long long)n_big > cap0) {
    check_cuda(cudaMalloc(&more.p, (size_t)n_big * 8), "cluster list");
    list = more.p;
    lsize = more.p + n_big;
    check_cuda(cudaMemsetAsync(cnt, 0, sizeof(unsigned long long), hd->stream), "clear count");
    k_select<<<grid, 256, 0, hd->stream>>>(size, N, std::max(1ll, min_size), list, lsize, (long long)n_big, cnt);
  }
  std::vector<int32_t> r(n_big), s(n_big);
  if (n_big) {
    check_cuda(cudaMemcpyAsync(r.data(), list, n_big * sizeof(int32_t), cudaMemcpyDeviceToHost, hd->stream),
               "list download");
    check_cuda(cudaMemcpyAsync(s.data(), lsize, n_big * sizeof(int32_t), cudaMemcpyDeviceToHost, hd->stream),
               "size download");
  }
  check_cuda(cudaStreamSynchronize(hd->stream), "summary sync");
  // the n largest (ties: smaller label first)
  const int n = (int)std::min<unsigned long long>(n_big, (unsigned long long)std::max(0, max_out));
  std::vector<uint32_t> order(n_big);
  for (size_t j = 0; j < n_big; j++) order[j] = (uint32_t)j;
  std::partial_sort(order.begin(), order.begin() + n, order.end(),
                    [&](uint32_t a, uint32_t b) { return s[a] != s[b] ? s[a] > s[b] : r[a] < r[b]; });
  std::vector<int32_t> top(n);
  for (int j = 0; j < n; j++) {
    top[j] = r[order[j]];
    roots[j] = top[j];
    sizes[j] = s[order[j]];
  }
  *n_out = n;
  if (n == 0 || !counts) return;
  // marks and counts of the listed clusters, in the list's place when they fit
  const size_t top_bytes = align16((size_t)n * 4), count_bytes = (size_t)n * M * sizeof(unsigned long long);
  More marks;
  uint8_t* mp = scr.p + size_bytes;
  if (mark_bytes(n) > room) {
    check_cuda(cudaMalloc(&marks.p, mark_bytes(n)), "cluster marks");
    mp = reinterpret_cast<uint8_t*>(marks.p);
  }
  int32_t* d_top = reinterpret_cast<int32_t*>(mp);
  unsigned long long* d_counts = reinterpret_cast<unsigned long long*>(mp + top_bytes);
  check_cuda(cudaMemcpyAsync(d_top, top.data(), n * sizeof(int32_t), cudaMemcpyHostToDevice, hd->stream), "top upload");
  check_cuda(cudaMemsetAsync(d_counts, 0, count_bytes, hd->stream), "clear counts");
  k_mark<<<(n + 255) / 256, 256, 0, hd->stream>>>(d_top, n, size);
  const long long bins = (long long)n * M;
  k_species<<<grid, 256, 0, hd->stream>>>(d_lab, size, hd->d_sites, hd->storage, N, M,
                                          (int)std::min<long long>(bins, kSpeciesBins + 1), d_counts);
  check_cuda(cudaGetLastError(), "summary launches");
  std::vector<unsigned long long> h((size_t)n * M);
  check_cuda(cudaMemcpyAsync(h.data(), d_counts, h.size() * sizeof(unsigned long long), cudaMemcpyDeviceToHost,
                             hd->stream),
             "counts download");
  check_cuda(cudaStreamSynchronize(hd->stream), "summary sync");
  for (size_t j = 0; j < h.size(); j++) counts[j] = (int64_t)h[j];
}

}  // namespace smcx

using namespace smcx;

extern "C" {

int smcx_local_energy(smcx_lattice* h, int32_t* d_e2) {
  return guarded_call([&] {
    if (!h || !d_e2) fail(SMCX_E_INVALID_ARG, "NULL argument");
    local_energy_device(h, d_e2);
  });
}

int smcx_clusters(smcx_lattice* h, int64_t thr2, int32_t* d_labels, int64_t* n_clusters) {
  return guarded_call([&] {
    if (!h || !d_labels) fail(SMCX_E_INVALID_ARG, "NULL argument");
    clusters_device(h, thr2, d_labels, n_clusters);
  });
}

int smcx_cluster_summary(smcx_lattice* h, const int32_t* d_labels, int64_t min_size, int max_out, int64_t* roots,
                         int64_t* sizes, int64_t* counts, int* n_out) {
  return guarded_call([&] {
    if (!h || !d_labels || !n_out || (max_out > 0 && (!roots || !sizes)))
      fail(SMCX_E_INVALID_ARG, "NULL argument");
    if (max_out < 0) fail(SMCX_E_INVALID_ARG, "max_out must be >= 0");
    cluster_summary_device(h, d_labels, min_size, max_out, roots, sizes, counts, n_out);
  });
}

}  // extern "C"
