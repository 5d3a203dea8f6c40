// Ordered pair counts and the qSRO energy of an FCC lattice from shared-memory
// tiles (the FCC counterparts of smcx_reduce_bcc.cu).
//
// Same results as k_pair_counts (smcx_aux.cu) and k_qsro_energy
// (smcx_sweep_qsro.cu), which gather every neighbour from global memory and,
// for the counts, make one shared atomic per neighbour, which bounds them.  Here a
// CTA stages a tile of at most 15 cells with its 2-cell halo into the even-point
// box of the FCC sweep, where a neighbour is one shared load at a constant offset,
// and counts in registers: 14.5M sites of five species and three shells 221 us
// against 1013; energy under the qSRO model at 6.9M sites (counts and quadratic
// term) 0.22 ms against 1.18.
#include <algorithm>

#include "smcx_fcc_tile.cuh"
#include "smcx_tiles.cuh"

namespace smcx {

namespace fccfast {

// Half of a shell: the vectors whose first nonzero half-unit component is
// positive (one of each +v / -v pair).
__host__ __device__ constexpr bool half_vec(const FVec& v) {
  return v.x > 0 || (v.x == 0 && (v.y > 0 || (v.y == 0 && v.z > 0)));
}

// Pair counts, MP species at most.  The box holds 4 s, so that a neighbour of
// the half shell k adds 1 << (4 s) to one word of eight 4-bit counters (at most
// 12 neighbours of a half shell).  Every unordered pair is visited once: C[p][q]
// = U[p][q] + U[q][p] with U over the half shells.  A thread keeps U in 16-bit
// fields (word w of species p: counters w and w + 4); the 60 accumulators of
// five species and three shells and the 63 instructions of the 21 neighbours
// bound it by issue.  Branch-free adds and three CTAs per SM (two where the
// accumulators need the registers): 151 x 180 x 133 cells 221 -> 130 us,
// 120^3 cells 118 -> 73.
template <int K, int MP>
__global__ void __launch_bounds__(256, MP == 8 && K == 3 ? 2 : 3)
    k_fcc_pair_counts(const LatDesc D, unsigned long long* __restrict__ counts) {
  constexpr int NW = MP < 4 ? MP : 4;  // counter words: species w and w + 4
  extern __shared__ __align__(16) unsigned char smem[];
  __shared__ unsigned int hist[K * 64];
  uint8_t* box = smem;
  const int tid = threadIdx.x, nth = blockDim.x;
  int t0[3], ts[3];
  bccfast::tile_of_index(D, blockIdx.x, t0, ts);
  for (int i = tid; i < K * 64; i += nth) hist[i] = 0;
  stage_box<4>(D, box, t0, ts, tid & 31, tid >> 5, nth >> 5);
  __syncthreads();
  uint32_t acc[K][MP][NW];
#pragma unroll
  for (int k = 0; k < K; k++)
#pragma unroll
    for (int p = 0; p < MP; p++)
#pragma unroll
      for (int w = 0; w < NW; w++) acc[k][p][w] = 0;
  constexpr FTable T = make_fvecs();
  const bccfast::CellIndex ci(ts);
  const int ncell = ts[0] * ts[1] * ts[2];
  for (int c = tid; c < ncell; c += nth) {
    int xr, yr, zr;
    ci.at(c, xr, yr, zr);
    const int base = hoff(2 * (xr + H), 2 * (yr + H), 2 * (zr + H));
#pragma unroll 1
    for (int b = 0; b < 4; b++) {
      const int s = base + boff(b);
      const uint32_t p = ld_chk(box, s, BOX_BYTES, kDbgFccBox);
      uint32_t h[K];
#pragma unroll
      for (int k = 0; k < K; k++) h[k] = 0;
#pragma unroll
      for (int j = 0; j < T.n; j++)
        if (T.v[j].k < K && half_vec(T.v[j]))
          h[T.v[j].k] += 1u << ld_chk(box, s + hoff(T.v[j].x, T.v[j].y, T.v[j].z), BOX_BYTES, kDbgFccBox);
      uint32_t is_p[MP];
#pragma unroll
      for (int pp = 0; pp < MP; pp++) is_p[pp] = p == 4u * pp;
#pragma unroll
      for (int k = 0; k < K; k++)
#pragma unroll
        for (int w = 0; w < NW; w++) {
          const uint32_t x = (h[k] >> (4 * w)) & 0x000F000Fu;
#pragma unroll
          for (int pp = 0; pp < MP; pp++) bccfast::add_if(acc[k][pp][w], x, is_p[pp]);
        }
    }
  }
  // 16-bit fields: a thread has at most 14 cells x 4 sites x 12, a warp 32 of them
#pragma unroll
  for (int k = 0; k < K; k++)
#pragma unroll
    for (int p = 0; p < MP; p++)
#pragma unroll
      for (int w = 0; w < NW; w++) {
        const uint32_t v = __reduce_add_sync(0xffffffffu, acc[k][p][w]);
        if ((tid & 31) == 0) {
          atomicAdd(&hist[k * 64 + p * 8 + w], v & 0xFFFFu);
          atomicAdd(&hist[k * 64 + p * 8 + w + 4], v >> 16);
        }
      }
  __syncthreads();
  for (int i = tid; i < K * 64; i += nth) {
    const int k = i / 64, p = (i / 8) % 8, q = i % 8;
    if (p < D.M && q < D.M && hist[i]) {
      atomicAdd(&counts[(k * D.M + p) * D.M + q], (unsigned long long)hist[i]);
      atomicAdd(&counts[(k * D.M + q) * D.M + p], (unsigned long long)hist[i]);
    }
  }
}

// sum_i sum_k W[k][s_i] n_k(i)^2 added to *E; n_k counted over the whole shell.
struct QWeights {
  int32_t w[3][8];
};
template <int K>
__global__ void __launch_bounds__(256, 4) k_fcc_qsro_energy(const LatDesc D, const QWeights W, long long* __restrict__ E) {
  extern __shared__ __align__(16) unsigned char smem[];
  __shared__ int32_t s_w[K * 8];
  __shared__ long long part[8];
  uint8_t* box = smem;
  const int tid = threadIdx.x, nth = blockDim.x;
  int t0[3], ts[3];
  bccfast::tile_of_index(D, blockIdx.x, t0, ts);
  for (int i = tid; i < K * 8; i += nth) s_w[i] = W.w[i / 8][i % 8];
  stage_box<1>(D, box, t0, ts, tid & 31, tid >> 5, nth >> 5);
  __syncthreads();
  constexpr FTable T = make_fvecs();
  const bccfast::CellIndex ci(ts);
  const int ncell = ts[0] * ts[1] * ts[2];
  long long acc = 0;
  for (int c = tid; c < ncell; c += nth) {
    int xr, yr, zr;
    ci.at(c, xr, yr, zr);
    const int base = hoff(2 * (xr + H), 2 * (yr + H), 2 * (zr + H));
#pragma unroll 1
    for (int b = 0; b < 4; b++) {
      const int s = base + boff(b);
      const int p = ld_chk(box, s, BOX_BYTES, kDbgFccBox);
      int n[K];
#pragma unroll
      for (int k = 0; k < K; k++) n[k] = 0;
#pragma unroll
      for (int j = 0; j < T.n; j++)
        if (T.v[j].k < K)
          n[T.v[j].k] += ld_chk(box, s + hoff(T.v[j].x, T.v[j].y, T.v[j].z), BOX_BYTES, kDbgFccBox) == p;
#pragma unroll
      for (int k = 0; k < K; k++) acc += (long long)s_w[k * 8 + (p & 7)] * (n[k] * n[k]);
    }
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) acc += __shfl_down_sync(0xffffffffu, acc, o);
  if ((tid & 31) == 0) part[tid >> 5] = acc;
  __syncthreads();
  if (tid == 0) {
    long long t = 0;
    for (int w = 0; w < nth / 32; w++) t += part[w];
    atomicAdd(reinterpret_cast<unsigned long long*>(E), (unsigned long long)t);
  }
}

}  // namespace fccfast

// Tiles for a reduction over an FCC lattice of at most eight species: edges of 2
// cells at least (the staging wraps a coordinate once) and a store whose cells
// can be read as words.
bool fcc_reduce_usable(const smcx_lattice* hd, int nt[3]) {
  if (hd->kind != kFCC || hd->M > kMaxSweepM || !hd->have_epi || hd->shells.K > 3) return false;
  if (hd->kernel_choice == SMCX_KERNEL_GENERIC || reinterpret_cast<uintptr_t>(hd->d_sites) % 4 != 0) return false;
  for (int a = 0; a < 3; a++)
    if (hd->n[a] < 2) return false;
  return bccfast::reduction_tiles(hd->n, fccfast::TMAX, nt) < (1ll << 31);
}

static bccfast::LatDesc reduce_desc(const smcx_lattice* hd, const int nt[3]) {
  bccfast::LatDesc D;
  memset(&D, 0, sizeof(D));
  D.sites = hd->d_sites;
  D.storage = hd->storage;
  D.M = hd->M;
  for (int a = 0; a < 3; a++) {
    D.n[a] = hd->n[a];
    D.nt[a] = nt[a];
  }
  return D;
}

// Ordered pair counts added into hd->d_counts (cleared by the caller).
void pair_counts_fcc_tiled(smcx_lattice* hd, const int nt[3]) {
  const bccfast::LatDesc D = reduce_desc(hd, nt);
  const int grid = nt[0] * nt[1] * nt[2];
  auto go = [&](auto kern) {
    check_cuda(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, fccfast::BOX_BYTES), "smem attr");
    kern<<<grid, 256, fccfast::BOX_BYTES, hd->stream>>>(D, hd->d_counts);
  };
  const int K = hd->shells.K, M = hd->M;
  if (M <= 4) {
    if (K == 1) go(fccfast::k_fcc_pair_counts<1, 4>);
    else if (K == 2) go(fccfast::k_fcc_pair_counts<2, 4>);
    else go(fccfast::k_fcc_pair_counts<3, 4>);
  } else if (M == 5) {
    if (K == 1) go(fccfast::k_fcc_pair_counts<1, 5>);
    else if (K == 2) go(fccfast::k_fcc_pair_counts<2, 5>);
    else go(fccfast::k_fcc_pair_counts<3, 5>);
  } else {
    if (K == 1) go(fccfast::k_fcc_pair_counts<1, 8>);
    else if (K == 2) go(fccfast::k_fcc_pair_counts<2, 8>);
    else go(fccfast::k_fcc_pair_counts<3, 8>);
  }
  check_cuda(cudaGetLastError(), "tiled fcc pair-count launch");
}

// sum_i sum_k W[k][s_i] n_k(i)^2 added to hd->d_energy; false when the tiled
// path does not apply.
bool qsro_energy_fcc_tiled(smcx_lattice* hd) {
  int nt[3];
  if (!fcc_reduce_usable(hd, nt)) return false;
  const bccfast::LatDesc D = reduce_desc(hd, nt);
  const int grid = nt[0] * nt[1] * nt[2], K = hd->shells.K;
  fccfast::QWeights W;
  memset(&W, 0, sizeof(W));
  for (int k = 0; k < K; k++)
    for (int p = 0; p < hd->M; p++) W.w[k][p] = hd->Wq[(size_t)k * hd->M + p];
  auto go = [&](auto kern) {
    check_cuda(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, fccfast::BOX_BYTES), "smem attr");
    kern<<<grid, 256, fccfast::BOX_BYTES, hd->stream>>>(D, W, hd->d_energy);
  };
  if (K == 1) go(fccfast::k_fcc_qsro_energy<1>);
  else if (K == 2) go(fccfast::k_fcc_qsro_energy<2>);
  else go(fccfast::k_fcc_qsro_energy<3>);
  check_cuda(cudaGetLastError(), "tiled fcc qSRO energy launch");
  return true;
}

}  // namespace smcx
