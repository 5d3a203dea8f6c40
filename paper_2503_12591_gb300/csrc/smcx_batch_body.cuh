// Persistent batched sweep body: every replica, every sweep, every tile
// colour in one cooperative launch (temperature parallelism, Supplementary
// "Parallelization opportunities").  Included by smcx_batch.cu (per-trial
// directions) and smcx_sweep_bcc_dir.cu (shared-direction proposals, whose
// trial body and constant-memory offset table live in that translation unit).
#pragma once

#include "smcx_bcc_group.cuh"

namespace smcx {
namespace bccfast {

__device__ __forceinline__ unsigned long long global_ns() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %globaltimer;" : "=l"(t));
  return t;
}

// Memory of one launch: the counter the CTAs draw from, and one counter per replica of
// the tile passes done (all zero before the launch).
struct Progress {
  unsigned long long drawn;
  unsigned long long done[1];  // [replicas]
};
__host__ __device__ constexpr size_t progress_bytes(size_t replicas) { return 8 * (1 + replicas); }

// The tile passes of a launch form one list: for every sweep and colour the pooled
// (replica, tile) items, largest tiles first.  CTAs take its entries in order, the
// first by their own index, the rest from a counter as they get done.  A pass waits
// only for its own replica: until all tiles of that replica's previous colour are done.
// They stand earlier in the list, so some CTA is at work on them or done, and the
// first unfinished entry never waits.  A wait lasts at most `timeout_ns`; a CTA that
// gives up sets the status, and all others stop when they see it.
// Thread 0 publishes, draws and waits: a CTA barrier and a fence come between the
// pass's writes and the counter, and between the counter and the next pass's reads.
//
// 64 replicas of 24 to 96 cells (L = 3, tiles of 12 to 18 cells, 4 sweeps) took 5.66 ms
// with CTA b on the items b, b + G, ... of a colour and a grid barrier after it: the
// last items of every colour left most SMs idle.  Drawn from a counter 4.55 ms; with
// the next colour begun before this one ends 4.00 ms.
// KEEP: with in_place set (and a CTA per item) every CTA keeps its item, nothing is drawn.
template <bool KEEP, class Pass>
__device__ __forceinline__ void batch_loop(const LatDesc* __restrict__ descs, const int2* __restrict__ items,
                                           int n_items, int n_sweeps, Progress* pr, int* status,
                                           long long timeout_ns, int skip_cta, int in_place, Pass pass) {
  __shared__ int s_item, s_epoch;  // item < 0: no more work
  unsigned long long base = 0;     // thread 0: list position of item 0 of this colour
  int item = blockIdx.x, epoch = 0;  // epoch: colours since the launch began
  const int n_epochs = 8 * n_sweeps;
  for (;;) {
    const int2 it = items[item];
    const LatDesc D = descs[it.x];
    pass(D, epoch & 7, it.y, D.sweep + (unsigned long long)(epoch >> 3));
    __syncthreads();
    if ((int)blockIdx.x == skip_cta) return;
    if (threadIdx.x == 0) {
      __threadfence();
      atomicAdd(&pr->done[it.x], 1ull);
      auto draw = [&]() {
        const unsigned long long g = atomicAdd(&pr->drawn, 1ull) + gridDim.x;
        while (g - base >= (unsigned)n_items) {
          base += (unsigned)n_items;
          epoch++;
        }
        return (int)(g - base);
      };
      // `next` once its replica's previous colour is done, -1 if the launch stops
      auto wait = [&](int next) {
        const int r = items[next].x;
        const LatDesc& R = descs[r];
        const unsigned per_colour = (unsigned)((R.nt[0] / 2) * (R.nt[1] / 2) * (R.nt[2] / 2));
        const unsigned long long need = (unsigned long long)epoch * per_colour;
        const unsigned long long t0 = global_ns();
        while (*(volatile unsigned long long*)&pr->done[r] < need) {
          const bool late = (long long)(global_ns() - t0) > timeout_ns;
          if (late) atomicCAS(status, 0, SMCX_E_TIMEOUT);
          if (late || *((volatile int*)status) != 0) {
            next = -1;
            break;
          }
          __nanosleep(64);
        }
        __threadfence();
        return next;
      };
      int next = -1;
      if constexpr (KEEP) {
        // two paths to `next` before the test of the epoch: fewer spills than one
        if (in_place) {
          next = item;
          epoch++;
        } else {
          next = draw();
        }
        if (epoch >= n_epochs) next = -1;
        if (next >= 0) next = wait(next);
      } else {
        const int drawn = draw();
        if (epoch < n_epochs) next = wait(drawn);
      }
      s_item = next;
      s_epoch = epoch;
    }
    __syncthreads();
    item = s_item;
    epoch = s_epoch;
    if (item < 0) return;
  }
}

template <int K, int NW, int PL, int SLOTS, int PROP>
__device__ __forceinline__ void batch_body(const Planes& Q, const LatDesc* __restrict__ descs,
                                           const int2* __restrict__ items, int n_items, int n_sweeps, Progress* pr,
                                           int* status, long long timeout_ns, int skip_cta, int in_place, int max_nA) {
  extern __shared__ __align__(16) unsigned char smem[];
  __shared__ unsigned long long s_stat[3];
  uint32_t* sA = reinterpret_cast<uint32_t*>(smem + 2 * SUB);
  uint32_t* sB = sA + max_nA;
  uint8_t* s_dir = reinterpret_cast<uint8_t*>(sB + kNB);
  batch_loop<(NW > 1)>(descs, items, n_items, n_sweeps, pr, status, timeout_ns, skip_cta, in_place,
             [&](const LatDesc& D, int tc, int jt, unsigned long long sweep) {
               bcc_tile_pass<K, NW, PL, SLOTS, PROP>(D, Q, tc, jt, sweep, smem, sA, sB, s_dir, s_stat);
             });
}

// 128-thread CTAs (one or two link-cell slots per thread), and 256-thread
// CTAs for tiles of up to 256 slots (6^3 with link cells of 3): one slot per
// thread, so a tile's phases take half the sequential steps of two slots.
template <int K, int NW, int PL, int SLOTS, int PROP>
__global__ void __launch_bounds__(128, 6)
    k_bcc_batch(const Planes Q, const LatDesc* __restrict__ descs, const int2* __restrict__ items, int n_items,
                int n_sweeps, Progress* pr, int* status, long long timeout_ns, int skip_cta, int in_place,
                int max_nA) {
  batch_body<K, NW, PL, SLOTS, PROP>(Q, descs, items, n_items, n_sweeps, pr, status, timeout_ns, skip_cta, in_place,
                             max_nA);
}
template <int K, int NW, int PL, int PROP>
__global__ void __launch_bounds__(256, 3)
    k_bcc_batch256(const Planes Q, const LatDesc* __restrict__ descs, const int2* __restrict__ items, int n_items,
                   int n_sweeps, Progress* pr, int* status, long long timeout_ns, int skip_cta, int in_place,
                   int max_nA) {
  batch_body<K, NW, PL, 1, PROP>(Q, descs, items, n_items, n_sweeps, pr, status, timeout_ns, skip_cta, in_place,
                             max_nA);
}

// Several lanes per trial (smcx_bcc_group.cuh), for few tiles of at most 3^3 slots.
template <int LN, int K, int NW, int PL>
__global__ void __launch_bounds__(kGroupThreads, 4)
    k_bcc_batch_group(const Planes Q, const LatDesc* __restrict__ descs, const int2* __restrict__ items, int n_items,
                      int n_sweeps, Progress* pr, int* status, long long timeout_ns, int skip_cta, int in_place,
                      int max_nA) {
  extern __shared__ __align__(16) unsigned char smem[];
  __shared__ __align__(16) GroupMem M;
  uint32_t* sA = reinterpret_cast<uint32_t*>(smem + 2 * SUB);
  batch_loop<false>(descs, items, n_items, n_sweeps, pr, status, timeout_ns, skip_cta, in_place,
             [&](const LatDesc& D, int tc, int jt, unsigned long long sweep) {
               group_pass<LN, K, NW, PL>(D, Q, tc, jt, sweep, smem, sA, sA + max_nA, M);
             });
}

using BatchKernelFn = void (*)(const Planes, const LatDesc*, const int2*, int, int, Progress*, int*, long long, int,
                               int, int);

}  // namespace bccfast

// The shared-direction batch kernel (4 shells, M <= 4, two byte planes, one
// link-cell slot per thread) for 128- or 256-thread CTAs.
bccfast::BatchKernelFn batch_dir_kernel(int threads);  // smcx_sweep_bcc_dir.cu
// Four lanes per trial (4 shells; nw counter words, pl byte planes).
bccfast::BatchKernelFn batch_group_kernel(int nw, int pl);  // smcx_sweep_bcc_group.cu

}  // namespace smcx
