// BCC sweeps with several lanes per trial (smcx_bcc_group.cuh): single lattices (one
// launch per tile colour, one CTA per tile of that colour) and batches.
#include "smcx_batch_body.cuh"

namespace smcx {

template <int LN, int K, int NW, int PL>
static void launch_group(smcx_lattice* hd, bccfast::LatDesc& D, const bccfast::Planes& Q, int64_t n_sweeps,
                         int n_colours) {
  auto kern = bccfast::k_bcc_group_sweep<LN, K, NW, PL>;
  const int smem = (int)bccfast::smem_bytes(D.nA);
  check_cuda(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, smem), "bcc group smem attribute");
  const int grid = (D.nt[0] / 2) * (D.nt[1] / 2) * (D.nt[2] / 2), threads = bccfast::group_threads(D.NQ);
  const unsigned long long first = D.sweep;
  for (int64_t s = 0; s < n_sweeps; s++) {
    D.sweep = first + (unsigned long long)s;
    for (int tc = 0; tc < n_colours; tc++) kern<<<grid, threads, smem, hd->stream>>>(D, Q, tc);
  }
  check_cuda(cudaGetLastError(), "bcc group launch");
}

template <int LN>
static void sweep_lanes(smcx_lattice* hd, bccfast::LatDesc& D, const bccfast::Planes& Q, int nw, int pl, int64_t n,
                        int nc) {
  const int K = hd->shells.K;
  if (K == 4) {
    if (nw == 1) return pl == 2 ? launch_group<LN, 4, 1, 2>(hd, D, Q, n, nc) : launch_group<LN, 4, 1, 3>(hd, D, Q, n, nc);
    return pl == 2 ? launch_group<LN, 4, 2, 2>(hd, D, Q, n, nc) : launch_group<LN, 4, 2, 3>(hd, D, Q, n, nc);
  }
  // fewer shells: the variants of the one-lane sweep
  const bool small = nw == 1 && pl == 2;
  if (K == 3) return small ? launch_group<LN, 3, 1, 2>(hd, D, Q, n, nc) : launch_group<LN, 3, 2, 3>(hd, D, Q, n, nc);
  // (one shell alone has another halo and never comes here)
  return small ? launch_group<LN, 2, 1, 2>(hd, D, Q, n, nc) : launch_group<LN, 2, 2, 3>(hd, D, Q, n, nc);
}

// nw counter words (1: M <= 4), pl byte planes of V.
void sweep_bcc_group(smcx_lattice* hd, bccfast::LatDesc& D, const bccfast::Planes& Q, int nw, int pl, int64_t n,
                     int nc) {
  if (bccfast::group_lanes(D.NQ) == 4) sweep_lanes<4>(hd, D, Q, nw, pl, n, nc);
  else sweep_lanes<2>(hd, D, Q, nw, pl, n, nc);
}

bccfast::BatchKernelFn batch_group_kernel(int nw, int pl) {
  using namespace bccfast;
  if (nw == 1) return pl == 2 ? k_bcc_batch_group<4, 4, 1, 2> : k_bcc_batch_group<4, 4, 1, 3>;
  return pl == 2 ? k_bcc_batch_group<4, 4, 2, 2> : k_bcc_batch_group<4, 4, 2, 3>;
}

}  // namespace smcx
