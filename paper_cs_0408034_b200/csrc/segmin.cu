// segmin_kernel: the segment-size search of Section 3.1 for plogp_predict on short candidate lists: for each segmented
// strategy of Table 1 (ids 2, 5, 9) on its own, the minimum of the model over the candidate segment sizes and the smallest
// size that attains it (lines.cuh).
#include "direct.cuh"
#include "lines.cuh"

namespace plogp {

template <bool STAGED>
__global__ void __launch_bounds__(STAGED ? kLineThreads : kDecThreads, STAGED ? 2 : 4) segmin_kernel(const SegminParams p)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    lines_block<true, STAGED>(p, blockIdx.x, smem_raw);
    last_block_waits(threadIdx.x);
}

__global__ void __launch_bounds__(kDecThreads, 8) segmin_direct_kernel(const SegminParams p)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    direct_block<true>(p, blockIdx.x, smem_raw);
    last_block_waits(threadIdx.x);
}

cudaError_t launch_segmin(const SegminParams &p, bool overlap, cudaStream_t st)
{
    const long long blocks = static_cast<long long>(p.n_mgroups) * p.n_ptiles * p.n_tables_launch;
    if (blocks <= 0 || blocks > 0x7FFFFFFFLL) return cudaErrorInvalidConfiguration;
    return launch(p.direct ? segmin_direct_kernel : p.staged ? segmin_kernel<true> : segmin_kernel<false>, static_cast<unsigned>(blocks), 1, static_cast<unsigned>(p.threads), lines_smem_bytes(p), st, overlap, p);
}

}  // namespace plogp
