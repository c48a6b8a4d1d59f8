// decide_kernel: Broadcast half of the decision table for short candidate lists (lines.cuh).
#include "direct.cuh"
#include "lines.cuh"

namespace plogp {

template <bool STAGED>
__global__ void __launch_bounds__(STAGED ? kLineThreads : kDecThreads, STAGED ? 2 : 4) decide_kernel(const DecideParams p)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    lines_block<false, STAGED>(p, blockIdx.x, smem_raw);
    last_block_waits(threadIdx.x);
}

__global__ void __launch_bounds__(kDecThreads, 8) decide_direct_kernel(const DecideParams p)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    direct_block<false>(p, blockIdx.x, smem_raw);
    last_block_waits(threadIdx.x);
}

cudaError_t launch_decide(const DecideParams &p, bool overlap, cudaStream_t st)
{
    const long long blocks = static_cast<long long>(p.n_mgroups) * p.n_ptiles * p.n_tables_launch;
    if (blocks <= 0 || blocks > 0x7FFFFFFFLL) return cudaErrorInvalidConfiguration;
    return launch(p.direct ? decide_direct_kernel : p.staged ? decide_kernel<true> : decide_kernel<false>, static_cast<unsigned>(blocks), 1, static_cast<unsigned>(p.threads), lines_smem_bytes(p), st, overlap, p);
}

}  // namespace plogp
