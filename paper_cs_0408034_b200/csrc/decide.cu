// decide_kernel: Broadcast half of the decision table for short candidate lists (decide.cuh).
#include "decide.cuh"

namespace plogp {

template <bool ENV, int R>
__global__ void __launch_bounds__(kDecThreads, 4) decide_kernel(const DecideParams p)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    decide_block<ENV, R>(p, blockIdx.x, smem_raw);
    last_block_waits(threadIdx.x);
}

size_t decide_smem_bytes(const DecideParams &p) { return decide::dec_layout(p.T.npad, p.G.n_s, p.n_pairs, p.tiles * 32 * p.rows, p.mg, nullptr, nullptr); }

cudaError_t launch_decide(const DecideParams &p, bool overlap, cudaStream_t st)
{
    const size_t smem = decide_smem_bytes(p);
    const long long blocks = static_cast<long long>(p.n_mgroups) * p.n_ptiles * p.n_tables_launch;
    if (blocks <= 0 || blocks > 0x7FFFFFFFLL) return cudaErrorInvalidConfiguration;
    const auto kernel = p.rows == 8 ? (p.envelope ? decide_kernel<true, 8> : decide_kernel<false, 8>)
                                    : (p.envelope ? decide_kernel<true, 4> : decide_kernel<false, 4>);
    return launch(kernel, static_cast<unsigned>(blocks), 1, kDecThreads, smem, st, overlap, p);
}

}  // namespace plogp
