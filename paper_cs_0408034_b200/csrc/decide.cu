// decide_kernel: Broadcast half of the decision table for short candidate lists (decide.cuh).
//
// Bound by issue (0.6 of the slots at 16 warps per SM, more with 20), not by memory (17 % of the DRAM rate): 4096 tables,
// P = 2..512, 128 message sizes, 32 candidates take 2.05 ms at five CTAs per SM, 2.17 at four (3.58 with FP64 cells).  A third
// of it are the bounds; lists, pilots, pairs, exact rows and the write-out, once per message size, are the rest.
#include "decide.cuh"

namespace plogp {

// B: CTAs per SM, 4 with 128 registers or 5 with 96 (no spills either way; the host says when).
template <bool ENV, int R, int B>
__global__ void __launch_bounds__(kDecThreads, B) decide_kernel(const DecideParams p)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    decide_block<ENV, R>(p, blockIdx.x, smem_raw);
    last_block_waits(threadIdx.x);
}

size_t decide_smem_bytes(const DecideParams &p) { return decide::dec_layout(p.gaps ? 0 : p.T.npad, p.G.n_s, p.n_pairs, p.tiles * 32 * p.rows, p.mg, nullptr, nullptr); }

cudaError_t launch_decide(const DecideParams &p, bool overlap, cudaStream_t st)
{
    const size_t smem = decide_smem_bytes(p);
    const long long blocks = static_cast<long long>(p.n_mgroups) * p.n_ptiles * p.n_tables_launch;
    if (blocks <= 0 || blocks > 0x7FFFFFFFLL) return cudaErrorInvalidConfiguration;
    const auto kernel = p.rows != 8 ? (p.envelope ? decide_kernel<true, 4, 4> : decide_kernel<false, 4, 4>)
                        : p.ctas_per_sm == 5 ? (p.envelope ? decide_kernel<true, 8, 5> : decide_kernel<false, 8, 5>)
                                             : (p.envelope ? decide_kernel<true, 8, 4> : decide_kernel<false, 8, 4>);
    return launch(kernel, static_cast<unsigned>(blocks), 1, kDecThreads, smem, st, overlap, p);
}

}  // namespace plogp
