// select_kernel: both halves of a decision table in one launch, for grids that the GPU holds in one go.  There a call is
// mostly launches: the first CTAs take the Broadcast half (lines.cuh), the others the Scatter half (scatter.cuh, with the
// Broadcast half's four warps per CTA).  One table, P = 2..50, 19 message sizes, 7 candidates: one launch less is 3 us of
// host time a call and 8.2 -> 6.2 us between calls on the GPU.
#include "lines.cuh"
#include "scatter.cuh"

namespace plogp {

template <bool CONTIG>
__global__ void __launch_bounds__(kDecThreads, 4) select_kernel(const SelectParams p)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    if (blockIdx.x < static_cast<unsigned>(p.n_decide)) {
        lines_block<false, false>(p.decide, blockIdx.x, smem_raw);
    } else {
        scatter_block<CONTIG ? kChainRun : kChainRange, false, 1, kDecWarps>(p.scatter, blockIdx.x - p.n_decide, smem_raw);
    }
}

cudaError_t launch_select(SelectParams &p, cudaStream_t st)
{
    const long long nd = static_cast<long long>(p.decide.n_mgroups) * p.decide.n_ptiles * p.decide.n_tables_launch;
    const long long ns = static_cast<long long>(p.scatter.n_mtiles) * p.scatter.n_ptiles * p.scatter.n_tables_launch;
    if (nd <= 0 || ns <= 0 || nd + ns > 0x7FFFFFFFLL) return cudaErrorInvalidConfiguration;
    p.n_decide = static_cast<int>(nd);
    const size_t a = lines_smem_bytes(p.decide), b = scatter_smem_bytes(p.scatter, kDecWarps);
    const bool contig = p.scatter.G.P_list == nullptr;
    const auto kernel = contig ? select_kernel<true> : select_kernel<false>;
    return launch(kernel, static_cast<unsigned>(nd + ns), 1, kDecThreads, a > b ? a : b, st, false, p);
}

}  // namespace plogp
