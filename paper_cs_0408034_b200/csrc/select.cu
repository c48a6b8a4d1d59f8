// select_kernel: both halves of a decision table in one launch, for grids that the GPU holds in one go.  There a call is
// mostly launches: some CTAs take the Broadcast half (direct.cuh on the smallest grids, else lines.cuh), the others the Scatter half
// (scatter.cuh, with the Broadcast half's four warps per CTA).  One table, P = 2..50, 19 message sizes, 7 candidates, between calls
// from a graph: 4.7 us (Ethernet strategies; with lines 6.5), all strategies 6.1 (6.3).
#include "direct.cuh"
#include "lines.cuh"
#include "scatter.cuh"

namespace plogp {

template <bool CONTIG, bool DIRECT>
__global__ void __launch_bounds__(kDecThreads, DIRECT ? 6 : 4) select_kernel(const SelectParams p)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    // the half with the longer CTAs first: the Scatter half beside a cell per thread (64 tables of 49 x 19: 8.4 -> 8.0 us), the
    // Broadcast half beside lines (16 tables of 199 x 33 the other way round: 8.7 -> 9.5)
    const int first = DIRECT ? gridDim.x - p.n_decide : p.n_decide, block = blockIdx.x;
    if ((block < first) != DIRECT) {
        const int b = DIRECT ? block - first : block;
        if constexpr (DIRECT) direct_block<false>(p.decide, b, smem_raw);
        else lines_block<false, false>(p.decide, b, smem_raw);
    } else {
        scatter_block<CONTIG ? kChainRun : kChainRange, false, 1, kDecWarps>(p.scatter, DIRECT ? block : block - first, smem_raw);
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
    const auto kernel = p.decide.direct ? (contig ? select_kernel<true, true> : select_kernel<false, true>)
                                        : (contig ? select_kernel<true, false> : select_kernel<false, false>);
    return launch(kernel, static_cast<unsigned>(nd + ns), 1, kDecThreads, a > b ? a : b, st, false, p);
}

}  // namespace plogp
