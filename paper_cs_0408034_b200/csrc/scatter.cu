// scatter_kernel: Scatter half of the decision table (scatter.cuh).
#include "scatter.cuh"

namespace plogp {

template <int CHAIN, bool ALL, int V>
__global__ void __launch_bounds__(kThreads, 4) scatter_kernel(const ScatterParams p)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    scatter_block<CHAIN, ALL, V, kWarps>(p, blockIdx.x, smem_raw);
    last_block_waits(threadIdx.x);
}

size_t scatter_smem_bytes(const ScatterParams &p, int warps)
{
    const size_t sums = p.chain_table ? static_cast<size_t>(warps) + 2 * (p.T.n_bp - 1) : 2 * static_cast<size_t>(warps) * p.vec;
    return (3 * static_cast<size_t>(p.T.npad) + static_cast<size_t>(p.G.lc_max) * 32 * p.vec + 32 * sums) * sizeof(double);
}

template <int CHAIN, bool ALL, int V>
static cudaError_t launch_scatter_t(const ScatterParams &p, bool overlap, cudaStream_t st)
{
    const size_t smem = scatter_smem_bytes(p, kWarps);
    const long long blocks = static_cast<long long>(p.n_mtiles) * p.n_ptiles * p.n_tables_launch;
    if (blocks <= 0 || blocks > 0x7FFFFFFFLL) return cudaErrorInvalidConfiguration;
    return launch(scatter_kernel<CHAIN, ALL, V>, static_cast<unsigned>(blocks), 1, kThreads, smem, st, overlap, p);
}

template <int V>
static cudaError_t launch_scatter_v(const ScatterParams &p, bool overlap, cudaStream_t st)
{
    const bool all = (p.G.mask & 0x1C00u) == 0x1C00u;
    if (!p.G.P_list) return all ? launch_scatter_t<kChainRun, true, V>(p, overlap, st) : launch_scatter_t<kChainRun, false, V>(p, overlap, st);
    if (V == 1 && p.chain_table) return all ? launch_scatter_t<kChainTable, true, 1>(p, overlap, st) : launch_scatter_t<kChainTable, false, 1>(p, overlap, st);
    return all ? launch_scatter_t<kChainRange, true, V>(p, overlap, st) : launch_scatter_t<kChainRange, false, V>(p, overlap, st);
}

cudaError_t launch_scatter(const ScatterParams &p, bool overlap, cudaStream_t st) { return p.vec == 2 ? launch_scatter_v<2>(p, overlap, st) : launch_scatter_v<1>(p, overlap, st); }

}  // namespace plogp
