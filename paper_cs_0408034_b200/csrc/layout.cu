// layout_kernel: the tables as the kernels read them (key | gap | slope, padded; internal.h) from the caller's arrays as
// they are.  The slope's division is the one step that costs; the host only checks the values and passes them on, a third of
// the bytes.
#include "device_common.cuh"

namespace plogp {

__global__ void __launch_bounds__(256) layout_kernel(const LayoutParams p)
{
    const long long total = static_cast<long long>(p.n_tables) * p.npad;
    for (long long idx = blockIdx.x * 256LL + threadIdx.x; idx < total; idx += gridDim.x * 256LL) {
        const long long t = idx / p.npad;
        const int i = static_cast<int>(idx - t * p.npad);
        const uint64_t *sz = p.sizes + (p.sizes_shared ? 0 : t * p.n_bp);
        const double *g = p.gap + t * p.n_bp;
        double key = CUDART_INF, gap = 0.0, slope = 0.0;
        if (i <= p.n_bp - 2) {
            key = static_cast<double>(sz[i]);
            gap = g[i];
            slope = (g[i + 1] - gap) / static_cast<double>(sz[i + 1] - sz[i]);
        }
        double *out = p.tab + t * 3 * p.npad + i;
        out[0] = key;
        out[p.npad] = gap;
        out[2 * p.npad] = slope;
    }
}

cudaError_t launch_layout(const LayoutParams &p, cudaStream_t st)
{
    const long long blocks = (static_cast<long long>(p.n_tables) * p.npad + 255) / 256;
    return launch(layout_kernel, static_cast<unsigned>(blocks < 4096 ? blocks : 4096), 1, 256, 0, st, false, p);
}

}  // namespace plogp
