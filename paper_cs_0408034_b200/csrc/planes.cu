// planes_kernel: the closed-form Broadcast and flat Scatter planes of plogp_predict (ids 0, 1, 3, 4, 6, 7, 8 of Table 1,
// id 10 of Table 2) where a row of message sizes is no multiple of a 32-byte sector.
//
// Bound by memory writes.  fused_kernel gives each lane a message size and stores row by row; with such rows every store
// straddles lines and sectors: 3 write requests for 2, two of them with part of a sector.  These models need nothing but g(m)
// and P, so here the cells of a plane are taken as they lie in memory: a warp's store is 32 cells from a 256-byte boundary,
// whatever row they belong to, and each thread follows its process count and message size as it steps through the plane.
// g(m) of all message sizes is in shared memory.  1024 tables, P = 2..513, n_m = 145: the eight planes take 0.90 ms (5.4 TB/s)
// where fused_kernel took 1.88 (2.45 for all ten; n_m = 127: 0.81 for 1.61).
#include "device_common.cuh"

namespace plogp {

constexpr int kPlThreads = 256;

__global__ void __launch_bounds__(kPlThreads) planes_kernel(const PlanesParams p)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    double *s_tab = reinterpret_cast<double *>(smem_raw);
    double *s_g = s_tab + 3 * p.T.npad;  // [n_m]
    const int npad = p.T.npad, n_m = p.G.n_m, tid = threadIdx.x;
    const int seg = blockIdx.x, table = p.table0 + blockIdx.y;
    dependents_may_start();
    const double L = p.T.lat[table];
    stage_table(s_tab, p.T, table);
    __syncthreads();
    for (int m = tid; m < n_m; m += kPlThreads) s_g[m] = gap_at(s_tab, npad, static_cast<double>(p.G.m_list[m]));
    const double rdv = 2.0 * gap_at_one(s_tab, npad) + 3.0 * L;  // rendezvous handshake: 2 g(1) + 3 L
    __syncthreads();

    const long long cells = static_cast<long long>(p.G.n_P) * n_m;
    const int dP = kPlThreads / n_m, dm = kPlThreads - dP * n_m;
    // one plane: value(P, g(m)) over this CTA's cells
    auto plane = [&](int id, auto &&value) {
        double *const out = p.p_time + (static_cast<long long>(table - p.out_table0) * 13 + id) * cells;
        const int shift = static_cast<int>((reinterpret_cast<uintptr_t>(out) >> 3) & 31u);  // cells behind a 256-byte boundary
        const long long a0 = seg * p.seg_cells, a1 = min(a0 + p.seg_cells, cells + shift);
        const long long f0 = a0 + tid - shift, lifted = f0 + 32LL * n_m;  // never negative: shift < 32 <= 32 n_m
        int pi = static_cast<int>(lifted / n_m) - 32, m = static_cast<int>(lifted % n_m);
        double *o = out + f0;
#pragma unroll 4
        for (long long a = a0 + tid; a < a1; a += kPlThreads, o += kPlThreads) {
            if (a >= shift) *o = value(P_at(p.G, pi), s_g[m]);
            pi += dP;
            m += dm;
            if (m >= n_m) { m -= n_m; ++pi; }
        }
    };
    auto x = [](int P) { return static_cast<double>(P - 1); };
    auto lf = [](int P) { return static_cast<double>(31 - __clz(P)); };
    auto lc = [](int P) { return static_cast<double>(32 - __clz(P - 1)); };
    const uint32_t mask = p.mask;
    if (mask & 1u) plane(0, [&](int P, double g) { return fma(x(P), g, L); });                           // Flat Tree
    if ((mask >> 1) & 1u) plane(1, [&](int P, double g) { return fma(x(P), g, rdv); });                  // Flat Tree Rendezvous
    if ((mask >> 3) & 1u) plane(3, [&](int P, double g) { return x(P) * (g + L); });                     // Chain
    if ((mask >> 4) & 1u) plane(4, [&](int P, double g) { return x(P) * (g + rdv); });                   // Chain Rendezvous
    if ((mask >> 6) & 1u) plane(6, [&](int P, double g) { return lc(P) * fma(2.0, g, L); });             // Binary Tree (the printed bound)
    if ((mask >> 7) & 1u) plane(7, [&](int P, double g) { return fma(lf(P), g, lc(P) * L); });           // Binomial Tree
    if ((mask >> 8) & 1u) plane(8, [&](int P, double g) { return fma(lf(P), g, lc(P) * rdv); });         // Binomial Tree Rendezvous
    if ((mask >> 10) & 1u) plane(10, [&](int P, double g) { return fma(x(P), g, L); });                  // Scatter Flat Tree
    last_block_waits(tid);
}

cudaError_t launch_planes(const PlanesParams &p, bool overlap, cudaStream_t st)
{
    const size_t smem = (3 * static_cast<size_t>(p.T.npad) + p.G.n_m) * sizeof(double);
    const long long segs = (static_cast<long long>(p.G.n_P) * p.G.n_m + 31 + p.seg_cells - 1) / p.seg_cells;
    if (segs <= 0 || segs > 0x7FFFFFFFLL || p.n_tables_launch <= 0 || p.n_tables_launch > 65535) return cudaErrorInvalidConfiguration;
    return launch(planes_kernel, static_cast<unsigned>(segs), static_cast<unsigned>(p.n_tables_launch), kPlThreads, smem, st, overlap, p);
}

}  // namespace plogp
