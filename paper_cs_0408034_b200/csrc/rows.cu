// scatter_rows_kernel: the Scatter half of the decision table, or the predictions of the Scatter chain and binomial tree
// (ids 11 and 12 of Table 2), where a row of message sizes is no multiple of a 32-byte sector.
//
// Bound by memory writes.  scatter_kernel and fused_kernel store row by row, 32 or 64 message sizes at a time; with such
// rows every store straddles lines and sectors.  Here a CTA has all message sizes of a table, one per thread, and walks one
// run of consecutive process counts: its cells are one piece of the plane.  The results of a few rows are put together in shared
// memory (two buffers, one barrier per flush) and go out from aligned addresses, whatever row they belong to.
// 2048 tables, P = 2..513, n_m = 127: 0.37 ms (4.7 TB/s) where scatter_kernel took 0.73; n_m = 145 0.46 for 0.88 (its rows of
// 128: 0.30).  Predictions, 1024 tables, n_m = 127: 0.30 ms for both ids where fused_kernel took 0.48, n_m = 145 0.34 for 0.57.
// A cell is about 60 instructions: groups of four per store instead of cells alone took 0.46 to 0.37 ms.
#include "device_common.cuh"

namespace plogp {

constexpr int kRowsThreads = kRowsMaxM;  // at most: one per message size, whole warps
constexpr int kRowsCells = 1280;         // of a flush, about

__host__ __device__ inline int rows_threads(int n_m) { return (n_m + 31) & ~31; }
__host__ __device__ inline int rows_per_flush(int n_m) { return n_m >= kRowsCells / 4 ? 4 : (n_m <= kRowsCells / 16 ? 16 : kRowsCells / n_m); }

// A piece of n cells starts `shift` cells behind a group of four that is aligned in the plane; it is staged with the same
// shift, so that a group is one 32-byte load and store (store4).  The cells of the groups at either end go one by one.
// PREDICT: times of ids 11 and 12 instead of the decision.  ALL: all ids that the kernel writes are enabled.
template <bool PREDICT, bool ALL>
__global__ void __launch_bounds__(kRowsThreads, 4) scatter_rows_kernel(const RowsParams p)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    constexpr int kPlanes = PREDICT ? 2 : 1;
    const int npad = p.T.npad, n_m = p.G.n_m, tid = threadIdx.x, threads = blockDim.x, R = rows_per_flush(n_m);
    const int cap = (R * n_m + 7) & ~3;  // of a buffer, with room for the shift
    double *const s_tab = reinterpret_cast<double *>(smem_raw);
    double *const s_t = s_tab + 3 * npad;                                        // [2][kPlanes][cap]
    uint8_t *const s_id = reinterpret_cast<uint8_t *>(s_t + 2 * kPlanes * cap);  // [2][cap]
    const uint32_t mask = p.G.mask;
    const bool on10 = !PREDICT && (ALL || ((mask >> 10) & 1u)), on11 = ALL || ((mask >> 11) & 1u), on12 = ALL || ((mask >> 12) & 1u);

    const int ptile = blockIdx.x % p.n_ptiles, table = p.table0 + blockIdx.x / p.n_ptiles;
    const int e0 = ptile * p.run_len, e1 = min(e0 + p.run_len, p.G.n_P);
    const bool m_ok = tid < n_m;
    const double md = static_cast<double>(p.G.m_list[min(tid, n_m - 1)]);

    dependents_may_start();
    const double L = p.T.lat[table];
    stage_table(s_tab, p.T, table);
    __syncthreads();
    const double gm = on10 ? gap_at(s_tab, npad, md) : 0.0;

    int P = p.G.P_lo + e0, lc = 0, P_next_lc = 2;  // ceil(log2 P) is lc below P_next_lc
    double pm1 = static_cast<double>(P - 1), cum = 0.0, s2 = 0.0;  // cum: sum of g(2^d m), d < lc
    double run = 0.0;                                              // Chain: sum of g(j m), j < P - 1
    ChainWalk walk;
    if (on11) {
        chain_front_parts(s_tab, npad, p.T.n_bp, nullptr, p.G.P_lo, md, e0, e0, e1, 0, 1, s_t + tid, s_t + threads + tid, 0);
        run = s_t[tid];
        walk.start(s_tab, npad, pm1 * md);
        __syncthreads();  // the buffers are now the rows'
    }

    const size_t plane = static_cast<size_t>(p.G.n_P) * n_m;
    // first cell of the run in planes 11 and 12 (predictions), or in the Scatter plane
    size_t at = (static_cast<size_t>(table - p.out_table0) * p.om.planes + (PREDICT ? 11 : p.om.plane_scat)) * plane + static_cast<size_t>(e0) * n_m;
    const uint32_t id10 = p.om.id_of[10], id11 = p.om.id_of[11], id12 = p.om.id_of[12];

    for (int e = e0, buf = 0; e < e1; e += R, buf ^= 1) {
        const int rows = min(R, e1 - e), n = rows * n_m;
        const int shift = static_cast<int>(at & 3u), shift12 = PREDICT ? static_cast<int>((at + plane) & 3u) : 0;
        double *const t_rows = s_t + buf * kPlanes * cap;
        uint8_t *const id_rows = s_id + buf * cap;
        if (m_ok) {
            double *ct = t_rows + shift + tid, *ct12 = t_rows + cap + shift12 + tid;
            uint8_t *ci = id_rows + shift + tid;
            for (int r = 0; r < rows; ++r) {
                if (on12 && P >= P_next_lc) {  // P passed a power of two
                    do {
                        cum += gap_at(s_tab, npad, md * static_cast<double>(1ull << lc));
                        ++lc;
                        P_next_lc = (1 << lc) + 1;
                    } while (P >= P_next_lc);
                    s2 = cum + static_cast<double>(lc) * L;
                }
                double t11 = CUDART_INF;
                if (on11) {
                    run += walk.at(s_tab, npad, pm1 * md);
                    t11 = fma(pm1, L, run);
                }
                if (PREDICT) {
                    *ct = t11;
                    *ct12 = s2;
                    ct12 += n_m;
                } else {
                    double t = CUDART_INF;
                    uint32_t id = 255;
                    if (on10) { t = fma(pm1, gm, L); id = id10; }  // Flat Tree
                    if (on11 && t11 < t) { t = t11; id = id11; }   // Chain
                    if (on12 && s2 < t) { t = s2; id = id12; }     // Binomial Tree
                    *ct = t;
                    *ci = static_cast<uint8_t>(id);
                    ci += n_m;
                }
                ct += n_m;
                ++P;
                pm1 += 1.0;
            }
        }
        __syncthreads();  // also: everyone is past the flush of the other buffer
        if (PREDICT) {
#pragma unroll
            for (int q = 0; q < 2; ++q) {
                if (!(q ? on12 : on11)) continue;
                const int first = q ? shift12 : shift, end = first + n;
                double *const out = p.d_time + (q ? at + plane : at) - first;
                const double *const in = t_rows + q * cap;
                for (int w = 4 * tid; w < end; w += 4 * threads) {
                    if (w >= first && w + 4 <= end) store4(out + w, in + w);
                    else
                        for (int i = max(w, first); i < min(w + 4, end); ++i) out[i] = in[i];
                }
            }
        } else {
            const int end = shift + n;
            double *const out_t = p.d_time + at - shift;
            uint8_t *const out_id = p.d_strategy + at - shift;
            uint32_t *const out_s = p.d_sbytes + at - shift;
            for (int w = 4 * tid; w < end; w += 4 * threads) {
                if (w >= shift && w + 4 <= end) {
                    store4(out_t + w, t_rows + w);
                    *reinterpret_cast<uint4 *>(out_s + w) = make_uint4(0u, 0u, 0u, 0u);
                    *reinterpret_cast<uint32_t *>(out_id + w) = *reinterpret_cast<const uint32_t *>(id_rows + w);
                } else {
                    for (int i = max(w, shift); i < min(w + 4, end); ++i) { out_t[i] = t_rows[i]; out_s[i] = 0u; out_id[i] = id_rows[i]; }
                }
            }
        }
        at += n;
    }
    last_block_waits(tid);
}

cudaError_t launch_rows(const RowsParams &p, bool predict, bool overlap, cudaStream_t st)
{
    const size_t cap = (static_cast<size_t>(rows_per_flush(p.G.n_m)) * p.G.n_m + 7) & ~size_t(3);
    const size_t smem = (3 * static_cast<size_t>(p.T.npad) + 2 * (predict ? 2 : 1) * cap) * sizeof(double) + (predict ? 0 : 2 * cap);
    const long long blocks = static_cast<long long>(p.n_ptiles) * p.n_tables_launch;
    if (blocks <= 0 || blocks > 0x7FFFFFFFLL || p.G.n_m > kRowsThreads) return cudaErrorInvalidConfiguration;
    const uint32_t ids = predict ? 0x1800u : 0x1C00u;
    const bool all = (p.G.mask & ids) == ids;
    const auto kernel = predict ? (all ? scatter_rows_kernel<true, true> : scatter_rows_kernel<true, false>)
                                : (all ? scatter_rows_kernel<false, true> : scatter_rows_kernel<false, false>);
    return launch(kernel, static_cast<unsigned>(blocks), 1, static_cast<unsigned>(rows_threads(p.G.n_m)), smem, st, overlap, p);
}

}  // namespace plogp
