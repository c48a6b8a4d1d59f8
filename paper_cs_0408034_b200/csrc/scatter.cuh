// scatter_block: one CTA of the Scatter half of the decision table (Table 2 of the paper: Flat Tree, Chain,
// Binomial Tree; selection as in Sections 1 and 5).
//
// Listed process counts: the Chain's sum up to any j from a table of sums per interval in shared memory (ChainTable), with
// no loop over the intervals between two process counts and no division per cell.  1000 tables of 50 sizes, 203 process
// counts up to 3000, 101 message sizes: 124 -> 110 us (issue, 0.75 of the slots); the call 339 -> 324 us.
//
// Lanes are message sizes (32 V consecutive m per warp, V = 1 or 2 neighbours per lane, so every store is one aligned
// row segment); each warp owns a contiguous run of process counts and walks it in ascending order, which turns
// the Chain model's sum over j = 1..P-1 of g(j m) into a running sum along the thread: the argument
// j m grows by m per step, the table interval is kept in registers and only reloaded when the
// argument crosses a breakpoint.  The sum in front of a warp's run is taken in closed form per table interval
// (chain_front_parts and chain_front_sum in device_common.cuh), so a range of process counts can be split over any number of CTAs in one launch.
#pragma once

#include "device_common.cuh"

namespace plogp {

constexpr int kChainRun = 0, kChainRange = 1, kChainTable = 2;

namespace scatter {

template <int V> struct Out;
template <> struct Out<1> {
    static __device__ __forceinline__ void put(double *t, uint32_t *s, uint8_t *id, const double *bt, const uint32_t *bid)
    {
        *t = bt[0]; *s = 0u; *id = static_cast<uint8_t>(bid[0]);
    }
};
template <> struct Out<2> {
    static __device__ __forceinline__ void put(double *t, uint32_t *s, uint8_t *id, const double *bt, const uint32_t *bid)
    {
        *reinterpret_cast<double2 *>(t) = make_double2(bt[0], bt[1]);
        *reinterpret_cast<uint2 *>(s) = make_uint2(0u, 0u);
        *reinterpret_cast<uint16_t *>(id) = static_cast<uint16_t>(bid[0] | bid[1] << 8);
    }
};

}  // namespace scatter

// CHAIN, the Scatter Chain's sums: kChainRun for the contiguous range P_lo + index (one new gap per step), kChainTable for
// listed process counts from a table of sums per interval (V = 1), kChainRange for them by closed forms along the run.
// ALL: the three Scatter strategies are enabled (the usual case), known at compile time.
// V: message sizes per lane.  W: warps of the CTA.
template <int CHAIN, bool ALL, int V, int W>
__device__ __forceinline__ void scatter_block(const ScatterParams &p, int block, unsigned char *smem_raw)
{
    double *s_tab = reinterpret_cast<double *>(smem_raw);
    double *s_cum = s_tab + 3 * p.T.npad;          // [lc_max][32 V]
    double *s_sum = s_cum + p.G.lc_max * 32 * V;   // [2][W][32 V]; kChainTable: [W][32], then [2][n_bp - 1][32]
    constexpr bool CONTIG = CHAIN == kChainRun;
    static_assert(CHAIN != kChainTable || V == 1, "a column per lane");
    const int npad = p.T.npad;
    const uint32_t mask = p.G.mask;
    const bool on10 = ALL || ((mask >> 10) & 1u), on11 = ALL || ((mask >> 11) & 1u), on12 = ALL || ((mask >> 12) & 1u);

    int b = block;
    const int mtile = b % p.n_mtiles;
    b /= p.n_mtiles;
    const int ptile = b % p.n_ptiles;
    const int trel = b / p.n_ptiles;
    const int table = p.table0 + trel;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int midx = mtile * 32 * V + lane * V;
    const bool m_ok = midx < p.G.n_m;  // V = 2 is taken for even n_m only: both of a lane's sizes exist or neither
    double md[V], gm[V];
#pragma unroll
    for (int v = 0; v < V; ++v) md[v] = static_cast<double>(p.G.m_list[min(midx + v, p.G.n_m - 1)]);

    dependents_may_start();
    const double L = p.T.lat[table];
    stage_table(s_tab, p.T, table);
    __syncthreads();
#pragma unroll
    for (int v = 0; v < V; ++v) gm[v] = gap_at(s_tab, npad, md[v]);

    // Binomial Tree: sums of g(2^j m); the gaps are looked up by all warps, warp 0 adds them up
    if (on12) {
        for (int d = warp; d < p.G.lc_max; d += W)
#pragma unroll
            for (int v = 0; v < V; ++v) s_cum[(d * V + v) * 32 + lane] = gap_at(s_tab, npad, md[v] * static_cast<double>(1ull << d));
    }

    // this warp's run of process-count indices
    const int c0 = ptile * (W * p.run_len);
    const int e0 = min(c0 + warp * p.run_len, p.G.n_P), e1 = min(e0 + p.run_len, p.G.n_P);

    // ---- Chain: the sum in front of the run ----
    ChainWalk walk[V];
    const ChainTable ct{s_sum + W * 32 + (threadIdx.x & 31), s_sum + (W + p.T.n_bp - 1) * 32 + (threadIdx.x & 31), s_sum + (threadIdx.x & 31)};
    ChainAt place;
    double run[V], j_last = 0.0;  // sum up to j_last
#pragma unroll
    for (int v = 0; v < V; ++v) run[v] = 0.0;
    if (on11 && CHAIN == kChainTable) ct.build(s_tab, npad, p.T.n_bp, md[0], static_cast<double>(p.G.P_list[p.G.n_P - 1] - 1), warp, W);
    if (on11 && CHAIN != kChainTable) {
#pragma unroll
        for (int v = 0; v < V; ++v)
            chain_front_parts(s_tab, npad, p.T.n_bp, p.G.P_list, p.G.P_lo, md[v], c0, e0, e1, warp, W, s_sum + v * 32 + lane, s_sum + (W * V + v) * 32 + lane, 32 * V);
    }
    __syncthreads();
    if (on12 && warp == 0) {
#pragma unroll
        for (int v = 0; v < V; ++v) {
            double acc = 0.0;
            for (int d = 0; d < p.G.lc_max; ++d) {
                acc += s_cum[(d * V + v) * 32 + lane];
                s_cum[(d * V + v) * 32 + lane] = acc;
            }
        }
    }
    if (on11 && CHAIN == kChainTable) ct.add_up(p.T.n_bp, warp, W);
    if (on12 || (on11 && CHAIN == kChainTable)) __syncthreads();
    if (e0 >= e1 || (CHAIN != kChainTable && !m_ok)) return;  // no barriers below; kChainTable shares process counts over the lanes

    int P = P_at(p.G, e0);
    if (on11 && CHAIN == kChainTable) place.start(s_tab, npad, ct, static_cast<double>(P - 1) * md[0]);
    if (on11 && CHAIN != kChainTable) {
        j_last = warp == 0 ? static_cast<double>(P - 2) : static_cast<double>(P_at(p.G, e0 - 1) - 1);
#pragma unroll
        for (int v = 0; v < V; ++v) {
            run[v] = chain_front_sum(s_sum + v * 32 + lane, s_sum + (W * V + v) * 32 + lane, 32 * V, warp, W);
            walk[v].start(s_tab, npad, (j_last + 1.0) * md[v]);
        }
    }

    const size_t plane = static_cast<size_t>(p.G.n_P) * p.G.n_m, row = static_cast<size_t>(p.G.n_m);
    const size_t o = (static_cast<size_t>(table - p.out_table0) * p.om.planes + p.om.plane_scat) * plane + static_cast<size_t>(e0) * row + midx;
    // running output pointers (one row of n_m cells further per process count) and the ids as the caller names them
    double *out_t = p.d_time + o;
    uint8_t *out_id = p.d_strategy + o;
    uint32_t *out_s = p.d_sbytes + o;
    const uint32_t id10 = p.om.id_of[10], id11 = p.om.id_of[11], id12 = p.om.id_of[12];
    int P_next_lc = 0;  // first process count with a larger ceil(log2 P)
    double s2[V], pm1 = static_cast<double>(P - 1), x[V];
#pragma unroll
    for (int v = 0; v < V; ++v) { s2[v] = 0.0; x[v] = pm1 * md[v]; }

    int P_lane = P;  // kChainTable: 32 listed process counts, one per lane
    for (int e = e0; e < e1; ++e) {
        if (!CONTIG) {
            if (CHAIN == kChainTable) {
                if (((e - e0) & 31) == 0) P_lane = p.G.P_list[min(e + lane, e1 - 1)];
                P = __shfl_sync(0xffffffffu, P_lane, (e - e0) & 31);
            } else {
                P = P_at(p.G, e);
            }
            pm1 = static_cast<double>(P - 1);
        }
        if (P >= P_next_lc) {  // P passed a power of two
            const int lc = 32 - __clz(P - 1);
            P_next_lc = (1 << lc) + 1;
            const double lcL = static_cast<double>(lc) * L;
#pragma unroll
            for (int v = 0; v < V; ++v) s2[v] = on12 ? s_cum[((lc - 1) * V + v) * 32 + lane] + lcL : 0.0;
        }
        double bt[V];
        uint32_t bid[V];
#pragma unroll
        for (int v = 0; v < V; ++v) {
            bt[v] = CUDART_INF;
            bid[v] = 255;
            if (on10) { bt[v] = fma(pm1, gm[v], L); bid[v] = id10; }  // Flat Tree
            if (on11) {                                               // Chain
                if (CONTIG) {
                    run[v] += walk[v].at(s_tab, npad, x[v]);
                    x[v] += md[v];  // exact: j m < 2^53
                } else if (CHAIN == kChainTable) {
                    run[v] = place.sum(s_tab, npad, ct, md[v], pm1);
                } else {
                    run[v] += walk[v].range(s_tab, npad, md[v], j_last + 1.0, pm1);
                }
                const double t = fma(pm1, L, run[v]);
                if (t < bt[v]) { bt[v] = t; bid[v] = id11; }
            }
            if (on12 && s2[v] < bt[v]) { bt[v] = s2[v]; bid[v] = id12; }  // Binomial Tree
        }
        if (CHAIN != kChainTable || m_ok) scatter::Out<V>::put(out_t, out_s, out_id, bt, bid);
        out_t += row; out_id += row; out_s += row;
        if (CONTIG) { ++P; pm1 += 1.0; }
        else j_last = pm1;
    }
}

}  // namespace plogp
