// direct_block: one CTA of the Broadcast half of the decision table, or of the segmented planes of the predictions, for short
// candidate lists on small grids.  A thread has one cell (P, m) and evaluates every candidate of every enabled strategy in
// FP64; cells go to threads as they lie in the plane, so no thread is idle and stores are whole segments whatever the rows are.
//
// What bounds it: latency, set-up and one pass over the candidates behind two barriers.  Where a call is less than a wave of CTAs,
// the phases of lines_block (lines.cuh) cost more than what they leave out: each is a barrier and code that runs once.  One table
// of 49 x 19 cells, 7 candidates: pilots, bars and lines are 4400 of a CTA's 11000 cycles there.  A call from a graph, lines -> cells:
// 6.5 -> 4.7 us; 18 x 101, 48 candidates 8.9 -> 5.7.  The host says where (api.cu, with both sides measured).
#pragma once

#include "device_common.cuh"

namespace plogp {

template <bool PREDICT>
__device__ __forceinline__ void direct_block(const LinesParams &p, int block, unsigned char *smem_raw)
{
    const int npad = p.T.npad, n_s = p.G.n_s, n_m = p.G.n_m, tid = threadIdx.x;
    double *const s_tab = reinterpret_cast<double *>(smem_raw);
    double2 *const s_size = reinterpret_cast<double2 *>(s_tab + 3 * npad);  // [n_s] (s, 1 / s)
    double *const s_gap = reinterpret_cast<double *>(s_size + n_s);         // [n_s] g(s)
    const uint32_t mask = p.G.mask;
    const int trel = block / p.n_ptiles, table = p.table0 + trel;
    const int cells = p.G.n_P * n_m, cell = (block - trel * p.n_ptiles) * kDecThreads + tid;
    const int at = min(cell, cells - 1), pidx = at / n_m, midx = at - pidx * n_m;  // threads past the last cell repeat it

    dependents_may_start();
    const double L = p.T.lat[table];
    const uint32_t m_u = p.G.m_list[midx];
    const int ns = p.G.ns_of_m[midx], P = P_at(p.G, pidx);
    const uint32_t s_mine = tid < n_s ? s_at(p.G, tid) : 1u;
    stage_table(s_tab, p.T, table);
    __syncthreads();
    if (tid < n_s) {
        const double s = static_cast<double>(s_mine);
        s_size[tid] = make_double2(s, 1.0 / s);
        s_gap[tid] = gap_at(s_tab, npad, s);
    }
    const double md = static_cast<double>(m_u), gm = gap_at(s_tab, npad, md);
    const double g1 = PREDICT ? 0.0 : gap_at_one(s_tab, npad);
    const double rdv = 2.0 * g1 + 3.0 * L;  // rendezvous handshake: 2 g(1) + 3 L
    const double x = static_cast<double>(P - 1), lf = static_cast<double>(31 - __clz(P)), lc = static_cast<double>(32 - __clz(P - 1)), lcL = lc * L;
    __syncthreads();

    const bool has2 = (mask >> 2) & 1u, has5 = (mask >> 5) & 1u, has9 = (mask >> 9) & 1u, up = p.G.k_mode == 0;
    // the smallest size wins ties: in ascending order, '<'
    double t2 = CUDART_INF, t5 = CUDART_INF, t9 = CUDART_INF;
    int c2 = 0, c5 = 0, c9 = 0;
#pragma unroll 4
    for (int c = 0; c < ns; ++c) {
        const double2 size = s_size[c];
        const double g = s_gap[c];
        // Section 2's k: a whole number next to m / s, and which side of it the quotient is on
        const double q = round_whole(md * size.y), rest = fma(-q, size.x, md);
        const double k = up ? (rest > 0.0 ? q + 1.0 : q) : (rest < 0.0 ? q - 1.0 : q);
        const double Q = g * k;
        if (has2) {
            const double t = fma(x, Q, L);  // (P-1) (g(s) k) + L
            if (t < t2) { t2 = t; c2 = c; }
        }
        if (has5) {
            const double t = fma(x, g + L, g * (k - 1.0));  // (P-1) (g(s) + L) + g(s) (k-1)
            if (t < t5) { t5 = t; c5 = c; }
        }
        if (has9) {
            const double t = fma(lf, Q, lcL);  // floor(log2 P) g(s) k + ceil(log2 P) L
            if (t < t9) { t9 = t; c9 = c; }
        }
    }
    uint32_t s2 = m_u, s5 = m_u, s9 = m_u;
    if (ns > 0) {
        s2 = static_cast<uint32_t>(s_size[c2].x);
        s5 = static_cast<uint32_t>(s_size[c5].x);
        s9 = static_cast<uint32_t>(s_size[c9].x);
    } else {  // no candidate fits: the message goes whole (s = m, k = 1)
        t2 = fma(x, gm, L);
        t5 = x * (gm + L);
        t9 = fma(lf, gm, lcL);
    }
    if (cell >= cells) return;

    const size_t plane = static_cast<size_t>(cells);
    if constexpr (PREDICT) {
        double *const out_t = p.p_time + static_cast<size_t>(table - p.out_table0) * 13 * plane + cell;
        if (has2) out_t[2 * plane] = t2;
        if (has5) out_t[5 * plane] = t5;
        if (has9) out_t[9 * plane] = t9;
        if (p.p_best_s) {
            uint32_t *const out_s = p.p_best_s + static_cast<size_t>(table - p.out_table0) * 3 * plane + cell;
            if (has2) out_s[0] = s2;
            if (has5) out_s[plane] = s5;
            if (has9) out_s[2 * plane] = s9;
        }
    } else {
        double t = CUDART_INF;
        uint32_t s = 0, id = 255;
        // the lower id wins ties: in descending order, '<='
        auto take = [&](int i, double v, uint32_t size) {
            if (((mask >> i) & 1u) && !(v > t)) { t = v; s = size; id = p.om.id_of[i]; }
        };
        take(9, t9, s9);
        take(8, fma(lf, gm, lc * rdv), 0u);           // Binomial Tree Rendezvous
        take(7, fma(lf, gm, lcL), 0u);                // Binomial Tree
        take(6, lc * fma(2.0, gm, L), 0u);            // Binary Tree (the printed bound)
        take(5, t5, s5);
        take(4, x * (gm + rdv), 0u);                  // Chain Rendezvous
        take(3, x * (gm + L), 0u);                    // Chain
        take(2, t2, s2);
        take(1, fma(x, gm, rdv), 0u);                 // Flat Tree Rendezvous
        take(0, fma(x, gm, L), 0u);                   // Flat Tree
        const size_t o = (static_cast<size_t>(table - p.out_table0) * p.om.planes + p.om.plane_bcast) * plane + cell;
        p.d_time[o] = t;
        p.d_sbytes[o] = s;
        p.d_strategy[o] = static_cast<uint8_t>(id);
    }
}

}  // namespace plogp
