// CUDA kernels (sm_100a) for the pLogP cost models of Table 1 (Broadcast) and Table 2 (Scatter)
// of "Fast Tuning of Intra-Cluster Collective Communications", the segment-size search of
// Section 3.1 and the strategy selection of Sections 1 and 5.
//
// This file:
//   sweep_kernel   lane <-> process count P.  One CTA owns one message size m, a tile of P values
//                  and a chunk of the candidate segment sizes, whose lines are bounded from below for many
//                  candidates at a time; what the FP32 bounds leave open is decided in FP64.  Used when the
//                  candidate list is long.
//   fused_kernel   lane <-> message size m (32 consecutive m per warp, so every output row is
//                  written as full, aligned segments).  Evaluates all enabled strategies, reduces the sweep
//                  kernel's partial minima where segmented ones are among them, keeps the
//                  Scatter Chain sum running along each warp's contiguous run of P, and writes either
//                  the predicted planes or the decision table.  The general path.
// Short candidate lists have faster, specialised kernels: decide.cu (Broadcast half of the decision
// table), scatter.cu (Scatter half), select.cu (both in one launch), segmin.cu (segmented planes of the predictions); the host
// routes them there, and fused_kernel writes the other prediction planes.  Rows off the sectors on large grids go to planes.cu
// and rows.cu.
#include "device_common.cuh"

namespace plogp {

// ------------------------------------------------------------------------------------------
// Segment sweep: partial minima over one chunk of candidates (Section 3.1 search)
// ------------------------------------------------------------------------------------------
//
// For a fixed (m, s) every segmented model of Table 1 is a line in P (or in floor(log2 P)):
//   id 5: (P-1) (g(s)+L) + g(s)(k-1)          = fma(P-1, B, C)   B = g(s)+L, C = g(s)(k-1)
//   id 2: (P-1) (g(s) k) + L                  = fma(P-1, Q, L)   Q = g(s) k
//   id 9: floor(log2 P) g(s) k + ceil(log2 P) L = fma(lf, Q, lc L)
// so the CTA computes (B, C, Q) once per candidate, and a line of the smallest B and C (or Q) of some candidates is below all of
// theirs at every process count.
//
// All terms are non-negative, and coefficients, process count and multiply-add are rounded down to FP32, so a bound is never above
// the FP64 time.  It is taken three times, each time for the process counts (lanes) in which the one before is not above the best
// time known there:
//   * for a sub-chunk of 256 candidates from its first and last size alone (the smallest g between them, the last one's number
//     of segments), before any candidate is looked at;
//   * for its groups of 32, from the smallest coefficients;
//   * for the group's candidates one by one.
// Four at a time, what is left is compared in FP64, unless the group's smallest coefficients in FP64 show that none is better than
// what the warp has (a rounded fused multiply-add is monotone in them): where gaps are equal over many sizes, times are
// equal and no bound in FP32 tells them apart, nor where times lie outside its range.  The results are those of the exhaustive FP64
// search, bit for bit.  The upper bounds of the best times start from log-spaced candidates of the whole list (rounded up in FP32), so a
// chunk far from the optimum never leaves the first step.  The best times themselves are touched by the exact pass alone and live in
// shared memory.
//
// What bounds it: the exact passes of the CTAs that have the best sizes, one vote after another, while the others are done.  P =
// 2..4096, 128 message sizes, every 4 B up to 1 MB, ids 2 and 5: 8.4 ms with a bound of every cell, 1.33 with groups of 32, 1.23 with
// the first 256 process counts in CTAs of their own, 0.64 with sub-chunks passed over.  Tables that defeat the bounds, ms for ids 2
// and 5 (id 9), with a bound of every cell -> groups compared in FP32 alone -> in FP64 as well: equal gaps 25.7 (12.1) -> 49.4 (19.5) ->
// 11.4 (4.5), in stairs 11.5 (6.7) -> 4.4 (3.7) -> 1.1 (0.88), a latency 1e9 times the gaps 26.3 (27.1) -> 28.6 (35.1) -> 7.7 (8.9),
// times outside FP32's range 86.8 (37.0) -> 108.9 (43.4) -> 30.3 (14.6).  Small sweeps pay 1 to 3 % for the groups' minima.
//
// A warp owns 256 consecutive process counts (lane + 32 r).  The CTA's 8 warps cover p.wp such tiles side by side and
// split the candidates of a sub-chunk 8 / p.wp ways, so that a short range of process counts leaves no warp idle.

template <bool HAS2, bool HAS5, bool IS9>
__global__ void __launch_bounds__(kThreads, 2) sweep_kernel(const SweepParams p)
{
    static_assert(!IS9 || !(HAS2 || HAS5), "id 9 has lines of its own");
    constexpr bool QL = HAS2 || IS9;  // lists of Q
    constexpr int R = kSweepR;
    constexpr unsigned kFull = 0xffffffffu;
    constexpr int kNid = (HAS2 ? 1 : 0) + (HAS5 ? 1 : 0) + (IS9 ? 1 : 0);
    extern __shared__ __align__(16) unsigned char smem_raw[];
    double *s_tab = reinterpret_cast<double *>(smem_raw);
    double2 *s_bc = reinterpret_cast<double2 *>(s_tab + 3 * p.T.npad);  // [2][kSweepSub]
    double *s_q = reinterpret_cast<double *>(s_bc + 2 * kSweepSub);     // [2][kSweepSub]
    double *s_best = s_q + 2 * kSweepSub;                               // [kNid][kWarps][R][32]
    double *s_db = s_best + kNid * kWarps * R * 32, *s_dc = s_db + 2 * kSweepGroups, *s_dq = s_dc + 2 * kSweepGroups;  // [2][kSweepGroups]: smallest of a group's
    float *s_bf = reinterpret_cast<float *>(s_dq + 2 * kSweepGroups);  // [2][kSweepSub]
    float *s_cf = s_bf + 2 * kSweepSub, *s_qf = s_cf + 2 * kSweepSub;
    float *s_gb = s_qf + 2 * kSweepSub, *s_gc = s_gb + 2 * kSweepGroups, *s_gq = s_gc + 2 * kSweepGroups;  // [2][kSweepGroups]: smallest of a group's
    float *s_lb = s_gq + 2 * kSweepGroups, *s_lc = s_lb + kThreads, *s_lq = s_lc + kThreads;  // [kThreads]: bounds of a sub-chunk's
    int *s_need = reinterpret_cast<int *>(s_lq + kThreads);                                   // [kThreads]: it has to be looked at
    uint32_t *s_idx = reinterpret_cast<uint32_t *>(s_need + kThreads);                        // [kNid][kWarps][R][32]

    const int tid = threadIdx.x;
    const int pi = blockIdx.x / p.n_ptiles;
    const int ptile = blockIdx.x - pi * p.n_ptiles;
    const int trel = blockIdx.y;
    const int table = p.table0 + trel;
    const int m_idx = p.pair_m[pi];
    const int chunk = p.pair_chunk[pi];
    const int row = p.pair_row[pi];
    const uint32_t m_u = p.G.m_list[m_idx];
    const int ns = p.G.ns_of_m[m_idx];
    const int s_begin = chunk * p.chunk_len;
    const int s_end = s_begin + min(p.chunk_len, ns - s_begin);  // (indices up to 2^31 - 1: differences only, no sums past the end)
    const int n_sub = (s_end - s_begin + kSweepSub - 1) / kSweepSub;

    dependents_may_start();
    stage_table(s_tab, p.T, table);
    const double L = p.T.lat[table];

    const int lane = tid & 31, warp = tid >> 5;
    // The first 256 process counts have CTAs of their own, whose warps split the candidates: where P is small the best size
    // moves fast, and most of the groups that have to be looked at are there.
    const int wp = ptile == 0 ? 1 : p.wp, wc = kWarps / wp, my_p = warp & (wp - 1), my_c = warp / wp;
    const int tile0 = ptile == 0 ? 0 : 32 * R * (1 + (ptile - 1) * wp);
    const int g_len = kSweepGroups / wc;  // this warp's groups of a sub-chunk
    const int p_first = tile0 + my_p * (32 * R) + lane;
    // a process count past the last one repeats the last one
    auto P_of = [&](int r) { return P_at(p.G, min(p_first + 32 * r, p.G.n_P - 1)); };
    auto x_exact = [&](int P) { return IS9 ? static_cast<double>(31 - __clz(P)) : static_cast<double>(P - 1); };
    auto c_exact = [&](int P) { return IS9 ? static_cast<double>(32 - __clz(P - 1)) * L : L; };

    float xf[R], cf[IS9 ? R : 1];  // multiplier and, where the offset is not a candidate's, offset, rounded down
    float T2[QL ? R : 1], T5[HAS5 ? R : 1];  // upper bounds of the best times
#pragma unroll
    for (int r = 0; r < R; ++r) {
        const int P = P_of(r);
        xf[r] = IS9 ? static_cast<float>(31 - __clz(P)) : __int2float_rd(P - 1);
        if (IS9) cf[r] = __double2float_rd(c_exact(P));
        if (QL) T2[r] = CUDART_INF_F;
        if (HAS5) T5[r] = CUDART_INF_F;
    }
    if (!IS9) cf[0] = __double2float_rd(L);
    double *best = s_best + warp * R * 32 + lane;  // + id slot * kWarps * R * 32 + r * 32
    uint32_t *bidx = s_idx + warp * R * 32 + lane;
    constexpr int kIdStep = kWarps * R * 32;
#pragma unroll
    for (int q = 0; q < kNid; ++q)
#pragma unroll
        for (int r = 0; r < R; ++r) { best[q * kIdStep + r * 32] = CUDART_INF; bidx[q * kIdStep + r * 32] = 0xFFFFFFFFu; }
    __syncthreads();

    auto coefficients = [&](int si, double &B, double &C, double &Q) {
        const uint32_t s = s_at(p.G, si);
        const double gs = gap_at(s_tab, p.T.npad, static_cast<double>(s));
        const double k = static_cast<double>(segments(m_u, s, p.G.k_mode));
        B = gs + L;
        C = gs * (k - 1.0);
        Q = gs * k;
    };
    auto fill = [&](int sub, int buf) {
        const int first = s_begin + sub * kSweepSub, o = buf * kSweepSub + tid;
        double B = CUDART_INF, C = CUDART_INF, Q = CUDART_INF;  // padding: the bound is +inf
        if (tid < s_end - first) coefficients(first + tid, B, C, Q);
        // a warp's candidates are a group
        if (HAS5) {
            const float b = __double2float_rd(B), c = __double2float_rd(C);
            s_bc[o] = make_double2(B, C);
            s_bf[o] = b;
            s_cf[o] = c;
            const double b_min = warp_min(B), c_min = warp_min(fmin(C, CUDART_INF));  // inf * 0 as inf
            if (lane == 0) {
                s_db[o >> 5] = b_min; s_gb[o >> 5] = __double2float_rd(b_min);
                s_dc[o >> 5] = c_min; s_gc[o >> 5] = __double2float_rd(c_min);
            }
        }
        if (QL) {
            const float q = __double2float_rd(Q);
            s_q[o] = Q;
            s_qf[o] = q;
            const double q_min = warp_min(Q);
            if (lane == 0) { s_dq[o >> 5] = q_min; s_gq[o >> 5] = __double2float_rd(q_min); }
        }
    };

    // ---- upper bounds from log-spaced candidates of the whole list ----
    const int n_seed = min(kSweepSeeds, ns);
    if (tid < kSweepSeeds) {
        float B = 0.f, C = CUDART_INF_F, Q = CUDART_INF_F;
        if (tid < n_seed) {
            int si = min(ns - 1, static_cast<int>(exp2f(log2f(static_cast<float>(ns)) * (static_cast<float>(tid + 1) / n_seed))) - 1);
            if (!p.G.s_list) {  // the smallest candidate with the same number of segments is the better one
                const uint32_t s = s_at(p.G, si), k = max(segments(m_u, s, p.G.k_mode), 1u);
                const uint32_t t = p.G.k_mode == 0 ? (m_u + k - 1) / k : m_u / (k + 1) + 1;
                si = t <= p.G.s_lo ? 0 : min(si, static_cast<int>((t - p.G.s_lo + p.G.s_step - 1) / p.G.s_step));
            }
            double Bd, Cd, Qd;
            coefficients(max(si, 0), Bd, Cd, Qd);
            B = __double2float_ru(Bd); C = __double2float_ru(Cd); Q = __double2float_ru(Qd);
        }
        s_bf[tid] = B; s_cf[tid] = C; s_qf[tid] = Q;
    }
    __syncthreads();
    {
        float xu[R], cu[IS9 ? R : 1];  // rounded up
#pragma unroll
        for (int r = 0; r < R; ++r) {
            const int P = P_of(r);
            xu[r] = IS9 ? static_cast<float>(31 - __clz(P)) : __int2float_ru(P - 1);
            if (IS9) cu[r] = __double2float_ru(c_exact(P));
        }
        if (!IS9) cu[0] = __double2float_ru(L);
#pragma unroll 1
        for (int i = 0; i < n_seed; ++i) {
            const float B = s_bf[i], C = s_cf[i], Q = s_qf[i];
#pragma unroll
            for (int r = 0; r < R; ++r) {
                if (HAS5) T5[r] = fminf(T5[r], __fmaf_ru(xu[r], B, C));
                if (QL) T2[r] = fminf(T2[r], __fmaf_ru(xu[r], Q, cu[IS9 ? r : 0]));
            }
        }
    }
    __syncthreads();

    // rows in which the line of these coefficients is not above the best time known: bit r: id 2 or 9, bit 16 + r: id 5
    auto rows_of = [&](float b, float c, float q) {
        unsigned hit = 0;
#pragma unroll
        for (int r = 0; r < R; ++r) {
            if (QL && __fmaf_rd(xf[r], q, cf[IS9 ? r : 0]) <= T2[r]) hit |= 1u << r;
            if (HAS5 && __fmaf_rd(xf[r], b, c) <= T5[r]) hit |= 0x10000u << r;
        }
        return hit;
    };
    for (int block0 = 0; block0 < n_sub; block0 += kThreads) {
        // ---- bounds of whole sub-chunks, a thread each: the smallest g between the first and the last size (at them, or at a
        // breakpoint between them), the last one's number of segments ----
        const int n_block = min(kThreads, n_sub - block0);
        __syncthreads();
        if (tid < n_block) {
            const int first = s_begin + (block0 + tid) * kSweepSub, last = first + min(kSweepSub, s_end - first) - 1;
            const uint32_t s_last = s_at(p.G, last);
            const double sa = static_cast<double>(s_at(p.G, first)), sb = static_cast<double>(s_last);
            const int npad = p.T.npad, ia = interval_of(s_tab, npad, sa), ib = interval_of(s_tab, npad, sb);
            const double ga = gap_at(s_tab, npad, sa), gz = gap_at(s_tab, npad, sb);
            double g_min = fmin(ga, gz), g_max = fmax(fmax(ga, gz), s_tab[npad + ia]);
            for (int i = ia + 1; i <= ib; ++i) {
                g_min = fmin(g_min, s_tab[npad + i]);
                g_max = fmax(g_max, s_tab[npad + i]);
            }
            // an interpolated g is off by the rounding of the larger of its interval's ends
            const double g = fmax(fma(g_max, -0x1p-48, g_min), 0.0), k = static_cast<double>(segments(m_u, s_last, p.G.k_mode));
            s_lb[tid] = __double2float_rd(g + L);
            s_lc[tid] = __double2float_rd(fmin(g * (k - 1.0), 1.7e308));
            s_lq[tid] = __double2float_rd(fmin(g * k, 1.7e308));
            s_need[tid] = 0;
        }
        __syncthreads();
#pragma unroll 2
        for (int i = 0; i < n_block; ++i)
            if (__any_sync(kFull, rows_of(s_lb[i], s_lc[i], s_lq[i]) != 0) && lane == 0) s_need[i] = 1;
        __syncthreads();
        auto next = [&](int i) {
            while (i < n_block && !s_need[i]) ++i;
            return i;
        };
        int sub = next(0);
        if (sub < n_block) fill(block0 + sub, 0);
        __syncthreads();
        for (int buf = 0; sub < n_block; buf ^= 1) {
            const int then = next(sub + 1);
            if (then < n_block) fill(block0 + then, buf ^ 1);
            const uint32_t base = static_cast<uint32_t>(s_begin + (block0 + sub) * kSweepSub);
            const float *const gb = s_gb + buf * kSweepGroups + my_c * g_len, *const gc = s_gc + buf * kSweepGroups + my_c * g_len,
                        *const gq = s_gq + buf * kSweepGroups + my_c * g_len;
            float b_all = CUDART_INF_F, c_all = CUDART_INF_F, q_all = CUDART_INF_F;
            for (int g = 0; g < g_len; ++g) {
                if (HAS5) { b_all = fminf(b_all, gb[g]); c_all = fminf(c_all, gc[g]); }
                if (QL) q_all = fminf(q_all, gq[g]);
            }
            if (__any_sync(kFull, rows_of(b_all, c_all, q_all) != 0))
#pragma unroll 1
            for (int g = 0; g < g_len; ++g) {
                const unsigned hit = rows_of(HAS5 ? gb[g] : 0.f, HAS5 ? gc[g] : 0.f, QL ? gq[g] : 0.f);
                const int j0 = 32 * (my_c * g_len + g), gd = buf * kSweepGroups + my_c * g_len + g;
                const float *bf = s_bf + buf * kSweepSub + j0, *cf4 = s_cf + buf * kSweepSub + j0, *qf = s_qf + buf * kSweepSub + j0;
                if (__any_sync(kFull, hit != 0)) {
                    // Exact pass over the group for the flagged rows: candidates in ascending order, strict '<' (smallest s on
                    // ties).  The bounds in T only ever shrink towards the best time, so nothing that could win is passed over.
#pragma unroll 1
                    for (unsigned rows = __reduce_or_sync(kFull, hit); rows; rows &= rows - 1) {
                        const int bit = __ffs(rows) - 1, r = bit & 15;
                        const bool five = HAS5 && (bit >> 4);
                        const int P = P_of(r);
                        const double x = x_exact(P), c = c_exact(P);
                        const float xr = IS9 ? static_cast<float>(31 - __clz(P)) : __int2float_rd(P - 1), cfl = __double2float_rd(c);
                        const int o = (five && HAS2 ? kIdStep : 0) + r * 32;
                        double bt = best[o];
                        uint32_t bi = bidx[o];
                        float T = CUDART_INF_F;
#pragma unroll
                        for (int q = 0; q < R; ++q) {
                            if (HAS5 && five && q == r) T = T5[q];
                            if (QL && !five && q == r) T = T2[q];
                        }
                        // The group's candidates one by one, in FP32 and all at once: mostly none is not above.  And none is better than what
                        // this warp has, which is of a smaller size, if the FP64 line of the group's smallest coefficients is not.
                        {
                            const f32x2 x2 = splat2(xr), c2 = splat2(cfl);
                            float low = CUDART_INF_F;
#pragma unroll
                            for (int i = 0; i < 32; i += 4) {
                                f32x2x2 a, c{c2, c2};
                                if (HAS5 && five) {
                                    a = *reinterpret_cast<const f32x2x2 *>(bf + i);
                                    c = *reinterpret_cast<const f32x2x2 *>(cf4 + i);
                                } else {
                                    a = *reinterpret_cast<const f32x2x2 *>(qf + i);
                                }
                                low = min_with2(min_with2(low, fma2_down(x2, a.x, c.x)), fma2_down(x2, a.y, c.y));
                            }
                            const double t_least = five ? fma(x, s_db[gd], s_dc[gd]) : fma(x, s_dq[gd], c);
                            if (!__any_sync(kFull, low <= T && t_least < bt)) continue;
                        }
#pragma unroll 1
                        for (int i = 0; i < 32; i += 4) {
                            float t[4];
                            if (HAS5 && five) {
                                const float4 b4 = *reinterpret_cast<const float4 *>(bf + i), c4 = *reinterpret_cast<const float4 *>(cf4 + i);
                                t[0] = __fmaf_rd(xr, b4.x, c4.x); t[1] = __fmaf_rd(xr, b4.y, c4.y);
                                t[2] = __fmaf_rd(xr, b4.z, c4.z); t[3] = __fmaf_rd(xr, b4.w, c4.w);
                            } else {
                                const float4 q4 = *reinterpret_cast<const float4 *>(qf + i);
                                t[0] = __fmaf_rd(xr, q4.x, cfl); t[1] = __fmaf_rd(xr, q4.y, cfl);
                                t[2] = __fmaf_rd(xr, q4.z, cfl); t[3] = __fmaf_rd(xr, q4.w, cfl);
                            }
                            if (__any_sync(kFull, fminf(fminf(t[0], t[1]), fminf(t[2], t[3])) <= T)) {
#pragma unroll
                                for (int u = 0; u < 4; ++u) {
                                    const int e = buf * kSweepSub + j0 + i + u;
                                    const double tt = five ? fma(x, s_bc[e].x, s_bc[e].y) : fma(x, s_q[e], c);
                                    if (tt < bt) { bt = tt; bi = base + j0 + i + u; }
                                }
                                T = fminf(T, __double2float_ru(bt));
                            }
                        }
                        best[o] = bt;
                        bidx[o] = bi;
#pragma unroll
                        for (int q = 0; q < R; ++q) {
                            if (HAS5 && five && q == r) T5[q] = T;
                            if (QL && !five && q == r) T2[q] = T;
                        }
                    }
                }
            }
            sub = then;
            __syncthreads();
        }
    }

    // partial results, one row per (table, strategy slot, (m, chunk) pair), P contiguous; the warps that shared a tile of
    // process counts hand over the smallest (time, s) of theirs
#pragma unroll
    for (int q = 0; q < kNid; ++q) {
        const int slot = IS9 ? p.n_seg - 1 : q;
        const size_t rbase = (static_cast<size_t>(trel) * p.n_seg + slot) * p.n_pairs + row;
        for (int i = tid; i < wp * 32 * R; i += kThreads) {
            const int pidx = tile0 + i;
            if (pidx >= p.G.n_P) break;
            double bt = s_best[q * kIdStep + i];
            uint32_t bi = s_idx[q * kIdStep + i];
            for (int w = 1; w < wc; ++w) {
                const double t = s_best[q * kIdStep + w * wp * 32 * R + i];
                const uint32_t e = s_idx[q * kIdStep + w * wp * 32 * R + i];
                if (t < bt || (t == bt && e < bi)) { bt = t; bi = e; }
            }
            p.part_time[rbase * p.G.n_P + pidx] = bt;
            p.part_idx[rbase * p.G.n_P + pidx] = bi;
        }
    }
    last_block_waits(tid);
}

// ------------------------------------------------------------------------------------------
// Fused evaluation: all strategies, strategy selection, stores
// ------------------------------------------------------------------------------------------

// table | Scatter Binomial sums [lc_max][32] | Scatter Chain [2][warps][32]
static size_t fused_smem_bytes(const TableDev &T, const GridDev &G)
{
    return (3 * static_cast<size_t>(T.npad) + static_cast<size_t>(G.lc_max) * 32 + 2 * kWarps * 32) * sizeof(double);
}

// (Four warps per CTA instead of eight halve the set-up per process count and are 1 to 25 % slower, whatever the grid.)
template <bool PREDICT>
__global__ void __launch_bounds__(kThreads, 2) fused_kernel(const FusedParams p)
{
    constexpr int R = kFusedR;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    double *const s_tab = reinterpret_cast<double *>(smem_raw);
    const int npad = p.T.npad;
    const uint32_t mask = p.G.mask;
    double *const s_cum = s_tab + 3 * npad, *const s_tot = s_cum + p.G.lc_max * 32;

    int b = blockIdx.x;
    const int mtile = b % p.n_mtiles;
    b /= p.n_mtiles;
    const int ptile = b % p.n_ptiles;
    const int trel = b / p.n_ptiles;
    const int table = p.table0 + trel;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int midx = mtile * 32 + lane;
    const bool m_ok = midx < p.G.n_m;
    const int midx_c = min(midx, p.G.n_m - 1);
    const uint32_t m_u = p.G.m_list[midx_c];
    const double md = static_cast<double>(m_u);
    const int ns = p.G.ns_of_m[midx_c];

    dependents_may_start();
    const double L = p.T.lat[table];
    stage_table(s_tab, p.T, table);
    if (p.part_time) wait_for_kernel_in_front();  // the partial minima
    __syncthreads();

    const double g1 = gap_at_one(s_tab, npad);
    const double gm = gap_at(s_tab, npad, md);

    // Scatter Binomial Tree: running sums of g(2^j m), j = 0..lc_max-1 (Table 2, third row)
    // (the gaps are looked up by all warps, one j per warp at a time; warp 0 then adds them up)
    if ((mask >> 12) & 1u) {
        for (int d = warp; d < p.G.lc_max; d += kWarps)
            s_cum[d * 32 + lane] = gap_at(s_tab, npad, md * static_cast<double>(1ull << d));
        __syncthreads();
        if (warp == 0) {
            double acc = 0.0;
            for (int d = 0; d < p.G.lc_max; ++d) {
                acc += s_cum[d * 32 + lane];
                s_cum[d * 32 + lane] = acc;
            }
        }
    }
    __syncthreads();

    // Process counts of the tile: warp w owns the contiguous run [w * run_len, (w + 1) * run_len), R of them
    // per pass, so that the Scatter Chain sum can run along a thread without a barrier per pass.
    const int run_len = p.passes_per_tile * R;
    const int p_warp = ptile * (kWarps * run_len) + warp * run_len;

    // Scatter Chain: the sum of g(j m) in front of this thread's run, then a walk along it
    double s1_run = 0.0, j_last = 0.0;
    ChainWalk s1_walk;
    if ((mask >> 11) & 1u) {
        const int c0 = ptile * (kWarps * run_len), e0 = min(p_warp, p.G.n_P), e1 = min(p_warp + run_len, p.G.n_P);
        chain_front_parts(s_tab, npad, p.T.n_bp, p.G.P_list, p.G.P_lo, md, c0, e0, e1, warp, kWarps, s_tot + lane, s_tot + kWarps * 32 + lane, 32);
        __syncthreads();
        if (e0 < e1) {
            s1_run = chain_front_sum(s_tot + lane, s_tot + kWarps * 32 + lane, 32, warp, kWarps);
            j_last = static_cast<double>(warp == 0 ? P_at(p.G, e0) - 2 : P_at(p.G, e0 - 1) - 1);
            s1_walk.start(s_tab, npad, (j_last + 1.0) * md);
        }
    }

    const size_t plane = static_cast<size_t>(p.G.n_P) * p.G.n_m;

    for (int pass = 0; pass < p.passes_per_tile; ++pass) {
        const int p0 = p_warp + pass * R;
        if (p0 >= p.G.n_P) break;  // this warp's run is exhausted (no barriers below)

        int Pv[R];
        bool ok[R];
        double pm1[R];
#pragma unroll
        for (int r = 0; r < R; ++r) {
            ok[r] = (p0 + r) < p.G.n_P;
            Pv[r] = P_at(p.G, min(p0 + r, p.G.n_P - 1));
            pm1[r] = static_cast<double>(Pv[r] - 1);
        }

        // ---- Scatter Chain: running sum of g(j m) along the thread's run ----
        double s1sum[R];
        if ((mask >> 11) & 1u) {
#pragma unroll
            for (int r = 0; r < R; ++r) {
                if (ok[r]) {
                    s1_run += j_last + 1.0 == pm1[r] ? s1_walk.at(s_tab, npad, pm1[r] * md) : s1_walk.range(s_tab, npad, md, j_last + 1.0, pm1[r]);
                    j_last = pm1[r];
                }
                s1sum[r] = s1_run;
            }
        }

        // ---- running decision per cell (strict '<' in ascending id keeps the lowest id on ties) ----
        double bt[R];
        uint32_t bsz[R];
        int bid[R];
#pragma unroll
        for (int r = 0; r < R; ++r) { bt[r] = CUDART_INF; bsz[r] = 0; bid[r] = 255; }

        auto out_index = [&](int id_or_coll, int planes, int r) {
            return (static_cast<size_t>(table - p.out_table0) * planes + id_or_coll) * plane +
                   static_cast<size_t>(p0 + r) * p.G.n_m + midx;
        };
        // Predictions: one pointer per row into the table's first plane; a strategy's plane is id * plane further on.
        // Rows past the last process count and lanes past the last message size compute the last valid cell again
        // (their indices are clamped), so they store the same value to the same address: no predicates on the stores.
        unsigned char *row_t[R];
        if (PREDICT) {
            const size_t tab0 = static_cast<size_t>(table - p.out_table0) * 13 * plane + midx_c;
#pragma unroll
            for (int r = 0; r < R; ++r)
                row_t[r] = reinterpret_cast<unsigned char *>(p.p_time + (tab0 + static_cast<size_t>(min(p0 + r, p.G.n_P - 1)) * p.G.n_m));
        }
        const size_t plane_bytes = plane * sizeof(double);
        auto consider = [&](int id, const double *val, const uint32_t *sval) {
#pragma unroll
            for (int r = 0; r < R; ++r) {
                if (PREDICT) {
                    *reinterpret_cast<double *>(row_t[r] + id * plane_bytes) = val[r];
                } else if (val[r] < bt[r]) {
                    bt[r] = val[r];
                    bid[r] = id;
                    bsz[r] = sval ? sval[r] : 0u;
                }
            }
        };
        auto flush = [&](int coll) {
            if constexpr (!PREDICT) {
#pragma unroll
                for (int r = 0; r < R; ++r) {
                    if (ok[r] && m_ok) {
                        const size_t o = out_index(coll == 0 ? p.om.plane_bcast : p.om.plane_scat, p.om.planes, r);
                        p.d_strategy[o] = bid[r] < 16 ? p.om.id_of[bid[r]] : static_cast<uint8_t>(bid[r]);
                        p.d_sbytes[o] = bsz[r];
                        p.d_time[o] = bt[r];
                    }
                    bt[r] = CUDART_INF; bsz[r] = 0; bid[r] = 255;
                }
            }
        };

        // Segmented model `id` (slot = its rank among the enabled segmented ids) reduced over
        // the candidates: a[r] * coef1 + c[r] (ids 2, 9) or a[r] * B + C (id 5).
        auto segmented = [&](int id, int seg_rank, int slot, const double *a, const double *c, bool two_coef) {
            double st[R];
            uint32_t si_best[R], sb[R];
#pragma unroll
            for (int r = 0; r < R; ++r) { st[r] = CUDART_INF; si_best[r] = 0; }
            if (ns == 0) {
                // no candidate fits: the message goes whole (s = m, k = 1)
#pragma unroll
                for (int r = 0; r < R; ++r) {
                    st[r] = two_coef ? fma(a[r], gm + L, 0.0) : fma(a[r], gm, c[r]);
                    sb[r] = m_u;
                }
            } else {
                // partial minima from the sweep kernel, chunks in ascending candidate order
                const int r0 = p.pair_base[midx_c], r1 = p.pair_base[midx_c + 1];
                for (int row = r0; row < r1; ++row) {
                    const size_t rb = ((static_cast<size_t>(trel) * p.n_seg + slot) * p.n_pairs + row) * p.G.n_P;
#pragma unroll
                    for (int r = 0; r < R; ++r) {
                        const int pr = min(p0 + r, p.G.n_P - 1);  // rows past the end repeat the last one
                        const double t = p.part_time[rb + pr];
                        if (t < st[r]) { st[r] = t; si_best[r] = p.part_idx[rb + pr]; }
                    }
                }
#pragma unroll
                for (int r = 0; r < R; ++r) sb[r] = s_at(p.G, static_cast<int>(si_best[r]));
            }
            if (PREDICT && p.p_best_s) {
#pragma unroll
                for (int r = 0; r < R; ++r)
                    if (ok[r] && m_ok) p.p_best_s[out_index(seg_rank, 3, r)] = sb[r];
            }
            consider(id, st, sb);
        };

        double v[R], lf[R], lc[R], lcL[R];
#pragma unroll
        for (int r = 0; r < R; ++r) {
            lf[r] = static_cast<double>(31 - __clz(Pv[r]));
            lc[r] = static_cast<double>(32 - __clz(Pv[r] - 1));
            lcL[r] = lc[r] * L;
        }
        double Lr[R];
#pragma unroll
        for (int r = 0; r < R; ++r) Lr[r] = L;
        const double rdv = 2.0 * g1 + 3.0 * L;  // rendezvous handshake: 2 g(1) + 3 L
        int slot = 0;

        // ---- Broadcast, Table 1 ----
        if (mask & 1u) {  // Flat Tree
#pragma unroll
            for (int r = 0; r < R; ++r) v[r] = fma(pm1[r], gm, L);
            consider(0, v, nullptr);
        }
        if ((mask >> 1) & 1u) {  // Flat Tree Rendezvous
#pragma unroll
            for (int r = 0; r < R; ++r) v[r] = fma(pm1[r], gm, rdv);
            consider(1, v, nullptr);
        }
        if ((mask >> 2) & 1u) segmented(2, 0, slot++, pm1, Lr, false);  // Segmented Flat Tree
        if ((mask >> 3) & 1u) {  // Chain
#pragma unroll
            for (int r = 0; r < R; ++r) v[r] = pm1[r] * (gm + L);
            consider(3, v, nullptr);
        }
        if ((mask >> 4) & 1u) {  // Chain Rendezvous
#pragma unroll
            for (int r = 0; r < R; ++r) v[r] = pm1[r] * (gm + rdv);
            consider(4, v, nullptr);
        }
        if ((mask >> 5) & 1u) segmented(5, 1, slot++, pm1, nullptr, true);  // Segmented Chain
        if ((mask >> 6) & 1u) {  // Binary Tree (the printed bound)
#pragma unroll
            for (int r = 0; r < R; ++r) v[r] = lc[r] * fma(2.0, gm, L);
            consider(6, v, nullptr);
        }
        if ((mask >> 7) & 1u) {  // Binomial Tree
#pragma unroll
            for (int r = 0; r < R; ++r) v[r] = fma(lf[r], gm, lcL[r]);
            consider(7, v, nullptr);
        }
        if ((mask >> 8) & 1u) {  // Binomial Tree Rendezvous
#pragma unroll
            for (int r = 0; r < R; ++r) v[r] = fma(lf[r], gm, lc[r] * rdv);
            consider(8, v, nullptr);
        }
        if ((mask >> 9) & 1u) segmented(9, 2, slot++, lf, lcL, false);  // Segmented Binomial Tree
        if (mask & 0x3FFu) flush(0);

        // ---- Scatter, Table 2 ----
        if ((mask >> 10) & 1u) {  // Flat Tree
#pragma unroll
            for (int r = 0; r < R; ++r) v[r] = fma(pm1[r], gm, L);
            consider(10, v, nullptr);
        }
        if ((mask >> 11) & 1u) {  // Chain
#pragma unroll
            for (int r = 0; r < R; ++r) v[r] = fma(pm1[r], L, s1sum[r]);
            consider(11, v, nullptr);
        }
        if ((mask >> 12) & 1u) {  // Binomial Tree
#pragma unroll
            for (int r = 0; r < R; ++r) v[r] = s_cum[(32 - __clz(Pv[r] - 1) - 1) * 32 + lane] + lcL[r];
            consider(12, v, nullptr);
        }
        if (mask & 0x1C00u) flush(1);
    }
    last_block_waits(tid);
}

// ------------------------------------------------------------------------------------------
// FP64 issue-rate probe (measurement aid)
// ------------------------------------------------------------------------------------------

// 16 independent chains per thread: with fewer, the loop's own counter and branch take issue slots from
// the DFMAs (8 chains reach 0.92 of the 64-lanes-per-SM rate, 12 or more reach 0.997).
constexpr int kProbeChains = 16;
__global__ void __launch_bounds__(kThreads) fp64_probe_kernel(double *sink, int iters)
{
    double a[kProbeChains];
    const double x = 1.0 + 1e-9 * threadIdx.x, y = 1e-12 * blockIdx.x;
#pragma unroll
    for (int i = 0; i < kProbeChains; ++i) a[i] = 0.5 + i;
    for (int it = 0; it < iters; ++it) {
#pragma unroll
        for (int u = 0; u < 2; ++u) {
#pragma unroll
            for (int i = 0; i < kProbeChains; ++i) a[i] = fma(a[i], x, y);
        }
    }
    double s = 0.0;
#pragma unroll
    for (int i = 0; i < kProbeChains; ++i) s += a[i];
    if (s == 1234.5678) sink[0] = s;  // keeps the chains alive; practically never true
}

// ------------------------------------------------------------------------------------------
// Launch wrappers
// ------------------------------------------------------------------------------------------

cudaError_t launch_fused(const FusedParams &p, bool predict, bool overlap, cudaStream_t st)
{
    const size_t smem = fused_smem_bytes(p.T, p.G);
    const long long blocks = static_cast<long long>(p.n_mtiles) * p.n_ptiles * p.n_tables_launch;
    if (blocks <= 0 || blocks > 0x7FFFFFFFLL) return cudaErrorInvalidConfiguration;
    return launch(predict ? fused_kernel<true> : fused_kernel<false>, static_cast<unsigned>(blocks), 1, kThreads, smem, st, overlap, p);
}

template <bool HAS2, bool HAS5, bool IS9>
static cudaError_t launch_sweep_t(const SweepParams &p, int n_tables_launch, bool overlap, cudaStream_t st)
{
    constexpr int n_id = (HAS2 ? 1 : 0) + (HAS5 ? 1 : 0) + (IS9 ? 1 : 0);
    const size_t smem = 3 * static_cast<size_t>(p.T.npad) * sizeof(double) +
                        2 * kSweepSub * (sizeof(double2) + sizeof(double) + 3 * sizeof(float)) + 2 * kSweepGroups * 3 * (sizeof(double) + sizeof(float)) + kThreads * 3 * sizeof(float) + kThreads * sizeof(int) +
                        static_cast<size_t>(n_id) * kWarps * kSweepR * 32 * (sizeof(double) + sizeof(uint32_t));
    const long long bx = static_cast<long long>(p.n_pairs) * p.n_ptiles;
    if (bx <= 0 || bx > 0x7FFFFFFFLL || n_tables_launch > 65535) return cudaErrorInvalidConfiguration;
    return launch(sweep_kernel<HAS2, HAS5, IS9>, static_cast<unsigned>(bx), static_cast<unsigned>(n_tables_launch), kThreads, smem, st, overlap, p);
}

// Ids 2 and 5 share a launch (one set of coefficients, lines in P); id 9, whose lines are in floor(log2 P), has its own.
cudaError_t launch_sweep(const SweepParams &p, int n_tables_launch, int *launches, cudaStream_t st)
{
    const bool has2 = (p.G.mask >> 2) & 1, has5 = (p.G.mask >> 5) & 1, has9 = (p.G.mask >> 9) & 1;
    cudaError_t e = cudaSuccess;
    *launches = 0;
    if (has2 || has5) {
        e = has2 && has5 ? launch_sweep_t<true, true, false>(p, n_tables_launch, false, st)
                         : (has2 ? launch_sweep_t<true, false, false>(p, n_tables_launch, false, st) : launch_sweep_t<false, true, false>(p, n_tables_launch, false, st));
        if (e != cudaSuccess) return e;
        ++*launches;
    }
    if (has9) {
        e = launch_sweep_t<false, false, true>(p, n_tables_launch, has2 || has5, st);
        if (e == cudaSuccess) ++*launches;
    }
    return e;
}

cudaError_t launch_fp64_probe(double *d_sink, int iters, int blocks, cudaStream_t st)
{
    fp64_probe_kernel<<<blocks, kThreads, 0, st>>>(d_sink, iters);
    return cudaGetLastError();
}

}  // namespace plogp
