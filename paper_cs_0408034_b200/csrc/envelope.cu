// envelope_kernel: the segment-size search of Section 3.1 without visiting every (P, m, s) cell.
//
// For a fixed message size m every segmented model of Table 1 is a line in x = P-1 (or in floor(log2 P)):
//   id 2: fma(P-1, Q, L)              Q = g(s) k
//   id 9: fma(floor(log2 P), Q, ceil(log2 P) L)
//   id 5: fma(P-1, B, C)              B = g(s) + L, C = g(s) (k-1)
// Ids 2 and 9 have non-negative multipliers, and a rounded fused multiply-add is monotone in Q, so
// their minimum over s is attained by the smallest Q for every P at once: one reduction per m.
// For id 5 the minimum over s is the lower envelope of the lines.  When g does not decrease along the
// candidate sizes (the host only selects this kernel for such tables) two facts hold:
//   * among candidates with the same segment count k the smallest s has the smallest B and C, so
//     only the first candidate of every run of equal k can ever win (its "representative"), for id 5 as for ids 2 and 9;
//   * the representatives are sorted by slope B, hence the index of the winner does not grow with P:
//     the winners at two process counts bracket the winners at all counts in between.  Rounded times keep that up to lines
//     that differ by rounding, so a bracket ends where times are further off than that (envelope_near, device_common.cuh).
// Where the candidates are equally spaced the representatives are found without visiting the others: below
// s = sqrt(m step) almost every candidate has a segment count of its own and is looked at, above it the counts are few
// and the first candidate of each is computed (4096 instead of 262144 candidates for m = 16 MB and every multiple of
// 4 B up to 1 MB: 298 -> 22 us for 128 message sizes).
// The kernel therefore (A) lists the representatives in shared memory, (B) finds the range of the best entries at a sequence of
// coarse process-count indices (all of the first 16, then ever wider apart up to `2 << coarse_log`: the winner moves fastest
// where P is small), every eighth over the whole list, the others between those, and (C) searches, for each
// process count, only the bracket given by its two coarse neighbours.  All comparisons are the exact ones of the
// exhaustive search: (time, s) in lexicographic order.
//
// One CTA per (table, m).  Results go to the scratch layout that the sweep kernel uses, one row per
// message size: [table][strategy slot][m][P] times and candidate indices; fused_kernel reads them.
#include "device_common.cuh"

namespace plogp {

namespace {

constexpr unsigned kFull = 0xffffffffu;
constexpr int kPad = 128;  // entries behind the list of representatives that never win

// coarse number c <-> process-count index: 0..15, then runs of 8 with distances 2, 4, 8, .. up to 2 << g_max, which stays
__device__ __forceinline__ int coarse_index(int c, int g_max)
{
    if (c < 16) return c;
    const int g = min((c - 16) >> 3, g_max);
    return (16 << g) + (c - 16 - 8 * g) * (2 << g);
}

}  // namespace

__host__ __device__ int envelope_coarse_of(int pidx, int g_max)
{
    if (pidx < 16) return pidx;
    int g = 0;
    while (g < g_max && (32 << g) <= pidx) ++g;
    return 16 + 8 * g + (pidx - (16 << g)) / (2 << g);
}

__global__ void __launch_bounds__(1024) envelope_kernel(const EnvParams p)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int npad = p.T.npad, T = blockDim.x, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, n_warps = T >> 5;
    double *s_tab = reinterpret_cast<double *>(smem_raw);
    double2 *s_line = reinterpret_cast<double2 *>(s_tab + 3 * npad);         // [rep_cap + kPad] (B, C)
    double *s_redt = reinterpret_cast<double *>(s_line + p.rep_cap + kPad);  // [32]
    uint32_t *s_I = reinterpret_cast<uint32_t *>(s_redt + 32);        // [rep_cap] candidate index of an entry
    uint32_t *s_k = s_I + p.rep_cap;                                  // [T] exchange of k
    unsigned *s_near = s_k + T;                                       // [max_coarse] first and (<< 16) last of the best entries
    int *s_cnt = reinterpret_cast<int *>(s_near + p.max_coarse);      // [32] + [32]

    const int midx = blockIdx.x, trel = blockIdx.y, table = p.table0 + trel;
    dependents_may_start();
    const uint32_t m_u = p.G.m_list[midx];
    const int ns = p.G.ns_of_m[midx];
    if (ns == 0) return;  // no candidate fits: the consumer evaluates the whole message itself
    const uint32_t mask = p.G.mask;
    const bool has2 = (mask >> 2) & 1u, has5 = (mask >> 5) & 1u, has9 = (mask >> 9) & 1u;
    const int slot2 = 0, slot5 = has2 ? 1 : 0, slot9 = slot5 + (has5 ? 1 : 0);
    const int n_P = p.G.n_P;
    auto out_row = [&](int slot) { return ((static_cast<size_t>(trel) * p.n_seg + slot) * p.G.n_m + midx) * n_P; };

    stage_table(s_tab, p.T, table);
    __syncthreads();
    const double L = p.T.lat[table];

    // ---- (A) one pass over the candidates: smallest Q, and the representatives of window `win` ----
    double qmin = CUDART_INF;
    int qidx = 0x7FFFFFFF;
    int n_rep = 0;  // all representatives (of every window), known after the first pass
    constexpr int V = 4;  // consecutive items per thread and chunk (independent searches and divisions in flight)
    // Items in ascending order of s: the first n_low candidates, then (equally spaced candidates only) one item for every
    // smaller segment count.  An item is a representative if its candidate's count differs from the one in front of it.
    int n_low = ns, n_items = ns;
    uint32_t k_low = 0;  // segment count of candidate n_low - 1
    if (!p.G.s_list) {
        n_low = min(ns, static_cast<int>(sqrtf(static_cast<float>(m_u) / static_cast<float>(p.G.s_step))) + 1);
        k_low = segments(m_u, s_at(p.G, n_low - 1), p.G.k_mode);
        n_items = n_low + static_cast<int>(k_low - segments(m_u, s_at(p.G, ns - 1), p.G.k_mode));
    }
    auto list_pass = [&](int win) {
        int base = 0;
        uint32_t carry_k = 0;  // thread 0: k of the last item of the previous chunk
        for (int c0 = 0; c0 < n_items; c0 += V * T) {
            double gs[V];
            uint32_t k[V];
            int cand[V];
#pragma unroll
            for (int v = 0; v < V; ++v) {
                const int it = c0 + V * tid + v;
                int si = it;
                gs[v] = 0.0;
                k[v] = 0;
                bool real = it < n_items;
                uint32_t want = 0;
                if (real && it >= n_low) {
                    // the smallest candidate with at most `want` segments: s >= m / want (k = ceil), s > m / (want + 1) (k = floor)
                    want = k_low - 1u - static_cast<uint32_t>(it - n_low);
                    uint32_t t;
                    if (p.G.k_mode == 0) { t = m_u / want; t += t * want != m_u ? 1u : 0u; }
                    else t = m_u / (want + 1u) + 1u;
                    si = t <= p.G.s_lo ? 0 : static_cast<int>((static_cast<unsigned long long>(t - p.G.s_lo) + p.G.s_step - 1u) / p.G.s_step);
                    real = si < ns;
                }
                cand[v] = si;
                if (real) {
                    const uint32_t s = s_at(p.G, si);
                    k[v] = segments(m_u, s, p.G.k_mode);
                    if (it >= n_low && k[v] != want) k[v] = 0;  // no candidate has that count
                    else {
                        gs[v] = gap_at(s_tab, npad, static_cast<double>(s));
                        if (win == 0) {
                            const double Q = gs[v] * static_cast<double>(k[v]);
                            if (Q < qmin) { qmin = Q; qidx = si; }  // ascending si per thread: the smallest index stays
                        }
                    }
                }
            }
            s_k[tid] = k[V - 1];
            __syncthreads();
            uint32_t k_prev = tid > 0 ? s_k[tid - 1] : carry_k;
            unsigned rep = 0;  // bit v: candidate v starts a run of equal segment count
            int cnt = 0;
#pragma unroll
            for (int v = 0; v < V; ++v) {
                const int it = c0 + V * tid + v;
                // behind n_low every item that has a candidate is a representative
                if (it < n_items && k[v] != 0 && (it == 0 || it >= n_low || k[v] != k_prev)) { rep |= 1u << v; ++cnt; }
                k_prev = k[v];
            }
            // ordered positions: inclusive scan of the counts over the warp, then the warps' totals
            int incl = cnt;
#pragma unroll
            for (int off = 1; off < 32; off <<= 1) {
                const int y = __shfl_up_sync(kFull, incl, off);
                if (lane >= off) incl += y;
            }
            if (lane == 31) s_cnt[warp] = incl;
            if (tid == 0) carry_k = s_k[T - 1];
            __syncthreads();
            int off = 0, total = 0;
            for (int w = 0; w < n_warps; ++w) {
                const int c = s_cnt[w];
                off += w < warp ? c : 0;
                total += c;
            }
            int pos = base + off + incl - cnt - win * p.rep_cap;
#pragma unroll
            for (int v = 0; v < V; ++v) {
                if ((rep >> v) & 1u) {
                    if (pos >= 0 && pos < p.rep_cap) {
                        s_line[pos] = make_double2(gs[v] + L, fmin(gs[v] * (static_cast<double>(k[v]) - 1.0), CUDART_INF));  // inf * 0 as inf
                        s_I[pos] = static_cast<uint32_t>(cand[v]);
                    }
                    ++pos;
                }
            }
            base += total;
        }
        return base;
    };
    n_rep = list_pass(0);

    // ---- ids 2 and 9: the smallest Q (smallest s on ties) serves every process count ----
    if (has2 || has9) {
        warp_min_pair(qmin, qidx);
        if (lane == 0) { s_redt[warp] = qmin; s_cnt[32 + warp] = qidx; }
        __syncthreads();
        double q = lane < n_warps ? s_redt[lane] : CUDART_INF;
        int qi = lane < n_warps ? s_cnt[32 + lane] : 0x7FFFFFFF;
        warp_min_pair(q, qi);
        for (int pidx = tid; pidx < n_P; pidx += T) {
            const int P = P_at(p.G, pidx);
            if (has2) {
                p.part_time[out_row(slot2) + pidx] = fma(static_cast<double>(P - 1), q, L);
                p.part_idx[out_row(slot2) + pidx] = static_cast<uint32_t>(qi);
            }
            if (has9) {
                const double lf = static_cast<double>(31 - __clz(P)), lcL = static_cast<double>(32 - __clz(P - 1)) * L;
                p.part_time[out_row(slot9) + pidx] = fma(lf, q, lcL);
                p.part_idx[out_row(slot9) + pidx] = static_cast<uint32_t>(qi);
            }
        }
    }
    if (!has5) return;

    // ---- id 5: lower envelope over the representatives, one window of the list at a time ----
    const int n_c = envelope_coarse_of(n_P - 1, p.coarse_log) + 2;  // the last one stands for n_P - 1
    const int n_win = (n_rep + p.rep_cap - 1) / p.rep_cap;
    for (int win = 0; win < n_win; ++win) {
        if (win > 0) {
            __syncthreads();  // the previous window's searches are done with the list
            list_pass(win);
        }
        const int n_e = min(p.rep_cap, n_rep - win * p.rep_cap);
        for (int i = tid; i < kPad; i += T) s_line[n_e + i] = make_double2(0.0, CUDART_INF);
        __syncthreads();
        // (B) the entries whose time is within (1 + near) of the best at the coarse process counts (a few more where times
        // close in on it in steps as small as that): every eighth and the last over the whole window, then the others
        auto x_of = [&](int c) { return P_at(p.G, min(coarse_index(c, p.coarse_log), n_P - 1)) - 1; };
        // between coarse indices a and b: from the first of the best at b to the last at a
        auto bracket = [&](int a, int b, int &lo, int &hi) {
            hi = static_cast<int>(s_near[a] >> 16);
            lo = min(static_cast<int>(s_near[b] & 0xFFFFu), hi);
        };
#pragma unroll 1
        for (int level = 8; level >= 1; level -= 7) {
            const int n = level == 8 ? (n_c - 1 + 7) / 8 + 1 : n_c - 1;  // 0, 8, 16, .. and n_c - 1
#pragma unroll 1
            for (int i = warp; i < n; i += n_warps) {
                const int c = min(level * i, n_c - 1);
                if (level == 1 && (c & 7) == 0) continue;
                const int xi = x_of(c);
                const double x = static_cast<double>(xi), r = __fdividef(static_cast<float>(x_of(min(c + level, n_c - 1))), static_cast<float>(xi));  // to 1e-6
                int lo = 0, hi = n_e - 1;
                if (level == 1) bracket(c & ~7, min((c & ~7) + 8, n_c - 1), lo, hi);
                // What is within `near` at an index in between must be inside the bracket as well, so that of every eighth
                // is wider: twice, and by the ratio of process counts once more.
                const double near = envelope_near(level == 8 ? 2.0 * r * r : r);
                // A long range is read once, which is what this costs (16 bytes an entry out of shared memory; with the nearest
                // times in a second read of it the kernel took 45.6 us instead of 41.4): per lane the entries from the first to
                // the last whose high word is at most one above the smallest.  Those behind hi are the list's as well, then
                // kPad that never win.
                int first = lo, last = hi;
                bool on;
                if (hi - lo >= 128 && near <= 0x1p-21) {  // no more than a high word's last bit
                    int h = 0x7FFFFFFE;
                    first = n_e - 1; last = 0;
#pragma unroll 1
                    for (int e = lo + lane; e <= hi; e += 128) {
#pragma unroll
                        for (int u = 0; u < 4; ++u) {
                            const int v = __double2hiint(fma(x, s_line[e + 32 * u].x, s_line[e + 32 * u].y));
                            first = v < h - 1 ? e + 32 * u : first;  // so much better than all before that none of them counts
                            last = v <= h + 1 ? e + 32 * u : last;
                            h = min(h, v);
                        }
                    }
                    on = h <= __reduce_min_sync(kFull, h) + 1;
                    first = __reduce_min_sync(kFull, on ? first : n_e - 1);
                    last = __reduce_max_sync(kFull, on ? min(last, n_e - 1) : 0);
                }
                // of these the ones that are within `near`
                double tb = CUDART_INF, up_to = CUDART_INF;
                const int begin = first, end = last;
                first = n_e - 1; last = 0;
#pragma unroll 1
                for (int e = begin + lane; e <= end; e += 32) {
                    const double t = fma(x, s_line[e].x, s_line[e].y);
                    if (t <= up_to) {
                        const double t_up = fma(t, near, t);
                        first = t_up < tb ? e : min(first, e);
                        last = e;
                        if (t < tb) { tb = t; up_to = t_up; }
                    }
                }
                const double m = warp_min(tb);
                on = tb <= fma(m, near, m);
                first = __reduce_min_sync(kFull, on ? first : n_e - 1);
                last = __reduce_max_sync(kFull, on ? last : 0);
                if (lane == 0) s_near[c] = static_cast<unsigned>(min(first, last)) | static_cast<unsigned>(last) << 16;
            }
            __syncthreads();
        }
        // (C) every process count: the bracket of its coarse neighbours
        for (int pidx = tid; pidx < n_P; pidx += T) {
            const int c = envelope_coarse_of(pidx, p.coarse_log);
            int lo, hi;
            bracket(c, coarse_index(c, p.coarse_log) == pidx ? c : min(c + 1, n_c - 1), lo, hi);
            const double x = static_cast<double>(P_at(p.G, pidx) - 1);
            double tb = CUDART_INF;
            int eb = lo;
            for (int e = lo; e <= hi; ++e) {
                const double t = fma(x, s_line[e].x, s_line[e].y);
                if (t < tb) { tb = t; eb = e; }  // ascending e: the smallest s stays on ties
            }
            const size_t o = out_row(slot5) + pidx;
            if (win == 0 || tb < p.part_time[o]) {  // later windows hold larger s: strict '<'
                p.part_time[o] = tb;
                p.part_idx[o] = s_I[eb];
            }
        }
    }
}

size_t envelope_smem_bytes(const TableDev &T, int threads, int rep_cap, int max_coarse)
{
    return (3 * static_cast<size_t>(T.npad) + 2 * (static_cast<size_t>(rep_cap) + kPad) + 32) * sizeof(double) +
           (static_cast<size_t>(rep_cap) + threads) * sizeof(uint32_t) + (static_cast<size_t>(max_coarse) + 64) * sizeof(int);
}

cudaError_t launch_envelope(const EnvParams &p, int threads, cudaStream_t st)
{
    const size_t smem = envelope_smem_bytes(p.T, threads, p.rep_cap, p.max_coarse);
    if (p.G.n_m <= 0 || p.n_tables_launch <= 0 || p.n_tables_launch > 65535) return cudaErrorInvalidConfiguration;
    return launch(envelope_kernel, static_cast<unsigned>(p.G.n_m), static_cast<unsigned>(p.n_tables_launch), static_cast<unsigned>(threads), smem, st, false, p);
}

}  // namespace plogp
