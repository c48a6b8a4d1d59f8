// lines_block: one CTA of the Broadcast half of the decision table (Sections 1, 3.1 and 5 of the paper), or of the segmented
// planes of the predictions, for short candidate lists.  (The Scatter half has no candidate lists and goes through
// scatter_kernel.)
//
// One CTA owns one table, up to 32 consecutive message sizes (STAGED: all of the table's, up to 256) and up to 512 process counts.
// Threads are message sizes: a group of 32 (16, 8; STAGED: as many as there are) threads holds the CTA's message sizes, and the groups
// share the candidate segment sizes while lines are ruled out, then the process counts while they are evaluated.  Every store is a
// row segment of consecutive m, whatever a row's alignment.
//
// Every model of Table 1 is, for a fixed message size (and segment size), a line in P or a function of
// floor(log2 P) and ceil(log2 P) alone:
//     ids 0 1 2 3 4 5:  t = fma(P-1, a, c)
//     ids 6 7 8 9:      constant while (floor, ceil) stays, i.e. between a power of two and the next
// all of them growing with P.  The decision is the lexicographic minimum of (t, id, s) over all cells of all enabled strategies
// (the minimum over s inside a strategy and then over strategies, smallest s and lowest id on ties).  A rendezvous variant is its
// sibling with a larger summand: with both enabled the sibling's lower id wins everywhere, and the variant is left out.
//
// Most lines are ruled out for a whole range of process counts at once.  The CTA's process counts are up to kSegs segments; at
// their ends ("knots") every line is evaluated once, and the line of the smallest time is the knot's pilot.  Inside a segment
//   * a line that is above a pilot of either end at both ends is above it everywhere in between: lines.  "Above" is two units
//     of the double's high word, more than 2^-21 of the time, so rounding cannot bring them together again;
//   * (decision) a line whose time at the lower end is above the smallest time of ids 6 to 9 at the upper end is above it
//     everywhere: both grow with P, and a rounded fused multiply-add is monotone.
// What is left (a mean of 1.5 lines of 67 per warp and process count on the batched workload) is evaluated in FP64 at each process
// count and compared with the pair's time.
// Ids 2 and 9 grow with Q = g(s) k at every P, so the candidate with the smallest Q stands for all whose Q + 2 L is two units
// of the high word above its own (the relative distance of two times is smallest there); the others, hardly ever any, are
// evaluated one by one.
// Results are those of the exhaustive FP64 search, bit for bit.
//
// What bounds it: memory writes and issue, about alike.  4096 tables, P = 2..512, 128 message sizes, 32 candidates: decision half
// 0.78 ms (its bytes take 0.53; 2.04 with lanes <-> process counts, an FP32 bound of every line at every process count and winners
// transposed through shared memory), segmented planes of 1024 tables 0.46 ms (0.75).  Per message size and 511 process counts
// about 1000 warp instructions (2800 before): set-up 80, pilots and lines 250, process counts 700.  Four segments: with six the lines per process count fall
// from 1.5 to 1.2 and the time stays; 128 registers and four CTAs per SM: with five or six what spills waits behind the stores (0.87,
// 0.91 ms), and so do loads of k from global memory (0.95).
//
// STAGED: rows off the sectors cost twice (parts of sectors at both ends of every row segment); put together first they go out whole,
// but the CTA's warps wait for the one with the most lines, and its set-up and shared memory are those of all message sizes (up to
// 256).  api.cu says where, with both sides measured.
#pragma once

#include "device_common.cuh"
#include "lines_layout.h"

#include <type_traits>

namespace plogp {

namespace lines {

constexpr unsigned kFlat = 64, kChain = 65;  // codes of the unsegmented lines beside the candidates
static_assert(kMaxInlineS <= 64, "candidates are bits of two words");

__device__ __forceinline__ unsigned high(double t) { return static_cast<unsigned>(__double2hiint(t)); }  // orders times, t >= 0

__device__ __forceinline__ void cp_async8(void *smem_dst, const void *gmem_src)
{
    unsigned s = static_cast<unsigned>(__cvta_generic_to_shared(smem_dst));
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8;\n" ::"r"(s), "l"(gmem_src));
}

}  // namespace lines

// PREDICT: times and best segment sizes of ids 2, 5 and 9 instead of the decision.  STAGED: the CTA has all message sizes of the
// table, so the cells of a step are one piece of the plane; they are put together in shared memory and go out in aligned groups of
// four, whatever row they belong to.
template <bool PREDICT, bool STAGED>
__device__ __forceinline__ void lines_block(const LinesParams &p, int block, unsigned char *smem_raw)
{
    using namespace lines;
    const int npad = p.T.npad, n_s = p.G.n_s, width = p.width, threads = blockDim.x;
    Smem sm;
    layout(p.gaps ? 0 : npad, n_s, p.n_pairs, p.n_p, width, threads, STAGED, smem_raw, &sm);
    const uint32_t mask = p.G.mask;

    int b = block;
    const int mgroup = b % p.n_mgroups;
    b /= p.n_mgroups;
    const int ptile = b % p.n_ptiles;
    const int trel = b / p.n_ptiles;
    const int table = p.table0 + trel;
    const int tid = threadIdx.x, groups = threads / width, lm = tid % width;
    const bool spare = tid >= groups * width;  // STAGED: threads behind the last group only carry cells out
    const int group = spare ? 1 << 20 : tid / width;
    const int midx = mgroup * width + lm;
    const bool m_ok = midx < p.G.n_m;
    const int midx_c = min(midx, p.G.n_m - 1);  // threads past the last message size repeat it
    const int tile0 = ptile * p.n_p;
    const int n_valid = min(p.n_p, p.G.n_P - tile0);
    const int *const knot = sm.knot;
    const int pair0 = pair_of(P_at(p.G, tile0));

    dependents_may_start();

    // ---- set-up: g, k, process counts ----
    // g at the kernel's arguments: read from the gap pre-pass where the host has run it, else interpolated here
    const double *grow = p.gaps ? p.gaps + static_cast<size_t>(trel) * p.gaps_stride : nullptr;
    const double L = p.T.lat[table];
    const uint32_t m_u = p.G.m_list[midx_c];
    const int ns = p.G.ns_of_m[midx_c];
    const uint32_t s_mine = tid < n_s ? s_at(p.G, tid) : 0u;
    // Everything is in shared memory before the first result goes out: loads from global memory wait behind the stores.
    for (int c = group, n = spare ? 0 : n_s; c < n; c += groups) cp_async8(sm.k + c * width + lm, p.G.k_list + static_cast<size_t>(c) * p.G.n_m + midx_c);
    if (tid <= kKnots) sm.knot[tid] = p.knots[ptile * (kKnots + 1) + tid];
    if (!grow) stage_table(sm.tab, p.T, table);
    for (int i = tid; i < p.n_p; i += threads) {
        const int P = P_at(p.G, min(tile0 + i, p.G.n_P - 1));
        sm.row[i].x = static_cast<double>(P - 1);
        sm.row[i].pair = (pair_of(P) - pair0) * width;
    }
    for (int i = tid; i < kSegs * 2 * width; i += threads) sm.live[i] = 0u;
    for (int i = tid; i < 2 * width; i += threads) sm.near[i] = 0u;
    cp_async_wait_all();
    if (grow) wait_for_kernel_in_front();  // the gap pre-pass
    __syncthreads();
    if (tid < n_s) {
        sm.sval[tid] = s_mine;
        sm.gs[tid] = grow ? grow[1 + tid] : gap_at(sm.tab, npad, static_cast<double>(s_mine));
    }
    const double gm = grow ? grow[1 + n_s + midx_c] : gap_at(sm.tab, npad, static_cast<double>(m_u));
    const double g1 = PREDICT ? 0.0 : grow ? grow[0] : gap_at_one(sm.tab, npad);
    const double rdv = 2.0 * g1 + 3.0 * L;  // rendezvous handshake: 2 g(1) + 3 L
    __syncthreads();

    const bool has0 = mask & 1u, has2 = (mask >> 2) & 1u, has3 = (mask >> 3) & 1u, has5 = (mask >> 5) & 1u, has6 = (mask >> 6) & 1u, has7 = (mask >> 7) & 1u,
               has78 = mask & 0x180u, has9 = (mask >> 9) & 1u;
    const bool any_log = mask & 0x3C0u;
    // the Flat Tree (P-1) g(m) + L or its rendezvous form (P-1) g(m) + rdv, the Chain (P-1) (g(m) + L) or its rendezvous form
    // (P-1) (g(m) + rdv).  Where no candidate fits, id 5 is the chain itself; its rendezvous form, which is never below it, then
    // wins where the two times are equal.
    const bool chain5 = !PREDICT && ns == 0 && has5 && !has3;
    const bool flat_on = !PREDICT && (mask & 3u), chain_on = !PREDICT && ((mask & 0x18u) || chain5);
    const double flat_c = has0 ? L : rdv, chain_a = gm + (has3 || chain5 ? L : rdv);
    const int n_seg = knot[kKnots];
    auto candidate = [&](int c, double &Q, double &B, double &C) {
        const double g = sm.gs[c], k = sm.k[c * width + lm];
        Q = g * k;
        B = g + L;  // (P-1) (g(s) + L) + g(s) (k-1)
        C = g * (k - 1.0);
    };
    // one segment: the unsegmented sibling's line, whose lower id wins the tie
    auto twin = [&](int c) { return !PREDICT && has3 && sm.sval[c] == m_u; };
    const int per = (n_s + groups - 1) / groups;  // candidates per group
    const int c0 = spare ? n_s : min(group * per, n_s), c1 = min(c0 + per, n_s);

    // ---- the pilots: smallest time at each knot, but for its last bits; and the smallest Q ----
    // N: segments looked at, kSegs, or 2 where there are no more (the knots behind the last one repeat it)
    auto find_pilots = [&](auto n_tag) {
        constexpr int N = decltype(n_tag)::value;
        double x[N + 1];
        unsigned key[N + 1], qkey = 0xFFFFFFFFu;
#pragma unroll
        for (int j = 0; j <= N; ++j) { x[j] = sm.row[knot[j]].x; key[j] = 0xFFFFFFFFu; }
        auto knots = [&](double a, double c, unsigned code) {
#pragma unroll
            for (int j = 0; j <= N; ++j) key[j] = min(key[j], (high(fma(x[j], a, c)) & ~0x7Fu) | code);
        };
#pragma unroll 2
        for (int c = c0; c < c1; ++c) {
            double Q, B, C;
            candidate(c, Q, B, C);
            if (c < ns) {
                qkey = min(qkey, (high(Q) & ~0x7Fu) | static_cast<unsigned>(c));
                if (has5 && !twin(c)) knots(B, C, c);
            }
        }
        if (group == groups - 1) {
            if (flat_on) knots(gm, flat_c, kFlat);
            if (chain_on) knots(chain_a, 0.0, kChain);
        }
        if (STAGED && spare) return;
        unsigned *out = sm.key + group * (kKnots + 1) * width + lm;
        out[0] = qkey;
#pragma unroll
        for (int j = 0; j <= N; ++j) out[(j + 1) * width] = key[j];
    };
    if (n_seg <= 2) find_pilots(std::integral_constant<int, 2>{});
    else find_pilots(std::integral_constant<int, kSegs>{});
    __syncthreads();

    auto least_of = [&](int item) {
        unsigned least = 0xFFFFFFFFu;
        const unsigned *key = sm.key + item * width + lm;
        for (int g = 0; g < groups; ++g, key += (kKnots + 1) * width) least = min(least, *key);
        return least;
    };
    const int q_best = ns > 0 ? least_of(0) & 0x3Fu : 0;
    const double Qb = ns > 0 ? sm.gs[q_best] * sm.k[q_best * width + lm] : gm;
    // a pilot per group: its times at its knot and at the knots beside it, and the smallest time of ids 6 to 9 at its knot (but
    // for the candidates near id 9's best)
    for (int j = group; j <= max(n_seg, 2); j += groups) {
        const unsigned key = least_of(j + 1), code = key & 0x7Fu;
        double a = CUDART_NAN, c = CUDART_NAN;
        unsigned at = 0xFFFFFFFFu;  // nothing below the pilot's time and its bit for rounding
        if (key != 0xFFFFFFFFu) {
            at = (key | 0x7Fu) + 1u;
            if (code == kFlat) { a = gm; c = flat_c; }
            else if (code == kChain) { a = chain_a; c = 0.0; }
            else {
                double Q;
                candidate(code, Q, a, c);
            }
        }
        const Row here = sm.row[knot[j]];
        if (!PREDICT && has2) {
            const unsigned h = high(fma(here.x, Qb, L)) + 1u;
            if (h < at) { at = h; a = Qb; c = L; }
        }
        unsigned *const bar = sm.bar + lm;
        bar[j * width] = at;
        if (j < kSegs) bar[(kKnots + j) * width] = high(fma(sm.row[knot[j + 1]].x, a, c)) + 1u;
        if (j > 0) bar[(kKnots + kSegs + j - 1) * width] = high(fma(sm.row[knot[j - 1]].x, a, c)) + 1u;
        if (!PREDICT && j > 0) {
            double t = CUDART_INF;
            const int li = pair_of(P_at(p.G, tile0 + knot[j]));
            const double lf = static_cast<double>(li >> 1), lc = static_cast<double>((li >> 1) + (li & 1));
            if (has9) t = fma(lf, Qb, lc * L);
            if (has78) t = fmin(t, fma(lf, gm, lc * (has7 ? L : rdv)));
            if (has6) t = fmin(t, lc * fma(2.0, gm, L));
            bar[(kKnots + 2 * kSegs + j - 1) * width] = any_log ? high(t) : 0xFFFFFFFFu;
        }
    }
    __syncthreads();

    // ---- which lines can win where ----
    auto find_lines = [&](auto n_tag) {
        constexpr int N = decltype(n_tag)::value;
        double x[N + 1];
        unsigned at[N + 1], a1[N], b0[N], top[N];
#pragma unroll
        for (int j = 0; j <= N; ++j) { x[j] = sm.row[knot[j]].x; at[j] = sm.bar[j * width + lm]; }
#pragma unroll
        for (int i = 0; i < N; ++i) {
            a1[i] = sm.bar[(kKnots + i) * width + lm];
            b0[i] = sm.bar[(kKnots + kSegs + i) * width + lm];
            top[i] = PREDICT ? 0xFFFFFFFFu : sm.bar[(kKnots + 2 * kSegs + i) * width + lm];
        }
        const double L2 = 2.0 * L;
        // (where times overflow, all candidates are near the best)
        const unsigned q_near = isinf(fma(sm.row[n_valid - 1].x, Qb + L, L)) ? 0xFFFFFFFFu : high(Qb + L2) + 1u;
        // segments in which the line (a, c) can win: bit `bit` of each
        auto where = [&](double a, double c, unsigned bit, unsigned *live) {
            unsigned h[N + 1];
#pragma unroll
            for (int j = 0; j <= N; ++j) h[j] = high(fma(x[j], a, c));
#pragma unroll
            for (int i = 0; i < N; ++i)
                if (!((h[i] > at[i] && h[i + 1] > a1[i]) || (h[i] > b0[i] && h[i + 1] > at[i + 1]) || (!PREDICT && h[i] > top[i]))) live[i] |= bit;
        };
#pragma unroll 1
        for (int word = c0 >> 5; 32 * word < c1; ++word) {
            const int first = max(c0, 32 * word), last = min(c1, 32 * word + 32);
            unsigned live[N], near = 0;
#pragma unroll
            for (int i = 0; i < N; ++i) live[i] = 0;
#pragma unroll 2
            for (int c = first; c < last; ++c) {
                double Q, B, C;
                candidate(c, Q, B, C);
                const unsigned bit = c < ns ? 1u << (c & 31) : 0u;
                if (high(Q + L2) <= q_near) near |= bit;
                if (has5) where(B, C, twin(c) ? 0u : bit, live);
            }
            if (word == q_best >> 5) near &= ~(1u << (q_best & 31));
#pragma unroll
            for (int i = 0; i < N; ++i)
                if (live[i]) atomicOr(sm.live + (2 * i + word) * width + lm, live[i]);
            if (near) atomicOr(sm.near + word * width + lm, near);
        }
        if (!PREDICT && group == groups - 1) {
            unsigned f[N];
#pragma unroll
            for (int i = 0; i < N; ++i) f[i] = 0;
            if (flat_on) where(gm, flat_c, 1u, f);
            if (has2 && !(has0 && (ns == 0 || sm.sval[q_best] == m_u))) where(Qb, L, 2u, f);
            if (chain_on) where(chain_a, 0.0, 4u, f);
#pragma unroll
            for (int i = 0; i < N; ++i) sm.flat[i * width + lm] = static_cast<uint8_t>(f[i]);
        }
    };
    if (n_seg <= 2) find_lines(std::integral_constant<int, 2>{});
    else find_lines(std::integral_constant<int, kSegs>{});
    __syncthreads();

    // ---- the best of ids 6 to 9 per (floor, ceil) pair ----
    const uint32_t near0 = sm.near[lm], near1 = sm.near[width + lm];
    auto near = [&](int word) { return word ? near1 : near0; };
    const uint32_t q_size = ns > 0 ? sm.sval[q_best] : m_u;
    if (!PREDICT || has9) {
        const uint8_t id9 = p.om.id_of[9], id78 = p.om.id_of[has7 ? 7 : 8], id6 = p.om.id_of[6];
        const double L78 = has7 ? L : rdv, g6 = fma(2.0, gm, L);
        const int pairs = pair_of(P_at(p.G, tile0 + n_valid - 1)) - pair0 + 1;
        for (int pr = group; pr < pairs; pr += groups) {
            const int li = pair0 + pr;
            const double lf = static_cast<double>(li >> 1), lc = static_cast<double>((li >> 1) + (li & 1)), lcL = lc * L;
            double t = CUDART_INF;
            uint32_t sz = 0;
            uint8_t who = 255;
            if (has9) {  // floor(log2 P) g(s) k + ceil(log2 P) L
                t = fma(lf, Qb, lcL);
                sz = q_size;
                who = id9;
                if (near0 | near1) {
                    int cb = q_best;
                    for (int w = 0; w < 2; ++w)
                        for (uint32_t bits = near(w); bits; bits &= bits - 1) {
                            const int c = 32 * w + __ffs(bits) - 1;
                            double Q, B, C;
                            candidate(c, Q, B, C);
                            const double v = fma(lf, Q, lcL);
                            if (v < t || (v == t && c < cb)) { t = v; cb = c; }
                        }
                    sz = sm.sval[cb];
                }
            }
            // lower ids win ties: in descending order, '<='
            if (!PREDICT && has78) {  // Binomial Tree floor(log2 P) g(m) + ceil(log2 P) L, or with rdv for L
                const double v = fma(lf, gm, lc * L78);
                if (v <= t) { t = v; sz = 0; who = id78; }
            }
            if (!PREDICT && has6) {  // Binary Tree (the printed bound): ceil(log2 P) (2 g(m) + L)
                const double v = lc * g6;
                if (v <= t) { t = v; sz = 0; who = id6; }
            }
            sm.pair_t[pr * width + lm] = t;
            sm.pair_s[pr * width + lm] = sz;
            if (!PREDICT) sm.pair_id[pr * width + lm] = who;
        }
    }
    __syncthreads();

    // ---- the process counts: eight consecutive ones per step, from the lines that can win there ----
    const size_t plane = static_cast<size_t>(p.G.n_P) * p.G.n_m;
    const uint32_t n_m = p.G.n_m;
    // candidates of a word in descending order
    auto each = [&](uint32_t bits, int word, auto &&f) {
        while (bits) {
            const int c = 31 - __clz(bits);
            bits ^= 1u << c;
            f(c + 32 * word);
        }
    };
    auto rows_out = [&](auto *out, auto &&value, int n) {  // row r is n_m elements further on
        using V = std::remove_pointer_t<decltype(out)>;
        char *const base = reinterpret_cast<char *>(out);
        if (n == kRows) {
#pragma unroll
            for (int r = 0; r < kRows; ++r) *reinterpret_cast<V *>(base + static_cast<uint64_t>(n_m) * (r * sizeof(V))) = static_cast<V>(value(r));
        } else {
#pragma unroll
            for (int r = 0; r < kRows; ++r)
                if (r < n) *reinterpret_cast<V *>(base + static_cast<uint64_t>(n_m) * (r * sizeof(V))) = static_cast<V>(value(r));
        }
    };
    const uint32_t id2 = p.om.id_of[2], id5 = p.om.id_of[5], id_chain = p.om.id_of[chain5 ? 5 : has3 ? 3 : 4], id_flat = p.om.id_of[has0 ? 0 : 1];
    // STAGED: a group of four cells w .. w + 3 of the step's, aligned in the plane; those at either end go one by one
    auto carry = [&](auto *out, const auto *in, int w, int begin, int end) {
        using V = std::remove_pointer_t<decltype(out)>;
        if (w >= begin && w + 4 <= end) {
            if constexpr (sizeof(V) == 8) store4(out + w, in + w);
            else if constexpr (sizeof(V) == 4) *reinterpret_cast<uint4 *>(out + w) = *reinterpret_cast<const uint4 *>(in + w);
            else *reinterpret_cast<uint32_t *>(out + w) = *reinterpret_cast<const uint32_t *>(in + w);
        } else {
            for (int i = max(w, begin); i < min(w + 4, end); ++i) out[i] = in[i];
        }
    };
    int seg = 0;
    for (int step = 0; step < n_valid; step += groups * kRows) {
        const int r0 = step + group * kRows;
        const bool on = !spare && r0 < n_valid;
        if (!STAGED && !on) break;
        const int step_rows = min(groups * kRows, n_valid - step);
        const int step_cells = step_rows * p.G.n_m;
        if (on) while (r0 > knot[seg + 1]) ++seg;
        const int n = min(kRows, n_valid - r0);
        const size_t o = static_cast<size_t>(tile0 + r0) * n_m + midx, o_step = static_cast<size_t>(tile0 + step) * n_m;
        const Row *const row = sm.row + (on ? r0 : 0);  // the rows behind the last process count repeat it
        // row r of this thread among the step's cells, which begin at a plane's cell `first`
        auto put = [&](auto *out, size_t first, auto &&value) {
            auto *cell = out + (static_cast<int>(first & 3u) + group * kRows * width + lm);
            if (n == kRows) {
#pragma unroll
                for (int r = 0; r < kRows; ++r) cell[r * width] = static_cast<std::remove_pointer_t<decltype(out)>>(value(r));
            } else {
                for (int r = 0; r < kRows; ++r)
                    if (r < n) cell[r * width] = static_cast<std::remove_pointer_t<decltype(out)>>(value(r));
            }
        };
        double t[kRows], x[kRows];
        uint32_t s[kRows];
        if constexpr (!PREDICT) {
            const size_t plane0 = (static_cast<size_t>(table - p.out_table0) * p.om.planes + p.om.plane_bcast) * plane;
            if (on) {
                const unsigned f = sm.flat[seg * width + lm];
                const uint32_t live0 = sm.live[2 * seg * width + lm], live1 = n_s > 32 ? sm.live[(2 * seg + 1) * width + lm] : 0u;
                const int pair = row[0].pair + lm;
                const bool one_pair = row[0].pair == row[kRows - 1].pair;
                const double tp = sm.pair_t[pair];
                const uint32_t sp = sm.pair_s[pair], ip = sm.pair_id[pair];
                auto result = [&](auto &&time, auto &&size, auto &&id) {
                    if constexpr (STAGED) {
                        put(sm.out_t, plane0 + o_step, time);
                        put(sm.out_s, plane0 + o_step, size);
                        put(sm.out_id, plane0 + o_step, id);
                    } else if (m_ok) {
                        rows_out(p.d_time + plane0 + o, time, n);
                        rows_out(p.d_sbytes + plane0 + o, size, n);
                        rows_out(p.d_strategy + plane0 + o, id, n);
                    }
                };
                const bool lines_here = (f | live0 | live1 | near0 | near1) != 0;
                // (a warp of one group goes the same way)
                if (one_pair && !(!STAGED && width == 32 ? __any_sync(0xffffffffu, lines_here) : lines_here)) {
                    result([&](int) { return tp; }, [&](int) { return sp; }, [&](int) { return ip; });
                } else {
                    uint32_t id[kRows];
#pragma unroll
                    for (int r = 0; r < kRows; ++r) { x[r] = row[r].x; t[r] = tp; s[r] = sp; id[r] = ip; }
                    if (!one_pair) {
#pragma unroll
                        for (int r = 1; r < kRows; ++r) {
                            const int q = row[r].pair + lm;
                            t[r] = sm.pair_t[q]; s[r] = sm.pair_s[q]; id[r] = sm.pair_id[q];
                        }
                    }
                    // the lower id and size wins ties: in descending order, '<='
                    auto line = [&](double a, double c, uint32_t sz, uint32_t who) {
                        if (fma(x[0], a, c) > t[kRows - 1]) return;  // all times grow with P: behind the best everywhere here
#pragma unroll
                        for (int r = 0; r < kRows; ++r) {
                            const double v = fma(x[r], a, c);
                            if (!(v > t[r])) { t[r] = v; s[r] = sz; id[r] = who; }
                        }
                    };
#pragma unroll 1
                    for (int w = n_s > 32 ? 1 : 0; w >= 0; --w)
                        each(w ? live1 : live0, w, [&](int c) {
                            double Q, B, C;
                            candidate(c, Q, B, C);
                            line(B, C, sm.sval[c], id5);
                        });
                    if (f & 4u) {
#pragma unroll 1
                        for (int again = chain5 && (mask & 0x10u) ? 1 : 0, i = 0; i <= again; ++i)
                            line(i ? gm + rdv : chain_a, 0.0, chain5 && !i ? m_u : 0u, i ? static_cast<uint32_t>(p.om.id_of[4]) : id_chain);
                    }
                    if (has2) {
                        if (near0 | near1) {
#pragma unroll 1
                            for (int w = 1; w >= 0; --w)
                                each(near(w) | ((f & 2u) && q_best >> 5 == w ? 1u << (q_best & 31) : 0u), w, [&](int c) {
                                    double Q, B, C;
                                    candidate(c, Q, B, C);
                                    line(Q, L, sm.sval[c], id2);
                                });
                        } else if (f & 2u) {
                            line(Qb, L, q_size, id2);
                        }
                    }
                    if (f & 1u) line(gm, flat_c, 0u, id_flat);
                    result([&](int r) { return t[r]; }, [&](int r) { return s[r]; }, [&](int r) { return id[r]; });
                }
            }
            if constexpr (STAGED) {
                __syncthreads();
                const int begin = static_cast<int>((plane0 + o_step) & 3u), end = begin + step_cells;
                const size_t at = plane0 + o_step - begin;
                for (int w = 4 * tid; w < end; w += 4 * threads) {
                    carry(p.d_time + at, sm.out_t, w, begin, end);
                    carry(p.d_sbytes + at, sm.out_s, w, begin, end);
                    carry(p.d_strategy + at, sm.out_id, w, begin, end);
                }
                __syncthreads();
            }
        } else {
            const size_t time0 = static_cast<size_t>(table - p.out_table0) * 13 * plane, size0 = static_cast<size_t>(table - p.out_table0) * 3 * plane;
            auto store = [&](int strategy, int w) {
                const size_t plane_t = time0 + strategy * plane, plane_s = size0 + w * plane;
                if constexpr (STAGED) {
                    if (on) {
                        put(sm.out_t, plane_t + o_step, [&](int r) { return t[r]; });
                        put(sm.out_s, plane_s + o_step, [&](int r) { return s[r]; });
                    }
                    __syncthreads();
                    const int begin_t = static_cast<int>((plane_t + o_step) & 3u), begin_s = static_cast<int>((plane_s + o_step) & 3u);
                    for (int w = 4 * tid; w < step_cells + 3; w += 4 * threads) {
                        carry(p.p_time + (plane_t + o_step - begin_t), sm.out_t, w, begin_t, begin_t + step_cells);
                        if (p.p_best_s) carry(p.p_best_s + (plane_s + o_step - begin_s), sm.out_s, w, begin_s, begin_s + step_cells);
                    }
                    __syncthreads();
                } else if (m_ok) {
                    rows_out(p.p_time + plane_t + o, [&](int r) { return t[r]; }, n);
                    if (p.p_best_s) rows_out(p.p_best_s + plane_s + o, [&](int r) { return s[r]; }, n);
                }
            };
            auto line = [&](double a, double c, uint32_t sz) {
#pragma unroll
                for (int r = 0; r < kRows; ++r) {
                    const double v = fma(x[r], a, c);
                    if (!(v > t[r])) { t[r] = v; s[r] = sz; }
                }
            };
            auto set = [&](double a, double c, uint32_t sz) {
#pragma unroll
                for (int r = 0; r < kRows; ++r) { t[r] = fma(x[r], a, c); s[r] = sz; }
            };
#pragma unroll
            for (int r = 0; r < kRows; ++r) x[r] = row[r].x;
            if (has2) {
                if (on) {
                    set(Qb, L, q_size);
                    if (near0 | near1) {
                        set(0.0, CUDART_INF, q_size);
#pragma unroll 1
                        for (int w = 1; w >= 0; --w)
                            each(near(w) | (q_best >> 5 == w ? 1u << (q_best & 31) : 0u), w, [&](int c) {
                                double Q, B, C;
                                candidate(c, Q, B, C);
                                line(Q, L, sm.sval[c]);
                            });
                    }
                }
                store(2, 0);
            }
            if (has5) {
                if (on) {
                    if (ns == 0) set(gm + L, 0.0, m_u);
                    else set(0.0, CUDART_INF, sm.sval[0]);
#pragma unroll 1
                    for (int w = n_s > 32 ? 1 : 0; w >= 0; --w)
                        each(sm.live[(2 * seg + w) * width + lm], w, [&](int c) {
                            double Q, B, C;
                            candidate(c, Q, B, C);
                            line(B, C, sm.sval[c]);
                        });
                }
                store(5, 1);
            }
            if (has9) {
                if (on) {
#pragma unroll
                    for (int r = 0; r < kRows; ++r) {
                        const int q = row[r].pair + lm;
                        t[r] = sm.pair_t[q];
                        s[r] = sm.pair_s[q];
                    }
                }
                store(9, 2);
            }
        }
    }
}

}  // namespace plogp
