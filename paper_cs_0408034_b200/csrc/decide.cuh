// decide_block: one CTA of the Broadcast half of the decision table (Sections 1 and 5 of the paper) for short
// candidate lists, with lanes mapped to the process count P.  (The Scatter half has no candidate
// lists and goes through scatter_kernel.)
//
// One CTA owns one table, a group of up to 16 message sizes and one or two tiles of 256 or 128 process counts (lane + 32 r,
// r = 0..7 or 0..3).  Its four warps split the message sizes, each over all process counts of the CTA, so a warp runs on its own
// from the candidate lists to the staged result and only the write-out needs the whole CTA.
//
// Every model of Table 1 is, for a fixed message size (and segment size), a line in P or a function of
// floor(log2 P) and ceil(log2 P) alone:
//     ids 0 1 2 3 4 5:  t = fma(P-1, a, c)
//     ids 6 7 8 9:      constant while (floor, ceil) stays, i.e. between a power of two and the next
// The decision is the lexicographic minimum of (t, id, s) over all cells of all enabled strategies
// (the minimum over s inside a strategy and then over strategies, smallest s and lowest id on ties).
// A warp numbers the cells of a message size in exactly that order: "slots" [lines of ids 0, 1, 2, 3, 4, 5]
// [one per (floor, ceil) pair of the tile], each with its coefficients (a, c) in shared memory (a pair's slot is
// (0, its smallest time)), so that a decision is a slot number and equal times go to the smaller one.
//
// Per message size:
//   1. lanes <-> candidates: the lines' coefficients, in FP64 and rounded down to FP32; the pilots, the lines that are
//      best at four of the CTA's process counts.
//   2. lanes <-> (floor, ceil) pairs: the best of ids 6 to 9 in FP64, one candidate after another.
//   3. per process count the best of the pilots and its pair: the running minimum's start.
//   4. every cell of every other line as a lower bound: FP32 coefficients, process count and fused multiply-add all
//      rounded down, two lines per instruction; the smallest bound per process count is compared with the running
//      minimum rounded up.  All terms are non-negative, so the bound is never above the FP64 time.
//   5. only rows of 32 process counts in which some bound is not above (1.4 of 8 on average) are searched exactly.  Where all
//      times lie outside FP32's range every row is, and a call takes 4 times as long.
// Results are those of the exhaustive FP64 search, bit for bit.  Staged as slot numbers [m][P] (1 byte); the write-out,
// rows of consecutive m per process count, evaluates the winner's line again (the same fma, the same double).
#pragma once

#include "device_common.cuh"

#include <algorithm>

namespace plogp {

namespace decide {

constexpr unsigned kFull = 0xffffffffu;
constexpr uint32_t kCandNone = 255;   // winner is an unsegmented strategy
constexpr uint32_t kCandWhole = 254;  // segmented winner with no fitting candidate: the whole message
constexpr int kPilots = 4;
static_assert(kMaxInlineS <= 64, "a lane builds at most two candidates");
constexpr int kStep = 16;  // lines per vote of the exact search
constexpr int kIntMax = 0x7FFFFFFF;

struct DecSmem {
    double *tab, *gs, *gm, *pm1;
    double2 *line;    // [mg][slots]: coefficients by slot
    float *x;         // [n_p]: P-1 rounded down
    float *fa, *fc;   // [kDecWarps][cap]: the lines' coefficients rounded down, for the warp's current message size
    double *q;        // [kDecWarps][cap_q]: g(s) k, for the warp's current message size
    float *fq;        // [kDecWarps][cap_q]: the same rounded down
    uint32_t *sval;   // [256]: segment sizes by candidate index; [kCandNone] = 0
    uint16_t *code;   // [mg][slots]: id << 8 | candidate index
    uint8_t *pair, *pos;  // [n_p]: pair of a process count; [mg][pos_stride]: winners
    int cap, lines, cap_q, slots, pos_stride;
};

__host__ __device__ inline int round_up(int x, int a) { return (x + a - 1) / a * a; }

// Shared-memory layout.  npad: 0 where the gap pre-pass has run; cap: the warps' lists of lines (a multiple of kStep); lines:
// of one message size at most; n_pairs: (floor, ceil) pairs of a CTA at most.  A slot number fits a byte: at most 132 lines and
// 61 pairs.
__host__ __device__ inline size_t dec_layout(int npad, int n_s, int n_pairs, int n_p, int mg, unsigned char *base, DecSmem *o)
{
    const int nsv = n_s > 0 ? n_s : 1;
    const int lines = 2 * nsv + 4, cap = round_up(lines, kStep), cap_q = round_up(nsv, 4), slots = lines + n_pairs, pos_stride = n_p + 4;
    size_t off = 0;
    auto take = [&](size_t bytes) { size_t at = off; off += (bytes + 15) & ~size_t(15); return at; };
    const size_t o_tab = take(3 * size_t(npad) * 8), o_gs = take(size_t(nsv) * 8), o_gm = take(mg * 8), o_pm = take(size_t(n_p) * 8), o_x = take(size_t(n_p) * 4),
                 o_line = take(size_t(mg) * slots * 16), o_fa = take(size_t(kDecWarps) * cap * 4), o_fc = take(size_t(kDecWarps) * cap * 4),
                 o_q = take(size_t(kDecWarps) * cap_q * 8), o_fq = take(size_t(kDecWarps) * cap_q * 4), o_sv = take(256 * 4), o_code = take(size_t(mg) * slots * 2),
                 o_pair = take(n_p), o_pos = take(size_t(mg) * pos_stride);
    if (o) {
        o->tab = reinterpret_cast<double *>(base + o_tab); o->gs = reinterpret_cast<double *>(base + o_gs);
        o->gm = reinterpret_cast<double *>(base + o_gm); o->pm1 = reinterpret_cast<double *>(base + o_pm);
        o->line = reinterpret_cast<double2 *>(base + o_line);
        o->fa = reinterpret_cast<float *>(base + o_fa); o->fc = reinterpret_cast<float *>(base + o_fc);
        o->q = reinterpret_cast<double *>(base + o_q); o->fq = reinterpret_cast<float *>(base + o_fq); o->sval = reinterpret_cast<uint32_t *>(base + o_sv);
        o->code = reinterpret_cast<uint16_t *>(base + o_code); o->pair = base + o_pair; o->pos = base + o_pos;
        o->x = reinterpret_cast<float *>(base + o_x);
        o->cap = cap; o->lines = lines; o->cap_q = cap_q; o->slots = slots; o->pos_stride = pos_stride;
    }
    return off;
}

}  // namespace decide

// ENV: lower-envelope search (DecideParams::envelope), compiled apart so that the exhaustive kernel carries none of it.
// R: process counts per lane and tile, 8, or 4 on grids that leave the GPU part empty (twice as many, shorter CTAs).
template <bool ENV, int R>
__device__ __forceinline__ void decide_block(const DecideParams &p, int block, unsigned char *smem_raw)
{
    using namespace decide;
    const int npad = p.T.npad;
    DecSmem sm;
    constexpr int kTileP = 32 * R;
    const int n_p = p.tiles * kTileP;
    dec_layout(p.gaps ? 0 : npad, p.G.n_s, p.n_pairs, n_p, p.mg, smem_raw, &sm);
    const uint32_t mask = p.G.mask;

    int b = block;
    const int mgroup = b % p.n_mgroups;
    b /= p.n_mgroups;
    const int ptile = b % p.n_ptiles;
    const int trel = b / p.n_ptiles;
    const int table = p.table0 + trel;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int m0 = mgroup * p.mg;  // p.mg <= kDecMG message sizes per CTA (fewer on small grids, for more CTAs)
    const int n_mi = min(p.mg, p.G.n_m - m0);
    const int tile0 = ptile * n_p;
    const int n_valid = min(n_p, p.G.n_P - tile0);
    const int pair0 = pair_of(P_at(p.G, tile0)), n_pairs = pair_of(P_at(p.G, tile0 + n_valid - 1)) - pair0 + 1;

    // g at the kernel's arguments: read from the gap pre-pass where the host has run it, else interpolated here
    const double *grow = p.gaps ? p.gaps + static_cast<size_t>(trel) * p.gaps_stride : nullptr;
    // what the set-up reads from global memory is on its way while the table is
    const double L = p.T.lat[table];
    const uint32_t m_mine = m0 + (tid & (kDecMG - 1)) < p.G.n_m ? p.G.m_list[m0 + (tid & (kDecMG - 1))] : 0u;
    const uint32_t s_mine = tid < p.G.n_s ? s_at(p.G, tid) : 0u;
    const int n_s = p.G.n_s;  // at most kMaxInlineS, fewer than the threads
    int ns_next = 0;
    uint32_t m_next = 0;
    double k_next[2] = {1.0, 1.0};  // Section 2's k of this lane's candidates, from the host's table
    auto fetch = [&](int mi) {
        if (mi >= n_mi) return;
        const int midx = m0 + mi;
        ns_next = p.G.ns_of_m[midx];
        m_next = p.G.m_list[midx];
        const double *krow = p.G.k_list + static_cast<size_t>(midx) * n_s;
        if (lane < n_s) k_next[0] = krow[lane];
        if (lane + 32 < n_s) k_next[1] = krow[lane + 32];
    };
    fetch(warp);
    if (!grow) stage_table(sm.tab, p.T, table);
    else wait_for_kernel_in_front();  // the gap pre-pass
    dependents_may_start();
    for (int i = tid; i < n_p; i += kDecThreads) {
        const int P = P_at(p.G, min(tile0 + i, p.G.n_P - 1));
        sm.pm1[i] = static_cast<double>(P - 1);
        sm.x[i] = __int2float_rd(P - 1);
        sm.pair[i] = static_cast<uint8_t>(min(pair_of(P) - pair0, n_pairs - 1));
    }
    __syncthreads();
    if (tid < n_s) {
        sm.sval[tid] = s_mine;
        sm.gs[tid] = grow ? grow[1 + tid] : gap_at(sm.tab, npad, static_cast<double>(s_mine));
    }
    if (tid == 0) sm.sval[kCandNone] = 0u;
    if (tid >= kDecThreads - kDecMG) {  // g(m) of the group's message sizes, by the last threads
        const int mi = tid - (kDecThreads - kDecMG);
        if (mi < n_mi) sm.gm[mi] = grow ? grow[1 + n_s + m0 + mi] : gap_at(sm.tab, npad, static_cast<double>(m_mine));
    }
    const double g1 = grow ? grow[0] : gap_at_one(sm.tab, npad);
    const double rdv = 2.0 * g1 + 3.0 * L;  // rendezvous handshake: 2 g(1) + 3 L
    __syncthreads();

    // the pilots' process counts: the winner changes more often where P is small
    float x_pilot[kPilots];
    {
        const int at[kPilots] = {n_valid >> 5, n_valid * 5 >> 5, n_valid * 15 >> 5, n_valid - 1};
#pragma unroll
        for (int i = 0; i < kPilots; ++i) x_pilot[i] = sm.x[at[i]];
    }
    // At P = 2 a segmented flat tree and a segmented chain cost the same for every s, which no bound can tell apart.
    const bool two = sm.pm1[0] == 1.0;

    // the codes carry the strategy ids as the caller names them
    auto idc = [&](int id) { return static_cast<uint32_t>(p.om.id_of[id]) << 8; };
    const uint32_t code2 = idc(2), code5 = idc(5), code9 = idc(9);
    const bool has0 = mask & 1u, has3 = (mask >> 3) & 1u, has2 = (mask >> 2) & 1u, has5 = (mask >> 5) & 1u, has6 = (mask >> 6) & 1u, has7 = (mask >> 7) & 1u,
               has8 = (mask >> 8) & 1u, has9 = (mask >> 9) & 1u;
    const bool any_log = mask & 0x3C0u;
    // The unsegmented lines do not depend on the message size beyond g(m): lanes 0..3 hold ids 0, 1, 3, 4
    // (Flat Tree (P-1) g + L, its rendezvous form (P-1) g + rdv; Chain (P-1)(g + L), rendezvous (P-1)(g + rdv)) as (g(m) + fa, fc).
    const int n01 = __popc(mask & 3u), n34 = __popc(mask & 0x18u);
    const int fid = lane < 4 ? lane + (lane >> 1) : 0;
    const bool f_on = lane < 4 && ((mask >> fid) & 1u);
    const double fa = fid == 3 ? L : (fid == 4 ? rdv : 0.0);
    const double fc = fid == 0 ? L : (fid == 1 ? rdv : 0.0);
    const uint16_t fcode = static_cast<uint16_t>(idc(fid) | kCandNone);
    float *const la = sm.fa + warp * sm.cap, *const lc = sm.fc + warp * sm.cap;
    double *const lq = sm.q + warp * sm.cap_q;
    float *const lqf = sm.fq + warp * sm.cap_q;

    // what a message size reads from global memory is fetched while the one before it is worked on
    for (int mi = warp; mi < n_mi; mi += kDecWarps) {
        const int ns = ns_next;
        const uint32_t m_u = m_next;
        const double k_of[2] = {k_next[0], k_next[1]};
        fetch(mi + kDecWarps);
        const int nsv = max(ns, 1);  // candidates actually evaluated (none fits: the whole message, k = 1)
        const double gm = sm.gm[mi];
        double2 *const line = sm.line + mi * sm.slots;
        uint16_t *const code = sm.code + mi * sm.slots;
        // Lower-envelope search (p.envelope, tables whose gaps never decrease): ids 2 and 9 keep only the candidate
        // with the smallest g(s) k (their minimum over s for every P at once, a rounded fused multiply-add being
        // monotone in it), id 5 only the candidates between its best ones at the tile's last and first process
        // count (envelope_near, device_common.cuh).  Otherwise every candidate enters the lists.
        const bool env = ENV && ns > 0;
        int q_c = 0, lo5 = 0, n5 = nsv;
        if constexpr (ENV) if (env) {
            const double x_first = sm.pm1[0], x_last = sm.pm1[n_valid - 1];
            double qb = CUDART_INF, t1[2] = {CUDART_INF, CUDART_INF}, t2[2] = {CUDART_INF, CUDART_INF};
            int qc = kIntMax;
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const int c = lane + 32 * h;
                if (c >= ns) break;
                const double gsv = sm.gs[c], k = k_of[h];
                const double Q = gsv * k, B = gsv + L, C = gsv * (k - 1.0);
                // a lane's first candidate always counts, and inf * 0 as inf: where times overflow, the index is still a candidate's
                if (h == 0 || Q < qb) { qb = Q; qc = c; }
                t1[h] = fmin(fma(x_first, B, C), CUDART_INF);
                t2[h] = fmin(fma(x_last, B, C), CUDART_INF);
            }
            warp_min_pair(qb, qc);
            q_c = qc;
            const double m1 = warp_min(fmin(t1[0], t1[1])), m2 = warp_min(fmin(t2[0], t2[1]));
            const double r = static_cast<double>(__fdividef(sm.x[n_valid - 1], sm.x[0]));  // to 1e-6: envelope_near has a third to spare
            const double up_to1 = fma(m1, envelope_near(r), m1), up_to2 = fma(m2, envelope_near(1.0), m2);
            int lo = kIntMax, hi = 0;
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const int c = lane + 32 * h;
                if (c < ns && t2[h] <= up_to2) lo = min(lo, c);
                if (c < ns && t1[h] <= up_to1) hi = c;
            }
            lo5 = __reduce_min_sync(kFull, lo);
            n5 = __reduce_max_sync(kFull, hi) - lo5 + 1;
        }
        const int nq = env ? 1 : nsv;  // entries of ids 2 and 9
        const int o2 = n01, o3 = o2 + (has2 ? nq : 0), o5 = o3 + n34, n1 = o5 + (has5 ? n5 : 0);
        const int n1p = round_up(n1, 4);

        // ---- the lines of this message size, and each lane's best ones at the pilots' process counts ----
        __syncwarp();  // the previous message size's loops have finished reading the warp's lists
        unsigned pilot[kPilots];  // bound (without its last 8 bits) and slot in one number
#pragma unroll
        for (int i = 0; i < kPilots; ++i) pilot[i] = 0xFFFFFFFFu;
        unsigned q_pilot = 0xFFFFFFFFu;  // the smallest g(s) k, likewise
        double t_two = CUDART_INF;       // P = 2: this lane's best line, exactly
        unsigned at_two = 0xFFu;
        auto put = [&](int slot, double a, double c, uint32_t cd, bool twin) {
            const float af = __double2float_rd(a), cf = __double2float_rd(c);
            line[slot] = make_double2(a, c);
            la[slot] = af;
            lc[slot] = twin ? CUDART_INF_F : cf;
            code[slot] = static_cast<uint16_t>(cd);
#pragma unroll
            for (int i = 0; i < kPilots; ++i)
                pilot[i] = min(pilot[i], (__float_as_uint(__fmaf_rd(x_pilot[i], af, cf)) & ~0xFFu) | static_cast<unsigned>(slot));
            if (two) {
                const double t = fma(1.0, a, c);
                if (t < t_two || (t == t_two && static_cast<unsigned>(slot) < at_two)) { t_two = t; at_two = static_cast<unsigned>(slot); }
            }
        };
        if (f_on) put((fid < 3 ? 0 : o3 - n01) + __popc(mask & 0x1Bu & ((1u << fid) - 1u)), gm + fa, fc, fcode, false);
        if (lane >= 16 && n1 + lane - 16 < round_up(n1, kStep)) {  // padding: the bound is +inf
            la[n1 + lane - 16] = 0.0f;
            lc[n1 + lane - 16] = CUDART_INF_F;
        }
        if (lane >= 16 && lane < 20 && nsv + lane - 16 < round_up(nsv, 4)) lqf[nsv + lane - 16] = CUDART_INF_F;
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            // the line coefficients of Table 1's segmented rows
            const int c = lane + 32 * h;
            if (c >= nsv) break;
            double gsv = gm, k = 1.0;
            uint32_t cand = kCandWhole;
            bool whole = true;  // one segment: the line of the unsegmented sibling, whose lower id wins the tie
            if (ns > 0) {
                gsv = sm.gs[c];
                k = k_of[h];
                cand = static_cast<uint32_t>(c);
                whole = sm.sval[c] == m_u;
            }
            const double Q = gsv * k;
            const float Qf = __double2float_rd(Q);
            lq[c] = Q;
            lqf[c] = Qf;
            q_pilot = min(q_pilot, (__float_as_uint(Qf) & ~0xFFu) | static_cast<unsigned>(c));
            if (has2 && (!env || c == q_c)) put(o2 + (env ? 0 : c), Q, L, code2 | cand, whole && has0);  // (P-1) (g(s) k) + L
            if (has5 && (!env || (c >= lo5 && c < lo5 + n5)))                                            // (P-1) (g(s) + L) + g(s) (k-1)
                put(o5 + (env ? c - lo5 : c), gsv + L, gsv * (k - 1.0), code5 | cand, whole && has3);
        }
#pragma unroll
        for (int i = 0; i < kPilots; ++i) pilot[i] = __reduce_min_sync(kFull, pilot[i]) & 0xFFu;
        q_pilot = env ? static_cast<unsigned>(q_c) : __reduce_min_sync(kFull, q_pilot) & 0xFFu;
        if ((q_pilot & 31u) == static_cast<unsigned>(lane)) lqf[q_pilot] = CUDART_INF_F;  // written by this lane itself above
        if (two && n1 > 0) {
            int e = at_two == 0xFFu ? kIntMax : static_cast<int>(at_two);
            warp_min_pair(t_two, e);
            at_two = static_cast<unsigned>(e);
        }
        __syncwarp();

        // ---- the best of ids 6 to 9 per (floor, ceil) pair, lanes <-> pairs ----
        if (any_log)
        for (int b0 = 0; b0 < n_pairs; b0 += 32) {
            const int pr = b0 + lane, li = pair0 + min(pr, n_pairs - 1);
            const double lf = static_cast<double>(li >> 1), lcd = static_cast<double>((li >> 1) + (li & 1)), lcL = lcd * L;
            double t = CUDART_INF;
            uint32_t cd = 0;
            if (has9) {  // floor(log2 P) g(s) k + ceil(log2 P) L: the smallest g(s) k, and bounds of all others
                unsigned cb = q_pilot;
                t = fma(lf, lq[cb], lcL);
                if (!env) {
                    const f32x2 x2 = splat2(static_cast<float>(li >> 1)), c2 = splat2(__double2float_rd(lcL));
                    float low = CUDART_INF_F;
                    for (int c = 0; c < nsv; c += 4) {
                        const f32x2x2 qq = *reinterpret_cast<const f32x2x2 *>(lqf + c);
                        low = min_with2(min_with2(low, fma2_down(x2, qq.x, c2)), fma2_down(x2, qq.y, c2));
                    }
                    if (__any_sync(kFull, low <= __double2float_ru(t))) {
#pragma unroll 1
                        for (int c = 0; c < nsv; ++c) {
                            const double v = fma(lf, lq[c], lcL);
                            if (v <= t && (v < t || static_cast<unsigned>(c) < cb)) { t = v; cb = static_cast<unsigned>(c); }
                        }
                    }
                }
                cd = code9 | (ns > 0 ? cb : kCandWhole);
            }
            // lower ids win ties: in descending order, '<='
            if (has8) {  // Binomial Tree Rendezvous: floor(log2 P) g(m) + ceil(log2 P) rdv
                const double v = fma(lf, gm, lcd * rdv);
                if (v <= t) { t = v; cd = idc(8) | kCandNone; }
            }
            if (has7) {  // Binomial Tree: floor(log2 P) g(m) + ceil(log2 P) L
                const double v = fma(lf, gm, lcL);
                if (v <= t) { t = v; cd = idc(7) | kCandNone; }
            }
            if (has6) {  // Binary Tree (the printed bound): ceil(log2 P) (2 g(m) + L)
                const double v = lcd * fma(2.0, gm, L);
                if (v <= t) { t = v; cd = idc(6) | kCandNone; }
            }
            if (pr < n_pairs) {
                line[sm.lines + pr] = make_double2(0.0, t);
                code[sm.lines + pr] = static_cast<uint16_t>(cd);
            }
        }

        // ---- the pilots leave the lists: their own bounds would always pass ----
        if (n1 > 0 && lane < kPilots) {
            unsigned mine = pilot[0];
#pragma unroll
            for (int i = 1; i < kPilots; ++i) mine = lane == i ? pilot[i] : mine;
            la[mine] = 0.0f;
            lc[mine] = CUDART_INF_F;
        }
        __syncwarp();

        for (int tile = 0; tile < p.tiles; ++tile) {
            if (tile * kTileP >= n_valid) break;
            const double *const xd = sm.pm1 + tile * kTileP + lane;
            uint8_t *const pos = sm.pos + mi * sm.pos_stride + tile * kTileP + lane;
            float T[R];
            // ---- start of the running minima: the best of the pilots and the pair ----
            {
                double t[R];
                unsigned at[R];
#pragma unroll
                for (int r = 0; r < R; ++r) { t[r] = CUDART_INF; at[r] = 0xFFu; }
                if (n1 > 0) {
                    const double2 e = line[pilot[0]];
#pragma unroll
                    for (int r = 0; r < R; ++r) { t[r] = fma(xd[32 * r], e.x, e.y); at[r] = pilot[0]; }
#pragma unroll
                    for (int i = 1; i < kPilots; ++i) {
                        if (pilot[i] == pilot[i - 1]) continue;
                        const double2 v = line[pilot[i]];
#pragma unroll
                        for (int r = 0; r < R; ++r) {
                            const double tt = fma(xd[32 * r], v.x, v.y);
                            if (tt < t[r] || (tt == t[r] && pilot[i] < at[r])) { t[r] = tt; at[r] = pilot[i]; }
                        }
                    }
                    if (two && tile == 0 && lane == 0) { t[0] = t_two; at[0] = at_two; }
                }
                if (any_log) {
#pragma unroll
                    for (int r = 0; r < R; ++r) {
                        const unsigned slot = sm.lines + sm.pair[tile * kTileP + 32 * r + lane];
                        const double tl = line[slot].y;
                        if (tl < t[r] || n1 == 0) { t[r] = tl; at[r] = slot; }  // lines have the lower ids
                    }
                }
#pragma unroll
                for (int r = 0; r < R; ++r) {
                    T[r] = __double2float_ru(t[r]);
                    pos[32 * r] = static_cast<uint8_t>(at[r]);
                }
                if (two && tile == 0 && lane == 0) T[0] = -1.0f;  // settled
            }

            // ---- lower bounds of all other lines ----
            float mn[R];
            f32x2 x2[R];
#pragma unroll
            for (int r = 0; r < R; ++r) { mn[r] = CUDART_INF_F; x2[r] = splat2(sm.x[tile * kTileP + 32 * r + lane]); }
#pragma unroll 2
            for (int j = 0; j < n1p; j += 4) {
                const f32x2x2 aa = *reinterpret_cast<const f32x2x2 *>(la + j), cc = *reinterpret_cast<const f32x2x2 *>(lc + j);
#pragma unroll
                for (int r = 0; r < R; ++r) mn[r] = min_with2(mn[r], fma2_down(x2[r], aa.x, cc.x));
#pragma unroll
                for (int r = 0; r < R; ++r) mn[r] = min_with2(mn[r], fma2_down(x2[r], aa.y, cc.y));
            }
            bool any = false;
#pragma unroll
            for (int r = 0; r < R; ++r) any |= mn[r] <= T[r];
            if (!__any_sync(kFull, any)) continue;

            // ---- exact search of the rows in which some bound is not above the running minimum ----
            unsigned hit = 0;
#pragma unroll
            for (int r = 0; r < R; ++r)
                if (mn[r] <= T[r]) hit |= 1u << r;
#pragma unroll 1
            for (unsigned rows = __reduce_or_sync(kFull, hit); rows; rows &= rows - 1) {
                const int r = __ffs(rows) - 1;
                const double x = xd[32 * r];
                const f32x2 xx = splat2(__double2float_rd(x));
                unsigned at = pos[32 * r];
                const double2 w = line[at];
                double t = fma(x, w.x, w.y);
                float Tr = (hit >> r) & 1u ? __double2float_ru(t) : -1.0f;
#pragma unroll 1
                for (int j = 0; j < n1; j += kStep) {
                    float low[kStep / 4];
#pragma unroll
                    for (int q = 0; q < kStep / 4; ++q) {
                        const f32x2x2 aa = *reinterpret_cast<const f32x2x2 *>(la + j + 4 * q), cc = *reinterpret_cast<const f32x2x2 *>(lc + j + 4 * q);
                        low[q] = min_with2(min_with2(CUDART_INF_F, fma2_down(xx, aa.x, cc.x)), fma2_down(xx, aa.y, cc.y));
                    }
                    if (!__any_sync(kFull, fminf(fminf(low[0], low[1]), fminf(low[2], low[3])) <= Tr)) continue;
#pragma unroll
                    for (int q = 0; q < kStep / 4; ++q) {
                        if (!__any_sync(kFull, low[q] <= Tr)) continue;
                        double tt[4];  // four loads in flight; behind the last line the last one again
#pragma unroll
                        for (int u = 0; u < 4; ++u) {
                            const double2 v = line[min(j + 4 * q + u, n1 - 1)];
                            tt[u] = fma(x, v.x, v.y);
                        }
#pragma unroll
                        for (int u = 0; u < 4; ++u) {
                            const unsigned slot = static_cast<unsigned>(min(j + 4 * q + u, n1 - 1));
                            if (tt[u] < t || (tt[u] == t && slot < at)) { t = tt[u]; at = slot; }
                        }
                        if (Tr >= 0.0f) Tr = __double2float_ru(t);
                    }
                }
                pos[32 * r] = static_cast<uint8_t>(at);
            }
        }
    }
    __syncthreads();

    // transposed write-out of the staged group: rows of p.mg consecutive m per process count, running pointers
    const size_t plane = static_cast<size_t>(p.G.n_P) * p.G.n_m;
    const size_t base = (static_cast<size_t>(table - p.out_table0) * p.om.planes + p.om.plane_bcast) * plane + static_cast<size_t>(tile0) * p.G.n_m + m0;
    if (p.vec_out) {
        // two message sizes per lane: 16-byte, 8-byte and 2-byte stores (the host has checked the alignment)
        const int half = p.mg >> 1;
        const int mi = 2 * (lane & (half - 1)), rows = 32 / half, pr0 = warp * rows + lane / half, prs = kDecWarps * rows;
        if (mi < n_mi) {
            const uint32_t m_u0 = p.G.m_list[m0 + mi], m_u1 = p.G.m_list[m0 + mi + 1];
            const size_t o = base + static_cast<size_t>(pr0) * p.G.n_m + mi;
            const size_t step = static_cast<size_t>(prs) * p.G.n_m;
            double *out_t = p.d_time + o;
            uint32_t *out_s = p.d_sbytes + o;
            uint8_t *out_id = p.d_strategy + o;
            const double2 *l0 = sm.line + mi * sm.slots, *l1 = l0 + sm.slots;
            const uint16_t *c0 = sm.code + mi * sm.slots, *c1 = c0 + sm.slots;
            const uint8_t *p0 = sm.pos + mi * sm.pos_stride + pr0, *p1 = p0 + sm.pos_stride;
            const double *px = sm.pm1 + pr0;
#pragma unroll 1  // (unrolled by the compiler it is 1.3 % slower on the batched workload)
            for (int pr = pr0; pr < n_valid; pr += prs) {
                const unsigned at0 = *p0, at1 = *p1;
                const double x = *px;
                const double2 e0 = l0[at0], e1 = l1[at1];
                const uint32_t code0 = c0[at0], code1 = c1[at1];
                const uint32_t cand0 = code0 & 255u, cand1 = code1 & 255u;
                uint32_t s0 = sm.sval[cand0], s1 = sm.sval[cand1];
                if (cand0 == kCandWhole) s0 = m_u0;
                if (cand1 == kCandWhole) s1 = m_u1;
                *reinterpret_cast<double2 *>(out_t) = make_double2(fma(x, e0.x, e0.y), fma(x, e1.x, e1.y));
                *reinterpret_cast<uint2 *>(out_s) = make_uint2(s0, s1);
                *reinterpret_cast<uint16_t *>(out_id) = static_cast<uint16_t>(__byte_perm(code0, code1, 0x0051));
                out_t += step; out_s += step; out_id += step;
                p0 += prs; p1 += prs; px += prs;
            }
        }
    } else {
        const int mi = lane & (p.mg - 1), prow = lane / p.mg, rows = 32 / p.mg;
        if (mi < n_mi) {
            const uint32_t m_u = p.G.m_list[m0 + mi];
            for (int pr = warp * rows + prow; pr < n_valid; pr += kDecWarps * rows) {
                const size_t o = base + static_cast<size_t>(pr) * p.G.n_m + mi;
                const unsigned at = sm.pos[mi * sm.pos_stride + pr];
                const double2 e = sm.line[mi * sm.slots + at];
                const uint32_t code = sm.code[mi * sm.slots + at];
                const uint32_t cand = code & 255u;
                p.d_time[o] = fma(sm.pm1[pr], e.x, e.y);
                p.d_strategy[o] = static_cast<uint8_t>(code >> 8);
                p.d_sbytes[o] = cand == kCandWhole ? m_u : sm.sval[cand];
            }
        }
    }
}

}  // namespace plogp
