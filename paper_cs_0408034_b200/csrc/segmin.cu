// segmin_kernel: the segment-size search of Section 3.1 for plogp_predict on short candidate lists, with lanes
// mapped to the process count P: for each segmented strategy of Table 1 (ids 2, 5, 9) on its own, the minimum
// of the model over the candidate segment sizes and the smallest size that attains it.
//
// Same building blocks as decide_kernel (decide.cuh), with one running minimum per strategy instead of one
// over all of them.  One CTA owns one table, up to 16 consecutive message sizes (32 with eight warps) and one or two tiles
// of 256 process counts (lane + 32 r, r = 0..7); its four (eight) warps split the message sizes.  For a fixed message size the models are
//     id 2: fma(P-1, Q, L)      id 9: fma(floor(log2 P), Q, ceil(log2 P) L)      Q = g(s) k
//     id 5: fma(P-1, B, C)      B = g(s) + L, C = g(s) (k-1)
// so a warp builds the coefficient lists of a message size (lanes <-> candidates), searches id 9 once per
// (floor, ceil) pair of log2 P (lanes <-> pairs) and sweeps ids 2 and 5 over the process counts: the running minimum
// starts from pilots (id 2: the smallest Q; id 5: the winners at four process counts), every cell of every other
// candidate is evaluated as a lower bound in FP32 (coefficients, process count and fused multiply-add rounded down, two
// candidates per instruction), and rows of 32 process counts in which some bound is not above the running minimum are
// searched exactly, (time, candidate) in lexicographic order.  Results are those of the exhaustive FP64 search, bit for
// bit.  The winners are staged as candidate numbers, one byte per cell; the write-out, rows of consecutive m per process
// count, evaluates the winner's model again (the same fma, the same double).  The outputs are the prediction planes
// time[table][13][P][m] and best_s[table][3][P][m].
#include "device_common.cuh"

#include <algorithm>
#include <type_traits>

namespace plogp {

namespace {

constexpr int kPilots = 4;
constexpr int kStep = 16;  // candidates per vote of the exact search
constexpr unsigned kFull = 0xffffffffu;
static_assert(kMaxInlineS <= 64, "a lane builds at most two candidates");

__host__ __device__ inline int round_up(int x, int a) { return (x + a - 1) / a * a; }

struct SegSmem {
    double *tab, *gs, *gm, *pm1;
    double2 *l5;      // [mg][list]: (B, C)
    double *q;        // [mg][list]: Q
    double *t9;       // [mg][n_pairs]: id 9's minimum
    float *x;         // [n_p]: P-1 rounded down
    float *fb, *fc, *fq;  // [warps][cap]: the lists of the warp's current message size rounded down, without the pilots
    uint32_t *sval;
    uint8_t *i9;      // [mg][n_pairs]: id 9's winner
    uint8_t *pair;    // [n_p]: pair of a process count
    uint8_t *pos2, *pos5;  // [mg][stride]: winners of ids 2 and 5
    int cap, list, stride;  // list: odd, so that neighbouring message sizes start in different banks
};

__host__ __device__ inline size_t seg_layout(int npad, int n_s, int n_pairs, int n_p, int mg, int warps, unsigned char *base, SegSmem *o)
{
    const int nsv = n_s > 0 ? n_s : 1;
    const int cap = round_up(nsv, kStep), list = nsv | 1, stride = n_p + 4;
    size_t off = 0;
    auto take = [&](size_t bytes) { size_t at = off; off += (bytes + 15) & ~size_t(15); return at; };
    const size_t o_tab = take(3 * size_t(npad) * 8), o_gs = take(size_t(nsv) * 8), o_gm = take(mg * 8), o_pm = take(size_t(n_p) * 8),
                 o_l5 = take(size_t(mg) * list * 16), o_q = take(size_t(mg) * list * 8), o_t9 = take(size_t(mg) * n_pairs * 8),
                 o_x = take(size_t(n_p) * 4), o_fb = take(size_t(warps) * cap * 4), o_fc = take(size_t(warps) * cap * 4),
                 o_fq = take(size_t(warps) * cap * 4), o_sv = take(size_t(nsv) * 4), o_i9 = take(size_t(mg) * n_pairs), o_pair = take(n_p),
                 o_p2 = take(size_t(mg) * stride), o_p5 = take(size_t(mg) * stride);
    if (o) {
        o->tab = reinterpret_cast<double *>(base + o_tab); o->gs = reinterpret_cast<double *>(base + o_gs);
        o->gm = reinterpret_cast<double *>(base + o_gm); o->pm1 = reinterpret_cast<double *>(base + o_pm);
        o->l5 = reinterpret_cast<double2 *>(base + o_l5); o->q = reinterpret_cast<double *>(base + o_q);
        o->t9 = reinterpret_cast<double *>(base + o_t9); o->x = reinterpret_cast<float *>(base + o_x);
        o->fb = reinterpret_cast<float *>(base + o_fb); o->fc = reinterpret_cast<float *>(base + o_fc);
        o->fq = reinterpret_cast<float *>(base + o_fq); o->sval = reinterpret_cast<uint32_t *>(base + o_sv);
        o->i9 = base + o_i9; o->pair = base + o_pair; o->pos2 = base + o_p2; o->pos5 = base + o_p5;
        o->cap = cap; o->list = list; o->stride = stride;
    }
    return off;
}

}  // namespace

// R: as in decide_kernel.  W: warps, four of them per 16 message sizes (the host says when eight are better).
template <int R, int W>
__global__ void __launch_bounds__(32 * W, W == 4 ? 5 : 2) segmin_kernel(const SegminParams p)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int npad = p.T.npad;
    SegSmem sm;
    constexpr int kTileP = 32 * R;
    const int n_p = p.tiles * kTileP;
    seg_layout(npad, p.G.n_s, p.n_pairs, n_p, p.mg, W, smem_raw, &sm);
    const uint32_t mask = p.G.mask;
    const bool has2 = (mask >> 2) & 1u, has5 = (mask >> 5) & 1u, has9 = (mask >> 9) & 1u;

    int b = blockIdx.x;
    const int mgroup = b % p.n_mgroups;
    b /= p.n_mgroups;
    const int ptile = b % p.n_ptiles;
    const int trel = b / p.n_ptiles;
    const int table = p.table0 + trel;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int m0 = mgroup * p.mg;
    const int n_mi = min(p.mg, p.G.n_m - m0);
    const int tile0 = ptile * n_p;
    const int n_valid = min(n_p, p.G.n_P - tile0);
    const int pair0 = pair_of(P_at(p.G, tile0)), n_pairs = pair_of(P_at(p.G, tile0 + n_valid - 1)) - pair0 + 1;

    // g at the kernel's arguments: read from the gap pre-pass where the host has run it, else interpolated here
    const double *grow = p.gaps ? p.gaps + static_cast<size_t>(trel) * p.gaps_stride : nullptr;
    // what the set-up reads from global memory is on its way while the table is
    const double L = p.T.lat[table];
    const uint32_t m_mine = m0 + (tid & (4 * W - 1)) < p.G.n_m ? p.G.m_list[m0 + (tid & (4 * W - 1))] : 0u;
    const uint32_t s_mine = tid < p.G.n_s ? s_at(p.G, tid) : 0u;
    const int n_s = p.G.n_s;  // at most kMaxInlineS, fewer than the threads
    int ns_next = 0;
    double k_next[2] = {1.0, 1.0};  // Section 2's k of this lane's candidates, from the host's table
    auto fetch = [&](int mi) {
        if (mi >= n_mi) return;
        ns_next = p.G.ns_of_m[m0 + mi];
        const double *krow = p.G.k_list + static_cast<size_t>(m0 + mi) * n_s;
        if (lane < n_s) k_next[0] = krow[lane];
        if (lane + 32 < n_s) k_next[1] = krow[lane + 32];
    };
    fetch(warp);
    if (!grow) stage_table(sm.tab, p.T, table);
    else wait_for_kernel_in_front();  // the gap pre-pass
    dependents_may_start();
    for (int i = tid; i < n_p; i += 32 * W) {
        const int P = P_at(p.G, min(tile0 + i, p.G.n_P - 1));
        sm.pm1[i] = static_cast<double>(P - 1);
        sm.x[i] = __int2float_rd(P - 1);
        sm.pair[i] = static_cast<uint8_t>(pair_of(P) - pair0);
    }
    __syncthreads();
    if (tid < n_s) {
        sm.sval[tid] = s_mine;
        sm.gs[tid] = grow ? grow[1 + tid] : gap_at(sm.tab, npad, static_cast<double>(s_mine));
    }
    if (tid >= 28 * W) {
        const int mi = tid - 28 * W;
        if (mi < n_mi) sm.gm[mi] = grow ? grow[1 + n_s + m0 + mi] : gap_at(sm.tab, npad, static_cast<double>(m_mine));
    }
    __syncthreads();

    float x_pilot[kPilots];  // the winner of id 5 changes more often where P is small
    {
        const int at[kPilots] = {n_valid >> 5, n_valid * 5 >> 5, n_valid * 15 >> 5, n_valid - 1};
#pragma unroll
        for (int i = 0; i < kPilots; ++i) x_pilot[i] = sm.x[at[i]];
    }
    float *const fb = sm.fb + warp * sm.cap, *const fc = sm.fc + warp * sm.cap, *const fq = sm.fq + warp * sm.cap;
    const float Lf = __double2float_rd(L);
    const f32x2 L2 = splat2(Lf);

    for (int mi = warp; mi < n_mi; mi += W) {
        // what a message size reads from global memory is fetched while the one before it is worked on
        const int ns = ns_next;
        const double k_of[2] = {k_next[0], k_next[1]};
        fetch(mi + W);
        const int nsv = max(ns, 1);  // candidates actually evaluated (none fits: the whole message, k = 1)
        const int np4 = round_up(nsv, 4), np16 = round_up(nsv, kStep);
        const double gm = sm.gm[mi];
        double *const q = sm.q + mi * sm.list;
        double2 *const l5 = sm.l5 + mi * sm.list;

        // ---- the lists (lanes <-> candidates) and the pilots: bound (without its last 8 bits) and index in one number ----
        __syncwarp();  // the previous message size's sweeps are done with the lists
        unsigned pilot[kPilots], q_pilot = 0xFFFFFFFFu;
#pragma unroll
        for (int i = 0; i < kPilots; ++i) pilot[i] = 0xFFFFFFFFu;
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int c = lane + 32 * h;
            if (c >= np16) break;
            float Bf = 0.f, Cf = CUDART_INF_F, Qf = CUDART_INF_F;  // padding: the bound is +inf
            if (c < nsv) {
                double gsv = gm, k = 1.0;
                if (ns > 0) {
                    gsv = sm.gs[c];
                    k = k_of[h];
                }
                const double Q = gsv * k, B = gsv + L, C = gsv * (k - 1.0);
                q[c] = Q;
                l5[c] = make_double2(B, C);
                Qf = __double2float_rd(Q); Bf = __double2float_rd(B); Cf = __double2float_rd(C);
                q_pilot = min(q_pilot, (__float_as_uint(Qf) & ~0xFFu) | static_cast<unsigned>(c));
#pragma unroll
                for (int i = 0; i < kPilots; ++i)
                    pilot[i] = min(pilot[i], (__float_as_uint(__fmaf_rd(x_pilot[i], Bf, Cf)) & ~0xFFu) | static_cast<unsigned>(c));
            }
            fb[c] = Bf; fc[c] = Cf; fq[c] = Qf;
        }
        q_pilot = __reduce_min_sync(kFull, q_pilot) & 0xFFu;
#pragma unroll
        for (int i = 0; i < kPilots; ++i) pilot[i] = __reduce_min_sync(kFull, pilot[i]) & 0xFFu;
        __syncwarp();
        // the pilots leave the lists: their own bounds would always pass
        if (lane < kPilots) {
            unsigned mine = pilot[0];
#pragma unroll
            for (int i = 1; i < kPilots; ++i) mine = lane == i ? pilot[i] : mine;
            fb[mine] = 0.0f;
            fc[mine] = CUDART_INF_F;
        }
        if (lane == kPilots) fq[q_pilot] = CUDART_INF_F;
        __syncwarp();

        // ---- id 9 per (floor, ceil) pair ----
        if (has9)
        for (int b0 = 0; b0 < n_pairs; b0 += 32) {
            const int pr = b0 + lane, li = pair0 + min(pr, n_pairs - 1);
            const double lf = static_cast<double>(li >> 1), lcL = static_cast<double>((li >> 1) + (li & 1)) * L;
            const f32x2 x2 = splat2(static_cast<float>(li >> 1)), c2 = splat2(__double2float_rd(lcL));
            unsigned at = q_pilot;
            double t = fma(lf, q[at], lcL);
            float low = CUDART_INF_F;
            for (int c = 0; c < np4; c += 4) {
                const f32x2x2 qq = *reinterpret_cast<const f32x2x2 *>(fq + c);
                low = min_with2(min_with2(low, fma2_down(x2, qq.x, c2)), fma2_down(x2, qq.y, c2));
            }
            if (__any_sync(kFull, low <= __double2float_ru(t))) {
#pragma unroll 1
                for (int c = 0; c < nsv; ++c) {
                    const double v = fma(lf, q[c], lcL);
                    if (v <= t && (v < t || static_cast<unsigned>(c) < at)) { t = v; at = static_cast<unsigned>(c); }
                }
            }
            if (pr < n_pairs) {
                sm.t9[mi * p.n_pairs + pr] = t;
                sm.i9[mi * p.n_pairs + pr] = static_cast<uint8_t>(at);
            }
        }

        for (int tile = 0; tile < p.tiles; ++tile) {
            if (tile * kTileP >= n_valid) break;
            const double *const xd = sm.pm1 + tile * kTileP + lane;
            uint8_t *const pos2 = sm.pos2 + mi * sm.stride + tile * kTileP + lane, *const pos5 = sm.pos5 + mi * sm.stride + tile * kTileP + lane;
            f32x2 x2[R];
#pragma unroll
            for (int r = 0; r < R; ++r) x2[r] = splat2(sm.x[tile * kTileP + 32 * r + lane]);
            unsigned hit = 0;  // bit r: id 5, bit 16 + r: id 2
            if (has5) {
                float T[R], mn[R];
                {
                    double t[R];
                    unsigned at[R];
                    const double2 e = l5[pilot[0]];
#pragma unroll
                    for (int r = 0; r < R; ++r) { t[r] = fma(xd[32 * r], e.x, e.y); at[r] = pilot[0]; }
#pragma unroll
                    for (int i = 1; i < kPilots; ++i) {
                        if (pilot[i] == pilot[i - 1]) continue;
                        const double2 v = l5[pilot[i]];
#pragma unroll
                        for (int r = 0; r < R; ++r) {
                            const double tt = fma(xd[32 * r], v.x, v.y);
                            if (tt < t[r] || (tt == t[r] && pilot[i] < at[r])) { t[r] = tt; at[r] = pilot[i]; }
                        }
                    }
#pragma unroll
                    for (int r = 0; r < R; ++r) { T[r] = __double2float_ru(t[r]); pos5[32 * r] = static_cast<uint8_t>(at[r]); }
                }
#pragma unroll
                for (int r = 0; r < R; ++r) mn[r] = CUDART_INF_F;
#pragma unroll 2
                for (int j = 0; j < np4; j += 4) {
                    const f32x2x2 bb = *reinterpret_cast<const f32x2x2 *>(fb + j), cc = *reinterpret_cast<const f32x2x2 *>(fc + j);
#pragma unroll
                    for (int r = 0; r < R; ++r) mn[r] = min_with2(mn[r], fma2_down(x2[r], bb.x, cc.x));
#pragma unroll
                    for (int r = 0; r < R; ++r) mn[r] = min_with2(mn[r], fma2_down(x2[r], bb.y, cc.y));
                }
#pragma unroll
                for (int r = 0; r < R; ++r)
                    if (mn[r] <= T[r]) hit |= 1u << r;
            }
            if (has2) {
                float T[R], mn[R];
                const double Q = q[q_pilot];
#pragma unroll
                for (int r = 0; r < R; ++r) {
                    T[r] = __double2float_ru(fma(xd[32 * r], Q, L));
                    pos2[32 * r] = static_cast<uint8_t>(q_pilot);
                    mn[r] = CUDART_INF_F;
                }
#pragma unroll 2
                for (int j = 0; j < np4; j += 4) {
                    const f32x2x2 qq = *reinterpret_cast<const f32x2x2 *>(fq + j);
#pragma unroll
                    for (int r = 0; r < R; ++r) mn[r] = min_with2(mn[r], fma2_down(x2[r], qq.x, L2));
#pragma unroll
                    for (int r = 0; r < R; ++r) mn[r] = min_with2(mn[r], fma2_down(x2[r], qq.y, L2));
                }
#pragma unroll
                for (int r = 0; r < R; ++r)
                    if (mn[r] <= T[r]) hit |= 0x10000u << r;
            }

            // ---- exact search of the rows in which some bound is not above the running minimum ----
#pragma unroll 1
            for (unsigned rows = __reduce_or_sync(kFull, hit); rows; rows &= rows - 1) {
                const int bit = __ffs(rows) - 1, r = bit & 15;
                const bool two = bit >> 4;  // id 2
                const double x = xd[32 * r];
                const f32x2 xx = splat2(sm.x[tile * kTileP + 32 * r + lane]);
                uint8_t *const pos = two ? pos2 : pos5;
                unsigned at = pos[32 * r];
                double t = two ? fma(x, q[at], L) : fma(x, l5[at].x, l5[at].y);
                const bool mine = (hit >> bit) & 1u;
                float T = mine ? __double2float_ru(t) : -1.0f;
#pragma unroll 1
                for (int j = 0; j < nsv; j += kStep) {
                    float low[kStep / 4];
#pragma unroll
                    for (int u = 0; u < kStep / 4; ++u) {
                        const f32x2x2 aa = *reinterpret_cast<const f32x2x2 *>((two ? fq : fb) + j + 4 * u);
                        f32x2x2 cc;
                        cc.x = cc.y = L2;
                        if (!two) cc = *reinterpret_cast<const f32x2x2 *>(fc + j + 4 * u);
                        low[u] = min_with2(min_with2(CUDART_INF_F, fma2_down(xx, aa.x, cc.x)), fma2_down(xx, aa.y, cc.y));
                    }
                    if (!__any_sync(kFull, fminf(fminf(low[0], low[1]), fminf(low[2], low[3])) <= T)) continue;
#pragma unroll
                    for (int u = 0; u < kStep / 4; ++u) {
                        if (!__any_sync(kFull, low[u] <= T)) continue;
                        double tt[4];  // four loads in flight; behind the last candidate the last one again
#pragma unroll
                        for (int v = 0; v < 4; ++v) {
                            const int c = min(j + 4 * u + v, nsv - 1);
                            const double2 e = two ? make_double2(q[c], L) : l5[c];
                            tt[v] = fma(x, e.x, e.y);
                        }
#pragma unroll
                        for (int v = 0; v < 4; ++v) {
                            const unsigned c = static_cast<unsigned>(min(j + 4 * u + v, nsv - 1));
                            if (tt[v] < t || (tt[v] == t && c < at)) { t = tt[v]; at = c; }
                        }
                        if (mine) T = __double2float_ru(t);
                    }
                }
                pos[32 * r] = static_cast<uint8_t>(at);
            }
        }
    }
    __syncthreads();

    // ---- transposed write-out: rows of p.mg consecutive m per process count, one plane after another ----
    const size_t plane = static_cast<size_t>(p.G.n_P) * p.G.n_m;
    const size_t cell0 = static_cast<size_t>(tile0) * p.G.n_m + m0;
    auto write_plane = [&](auto w_tag, int strategy) {
        constexpr int w = decltype(w_tag)::value;  // 0, 1, 2: ids 2, 5, 9
        double *plane_t = p.p_time + (static_cast<size_t>(table - p.out_table0) * 13 + strategy) * plane + cell0;
        uint32_t *plane_s = p.p_best_s ? p.p_best_s + (static_cast<size_t>(table - p.out_table0) * 3 + w) * plane + cell0 : nullptr;
        const uint8_t *const pos = w == 0 ? sm.pos2 : sm.pos5;
        // winner and time of one cell
        auto cell = [&](int mi, int pr, double x, unsigned &at) {
            if (w == 2) {
                const int i = mi * p.n_pairs + sm.pair[pr];
                at = sm.i9[i];
                return sm.t9[i];
            }
            at = pos[mi * sm.stride + pr];
            if (w == 0) return fma(x, sm.q[mi * sm.list + at], L);
            const double2 e = sm.l5[mi * sm.list + at];
            return fma(x, e.x, e.y);
        };
        if (p.vec_out) {
            // two message sizes per lane (16-byte and 8-byte stores; the host has checked the alignment)
            const int half = p.mg >> 1;
            const int mi = 2 * (lane & (half - 1)), rows = 32 / half, step = W * rows, pr0 = warp * rows + lane / half;
            if (mi < n_mi) {  // n_m is even, so mi + 1 is a message size of the grid too
                const uint32_t m_u0 = p.G.m_list[m0 + mi], m_u1 = p.G.m_list[m0 + mi + 1];
                const bool w0 = p.G.ns_of_m[m0 + mi] == 0, w1 = p.G.ns_of_m[m0 + mi + 1] == 0;  // the whole message
                const size_t o = static_cast<size_t>(pr0) * p.G.n_m + mi, go = static_cast<size_t>(step) * p.G.n_m;
                double *out_t = plane_t + o;
                uint32_t *out_s = plane_s ? plane_s + o : nullptr;
#pragma unroll 1
                for (int pr = pr0; pr < n_valid; pr += step) {
                    const double x = sm.pm1[pr];
                    unsigned a0, a1;
                    const double t0 = cell(mi, pr, x, a0), t1 = cell(mi + 1, pr, x, a1);
                    *reinterpret_cast<double2 *>(out_t) = make_double2(t0, t1);
                    out_t += go;
                    if (out_s) {
                        *reinterpret_cast<uint2 *>(out_s) = make_uint2(w0 ? m_u0 : sm.sval[a0], w1 ? m_u1 : sm.sval[a1]);
                        out_s += go;
                    }
                }
            }
        } else {
            const int mi = lane & (p.mg - 1), rows = 32 / p.mg;
            if (mi < n_mi) {
                const uint32_t m_u = p.G.m_list[m0 + mi];
                const bool whole = p.G.ns_of_m[m0 + mi] == 0;
                for (int pr = warp * rows + lane / p.mg; pr < n_valid; pr += W * rows) {
                    const size_t o = static_cast<size_t>(pr) * p.G.n_m + mi;
                    unsigned at;
                    plane_t[o] = cell(mi, pr, sm.pm1[pr], at);
                    if (plane_s) plane_s[o] = whole ? m_u : sm.sval[at];
                }
            }
        }
    };
    if (has2) write_plane(std::integral_constant<int, 0>{}, 2);
    if (has5) write_plane(std::integral_constant<int, 1>{}, 5);
    if (has9) write_plane(std::integral_constant<int, 2>{}, 9);
    last_block_waits(tid);
}

cudaError_t launch_segmin(const SegminParams &p, bool overlap, cudaStream_t st)
{
    const long long blocks = static_cast<long long>(p.n_mgroups) * p.n_ptiles * p.n_tables_launch;
    if (blocks <= 0 || blocks > 0x7FFFFFFFLL) return cudaErrorInvalidConfiguration;
    const size_t smem = seg_layout(p.T.npad, p.G.n_s, p.n_pairs, p.tiles * 32 * p.rows, p.mg, p.warps, nullptr, nullptr);
    const auto kernel = p.warps == 8 ? segmin_kernel<8, 8> : (p.rows == 8 ? segmin_kernel<8, 4> : segmin_kernel<4, 4>);
    return launch(kernel, static_cast<unsigned>(blocks), 1, 32u * p.warps, smem, st, overlap, p);
}

}  // namespace plogp
