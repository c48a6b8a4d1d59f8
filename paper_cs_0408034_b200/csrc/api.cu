// Host side of the C ABI declared in include/plogp.h: argument validation, table upload, the
// launch plan for a grid (tiling, chunking of long candidate lists, scratch layout) and the
// kernel launches.  Every step of the evaluation itself runs on the device.
#include "../../include/plogp.h"
#include "internal.h"
#include "lines_layout.h"

#include <algorithm>
#include <atomic>
#include <cmath>
#include <cstring>
#include <exception>
#include <limits>
#include <new>
#include <string>
#include <vector>

using namespace plogp;

namespace {

thread_local std::string g_cuda_error;
std::atomic<unsigned long long> g_launches{0};

int cuda_fail(cudaError_t e, const char *what)
{
    try {
        g_cuda_error = std::string(what) + ": " + cudaGetErrorName(e) + " (" + cudaGetErrorString(e) + ")";
    } catch (const std::bad_alloc &) { g_cuda_error.clear(); }
    cudaGetLastError();  // clear the sticky-free error state
    return PLOGP_E_CUDA;
}

#define CK(call)                                                  \
    do {                                                          \
        cudaError_t e_ = (call);                                  \
        if (e_ != cudaSuccess) return cuda_fail(e_, #call);       \
    } while (0)

constexpr uint32_t kSegBits = (1u << 2) | (1u << 5) | (1u << 9);
constexpr uint64_t kTwo32 = 1ull << 32;
constexpr double kTwo53 = 9007199254740992.0;
constexpr int64_t kMaxP = int64_t(1) << 30;  // process counts: 32-bit tiling arithmetic and 1 << ceil(log2 P) stay in range
constexpr size_t kSweepScratchLimit = size_t(1) << 30;  // per launch batch of tables

int ceil_log2(int64_t P)
{
    int e = 0;
    while ((int64_t(1) << e) < P) ++e;
    return e;
}

// 2 floor(log2 P) + (P is no power of two): numbers the (floor, ceil) pairs in the order of P
int log2_pair(int64_t P) { return 2 * ceil_log2(P) - ((P & (P - 1)) ? 1 : 0); }

// Everything derived from a grid that the launches need.  A handle keeps the plans of the last kMaxPlans grids it was
// given (a tuner that asks for several collectives passes several masks in turn), each with its own device arrays.
constexpr size_t kMaxPlans = 8;
struct Plan {
    std::vector<unsigned char> key;  // serialised grid, for the cache comparison; empty: no plan
    unsigned char *d_grid = nullptr; // the grid's device arrays
    size_t grid_cap = 0;
    uint64_t used = 0;               // handle's tick of its last use
    bool empty = true;
    GridDev G{};
    int n_seg = 0;
    bool inline_sweep = true;
    bool envelope = false;        // envelope_kernel instead of the sweep kernel (long candidate lists)
    int env_threads = 256, env_rep_cap = 0, env_coarse_log = 5, env_max_coarse = 0;
    // fused kernel tiling
    int n_mtiles = 0, n_ptiles = 1, passes_per_tile = 1;
    // Scatter decision kernel: its own split of P (vec = 2: two message sizes per lane, where the outputs allow it)
    int sc_vec = 1, sc_ptiles = 1, sc_run = 1;
    // both halves in one launch, and then the Scatter half's split of P
    bool select = false;
    int sel_ptiles = 1, sel_run = 1;
    // tiling of decide_kernel and segmin_kernel (short candidate lists)
    struct Tiling {
        int width = 32, mgroups = 0, np = 512, ptiles = 1, pairs = 1;
        size_t off_knots = 0;
        bool gaps = false;  // run the gap pre-pass in front
    };
    Tiling ln, lp;      // of the decision and of the predictions
    int all_threads = 0;        // threads of a CTA that has all message sizes, or 0
    bool all_decide = false, all_predict = false;  // where such CTAs are taken, if two of them fit an SM
    bool all_alone = false;     // (predictions) or if one does
    bool dr_decide = false, dr_predict = false;  // small grids: a cell per thread
    int dr_ptiles = 1;
    // sweep kernel
    int n_pairs = 0, sweep_ptiles = 0, sweep_wp = 8, chunk_len = 0;
    size_t off_pair_m = 0, off_pair_chunk = 0, off_pair_row = 0, off_pair_base = 0;
    int tables_per_batch = 0;
    size_t scratch_bytes = 0;
    size_t off_k = 0;          // their k table inside the grid blob
    int gaps_stride = 0;       // doubles per table in its output
    size_t gaps_bytes_per_table = 0;
};

}  // namespace

struct plogp_tables {
    int device = 0;
    int sm_count = 148;
    TableDev T{};
    bool monotone = false;  // no table's gap ever decreases with the size (the envelope search relies on it)
    double *d_tab = nullptr;           // T.tab
    unsigned char *d_raw = nullptr;    // behind it, in the same allocation: the caller's arrays (T.lat first)
    std::vector<unsigned char> pack;   // the same on the host, kept for its memory
    unsigned char *d_ws = nullptr;
    size_t ws_cap = 0;
    std::vector<Plan> plans;
    uint64_t tick = 0;
    std::vector<unsigned char> key;  // of the grid at hand (kept for its memory)
    // optional per-kernel timing: event pairs recorded around every launch while enabled
    // host-output path: two device staging sets and a copy stream
    unsigned char *d_stage[2] = {nullptr, nullptr};
    size_t stage_cap = 0;
    cudaStream_t copy_stream = nullptr;
    cudaEvent_t ev_done[2] = {nullptr, nullptr}, ev_copied[2] = {nullptr, nullptr};
    bool profiling = false;
    struct Timed { int kind; cudaEvent_t a, b; };
    std::vector<Timed> timed;
};

namespace {

// Brackets one kernel launch with events on the caller's stream when timing is enabled.
struct LaunchTimer {
    plogp_tables *h;
    cudaStream_t st;
    cudaEvent_t a = nullptr, b = nullptr;
    int kind;
    LaunchTimer(plogp_tables *h_, int kind_, cudaStream_t st_) : h(h_), st(st_), kind(kind_)
    {
        if (!h->profiling) return;
        if (cudaEventCreate(&a) != cudaSuccess || cudaEventCreate(&b) != cudaSuccess || cudaEventRecord(a, st) != cudaSuccess) {
            if (a) cudaEventDestroy(a);
            if (b) cudaEventDestroy(b);
            a = b = nullptr;
            cudaGetLastError();
        }
    }
    ~LaunchTimer()
    {
        if (!a) return;
        bool kept = false;
        try {
            if (cudaEventRecord(b, st) == cudaSuccess) { h->timed.push_back({kind, a, b}); kept = true; }
        } catch (const std::bad_alloc &) {}
        if (!kept) { cudaEventDestroy(a); cudaEventDestroy(b); cudaGetLastError(); }
    }
};


template <typename V>
void put(std::vector<unsigned char> &buf, const V &v)
{
    const unsigned char *p = reinterpret_cast<const unsigned char *>(&v);
    buf.insert(buf.end(), p, p + sizeof(V));
}

template <typename V>
void put_array(std::vector<unsigned char> &buf, const V *v, size_t n)
{
    const unsigned char *p = reinterpret_cast<const unsigned char *>(v);
    buf.insert(buf.end(), p, p + n * sizeof(V));
}

template <typename V>
size_t append_aligned(std::vector<unsigned char> &blob, const std::vector<V> &v)
{
    while (blob.size() % 16) blob.push_back(0);
    const size_t off = blob.size();
    put_array(blob, v.data(), v.size());
    return off;
}

int validate_grid(const plogp_tables *h, const plogp_grid *g, int64_t *n_s_out)
{
    if (!g) return PLOGP_E_INVAL;
    if (g->strategy_mask >> PLOGP_N_STRATEGIES) return PLOGP_E_INVAL;
    if (g->k_mode != 0 && g->k_mode != 1) return PLOGP_E_INVAL;
    if (g->search_mode != 0 && g->search_mode != 1) return PLOGP_E_INVAL;
    if (g->dtype_bytes == 0) return PLOGP_E_INVAL;
    if (g->n_m < 0) return PLOGP_E_INVAL;
    if (g->n_m > 0 && !g->m) return PLOGP_E_INVAL;
    int64_t P_hi;
    if (g->P) {
        if (g->n_P < 0) return PLOGP_E_INVAL;
        for (int i = 0; i < g->n_P; ++i) {
            if (g->P[i] < 2) return PLOGP_E_INVAL;
            if (i && g->P[i] <= g->P[i - 1]) return PLOGP_E_INVAL;
        }
        P_hi = g->n_P ? g->P[g->n_P - 1] : 2;
    } else {
        if (g->P_lo < 2 || g->P_hi < g->P_lo) return PLOGP_E_INVAL;
        P_hi = g->P_hi;
    }
    if (P_hi > kMaxP) return PLOGP_E_RANGE;
    for (int i = 0; i < g->n_m; ++i) {
        const uint64_t m = g->m[i];
        if (m == 0 || m % g->dtype_bytes) return PLOGP_E_INVAL;
        if (i && m <= g->m[i - 1]) return PLOGP_E_INVAL;
        if (m >= kTwo32) return PLOGP_E_RANGE;
    }
    if (g->n_m > 0 && double(P_hi) * double(g->m[g->n_m - 1]) >= kTwo53) return PLOGP_E_RANGE;
    int64_t n_s = 0;
    if (g->strategy_mask & kSegBits) {
        if (g->s) {
            if (g->n_s < 0) return PLOGP_E_INVAL;
            for (int64_t i = 0; i < g->n_s; ++i) {
                const uint64_t s = g->s[i];
                if (s == 0 || s % g->dtype_bytes) return PLOGP_E_INVAL;
                if (i && s <= g->s[i - 1]) return PLOGP_E_INVAL;
                if (s >= kTwo32) return PLOGP_E_RANGE;
            }
            n_s = g->n_s;
        } else {
            if (g->s_step == 0 || g->s_step % g->dtype_bytes) return PLOGP_E_INVAL;
            if (g->s_lo == 0 || g->s_lo % g->dtype_bytes) return PLOGP_E_INVAL;
            if (g->s_hi >= g->s_lo) {
                if (g->s_hi >= kTwo32) return PLOGP_E_RANGE;
                n_s = int64_t((g->s_hi - g->s_lo) / g->s_step) + 1;
            }
        }
        if (n_s >= (int64_t(1) << 31)) return PLOGP_E_RANGE;
    }
    (void)h;
    *n_s_out = n_s;
    return PLOGP_OK;
}

// Grows the handle's scratch to what a plan needs.  Asked for by every call that launches kernels on it, with a kept plan too:
// a growth that fails for one grid leaves the handle without scratch for all of them.
int ensure_scratch(plogp_tables *h, size_t bytes)
{
    if (bytes <= h->ws_cap) return PLOGP_OK;
    if (h->d_ws) CK(cudaFree(h->d_ws));
    h->d_ws = nullptr;
    h->ws_cap = 0;
    cudaError_t e = cudaMalloc(&h->d_ws, bytes);
    if (e != cudaSuccess) h->d_ws = nullptr;
    if (e == cudaErrorMemoryAllocation) { cudaGetLastError(); return PLOGP_E_NOMEM; }
    if (e != cudaSuccess) return cuda_fail(e, "cudaMalloc(scratch)");
    h->ws_cap = bytes;
    return PLOGP_OK;
}

// Finds or builds the launch plan of a grid; *out is valid until the next call.  Throws where host memory runs out; a plan that
// was being built is then no plan.
int find_or_build(plogp_tables *h, const plogp_grid *g, cudaStream_t st, const Plan **out)
{
    if (!g || g->n_m < 0 || (g->n_m > 0 && !g->m)) return PLOGP_E_INVAL;
    if (g->P && g->n_P < 0) return PLOGP_E_INVAL;
    if ((g->strategy_mask & kSegBits) && g->s && g->n_s < 0) return PLOGP_E_INVAL;
    // ---- cache key: every input that the plan depends on ----
    std::vector<unsigned char> &key = h->key;
    key.clear();
    const int has_P = g->P != nullptr, has_s = g->s != nullptr;
    put(key, has_P);
    if (has_P) { put(key, g->n_P); put_array(key, g->P, size_t(std::max(g->n_P, 0))); }
    else { put(key, g->P_lo); put(key, g->P_hi); }
    put(key, g->n_m);
    put_array(key, g->m, size_t(std::max(g->n_m, 0)));
    put(key, g->strategy_mask); put(key, g->k_mode); put(key, g->dtype_bytes);
    put(key, g->search_mode); put(key, int(h->monotone));
    if (g->strategy_mask & kSegBits) {
        put(key, has_s);
        if (has_s) { put(key, g->n_s); put_array(key, g->s, size_t(std::max<int64_t>(g->n_s, 0))); }
        else { put(key, g->s_lo); put(key, g->s_hi); put(key, g->s_step); }
    }
    for (Plan &c : h->plans) {
        if (c.key != key) continue;
        c.used = ++h->tick;
        *out = &c;
        return PLOGP_OK;
    }

    int64_t n_s64 = 0;
    int rc = validate_grid(h, g, &n_s64);
    if (rc != PLOGP_OK) return rc;

    Plan pl;
    const int n_P = g->P ? g->n_P : (g->P_hi - g->P_lo + 1);
    const int n_m = g->n_m;
    const int n_s = int(n_s64);
    pl.empty = (n_P == 0 || n_m == 0 || g->strategy_mask == 0);
    if (h->plans.capacity() < kMaxPlans) h->plans.reserve(kMaxPlans);
    if (h->plans.size() < kMaxPlans) h->plans.emplace_back();
    // the newest slot is still without a key, else the one that was not used for longest gives way
    Plan &slot = h->plans.back().key.empty() ? h->plans.back()
                                             : *std::min_element(h->plans.begin(), h->plans.end(), [](const Plan &a, const Plan &b) { return a.used < b.used; });
    slot.key.clear();
    auto keep = [&]() {
        pl.d_grid = slot.d_grid; pl.grid_cap = slot.grid_cap;
        pl.key = key;
        pl.used = ++h->tick;
        slot = std::move(pl);
        *out = &slot;
        return int(PLOGP_OK);
    };
    if (pl.empty) return keep();

    const int64_t P_hi = g->P ? g->P[n_P - 1] : g->P_hi;
    pl.n_seg = __builtin_popcount(g->strategy_mask & kSegBits);
    pl.inline_sweep = pl.n_seg == 0 || n_s <= kMaxInlineS;
    // search_mode 1 on tables with non-decreasing gaps.  Long candidate lists: envelope_kernel writes the segmented
    // minima to the scratch rows that fused_kernel reads.  Short lists: decide_kernel and segmin_kernel, as with search_mode 0.
    const bool env_ok = g->search_mode == 1 && pl.n_seg > 0 && n_s > 0 && h->monotone;
    pl.envelope = env_ok && n_s > kMaxInlineS;
    if (pl.envelope) pl.inline_sweep = false;

    // candidates per message size (grid values s <= m)
    std::vector<int32_t> ns_of_m(n_m, 0);
    int ns_max = 0;
    if (pl.n_seg) {
        for (int i = 0; i < n_m; ++i) {
            const uint64_t m = g->m[i];
            int64_t c;
            if (g->s) c = std::upper_bound(g->s, g->s + n_s, m) - g->s;
            else {
                const uint64_t top = std::min<uint64_t>(m, g->s_hi);
                c = (n_s > 0 && top >= g->s_lo) ? int64_t((top - g->s_lo) / g->s_step) + 1 : 0;
            }
            ns_of_m[i] = int32_t(c);
            ns_max = std::max(ns_max, int(c));
        }
    }

    // ---- fused kernel tiling ----
    const int pass_P = kWarps * kFusedR;
    const int total_passes = (n_P + pass_P - 1) / pass_P;
    pl.n_mtiles = (n_m + 31) / 32;
    const long long base_blocks = (long long)pl.n_mtiles * h->T.n_tables;
    const long long target = (long long)h->sm_count * 8;
    int n_ptiles = 1;
    if (base_blocks < target) n_ptiles = int(std::min<long long>(total_passes, (target + base_blocks - 1) / base_blocks));
    n_ptiles = std::min(n_ptiles, 256);
    pl.passes_per_tile = (total_passes + n_ptiles - 1) / n_ptiles;
    pl.n_ptiles = (total_passes + pl.passes_per_tile - 1) / pl.passes_per_tile;
    // Two message sizes per lane halve the stores and the address arithmetic per cell: taken where the message sizes alone
    // give four CTAs per SM (4096 tables, P = 2..512, 128 m: 0.55 ms against 0.58) and leave no warp half empty.  Smaller
    // grids take one per lane (one table, P = 2..65536, 64 m: 17 us against 24, P = 2..1024, 256 m: 5.7 against 8.1) and
    // split the process counts over CTAs, 8 runs of at least 4 each, until four CTAs per SM are there.
    {
        const long long base = (long long)pl.n_mtiles * h->T.n_tables, want = (long long)h->sm_count * 4;
        pl.sc_vec = n_m % 2 == 0 && (n_m + 63) / 64 * 2 == pl.n_mtiles && base / 2 >= want ? 2 : 1;
        const long long split = std::max<long long>(1, (want + base - 1) / base);
        pl.sc_run = int(std::max<long long>(4, (n_P + kWarps * split - 1) / (kWarps * split)));
        pl.sc_ptiles = (n_P + kWarps * pl.sc_run - 1) / (kWarps * pl.sc_run);
    }

    // Tiling of decide_kernel and segmin_kernel: the width and the process counts of a CTA with the smallest number of CTAs (at
    // least what the GPU holds at once) times the instructions of one of its warps: 1000 for itself, 70 per candidate of a
    // group, 44 per process count of a group with 32 message sizes side by side, more with the shorter stores of fewer (4096
    // tables, P = 2..512, 32 candidates, on average; 72 message sizes 473 us with 8 side by side, 100 513 with 16, 50 253 with
    // 32).  Small grids so get many groups with few candidates each.
    // CTAs of the Scatter half, four warps each, for runs of at most 64 process counts: with longer ones its chains are what a launch of
    // both halves waits for (48 tables of 1384 x 24, 10 candidates 48.6 us, in two launches 18.9; 4 of 2696 x 33 16.8, where there had been
    // more room 11.5)
    const bool both = (g->strategy_mask & 0x3FFu) && (g->strategy_mask & 0x1C00u);
    const long long scatter_ctas = (long long)pl.n_mtiles * h->T.n_tables * ((n_P + 255) / 256);
    if (pl.inline_sweep && pl.n_seg > 0) {
        const long long hold = (long long)h->sm_count * 4;
        auto choose = [&](Plan::Tiling &best_tiling, long long floor, long long most) {  // with at most `most` CTAs; its cost, 0 if there is none
            long long best = 0;
            for (int width = 32; width >= 8; width >>= 1) {
                const int groups = kDecThreads / width;
                for (int np = 512; np >= groups * 8; np >>= 1) {
                    if (np > groups * 8 && np / 2 >= n_P) continue;
                    Plan::Tiling t;
                    t.width = width; t.np = np; t.mgroups = (n_m + width - 1) / width; t.ptiles = (n_P + np - 1) / np;
                    const long long ctas = (long long)t.mgroups * t.ptiles * h->T.n_tables;
                    const long long per_cta = 1000 + 70 * ((n_s + groups - 1) / groups) + np / groups * (width == 32 ? 44 : width == 16 ? 53 : 77);
                    const long long cost = std::max(ctas, floor) * per_cta;
                    if (ctas > most || (best && cost >= best)) continue;
                    best = cost;
                    best_tiling = t;
                }
            }
            return best;
        };
        const long long any = std::numeric_limits<long long>::max(), best = choose(pl.ln, hold, any);
        pl.lp = pl.ln;
        // Fewer and larger CTAs where the Scatter half then has room beside them in one launch (below) for runs of at most 32 process
        // counts (17 tables of 201 x 185, 8 candidates, with runs of 51 17.7 -> 22.0 us a call), for up to 1.45 of the instructions: 200 tables
        // of 99 x 9, 10 candidates 15.8 -> 11.0, 16 of 1023 x 64, 32 candidates 30.2 -> 16.7; at 1.64 (64 of 511 x 128, 32 candidates) 33.8 ->
        // 38.4, with 40 candidates, of which a group then has more (108 of 32 x 61) 11.6 -> 12.7.
        auto fits = [&](const Plan::Tiling &t) { return (long long)t.mgroups * t.ptiles * h->T.n_tables + scatter_ctas <= hold; };
        const long long lines_ctas = (long long)pl.ln.mgroups * pl.ln.ptiles * h->T.n_tables;
        if (n_s <= 32 && both && !fits(pl.ln)) {
            Plan::Tiling beside;
            const long long cost = choose(beside, hold, hold - (long long)pl.n_mtiles * h->T.n_tables * ((n_P + 127) / 128));
            if (cost && 20 * cost <= 29 * best) pl.ln = beside;
        }
        // Where another kernel of the call takes what is left of the GPU, the total counts more than a CTA's length: 34 tables of 134 x 126, 10
        // candidates 16.8 -> 12.0, 200 of 299 x 50, 30 candidates 39.3 -> 34.2, 159 of 594 x 9, 5 candidates 31.2 -> 26.0; with more
        // candidates, of which a group then has more, either way: 27 of 83 x 168, 34 candidates 15.1 -> 11.2, 64 of 511 x 128, 32 candidates 33.8
        // -> 35.7, 99 of 957 x 24, 62 candidates 73.9 -> 88.1 (two decisions).
        if (n_s <= 30 && both && !fits(pl.ln)) choose(pl.ln, hold / 2, any);
        // (predictions: 5 tables of 503 x 150, 20 candidates 16.6 -> 13.6, 22 of 31 x 163, 48 candidates 13.8 -> 10.7, 200 of 299 x 50, 30
        // candidates 95.7 -> 100.0; of few candidates, CTAs mostly set-up: 72 tables of 713 x 25, 4 candidates 40.8 -> 38.0; not where there are few
        // CTAs: 11 tables of 91 x 119, 8 candidates 8.1 -> 9.7)
        if (lines_ctas >= (long long)h->sm_count * 2) choose(pl.lp, n_s <= 8 ? hold / 4 : hold / 2, any);
        // A cell per thread (direct.cuh), 250 instructions and 30 per candidate: where that is half as many as a line for a range of
        // process counts, or no more and the GPU is nearly empty, so that only the length of a CTA counts.  Calls from a graph, lines ->
        // cells, us: one table, 49 process counts, 19 message sizes, 7 candidates 6.8 -> 4.6; 18 x 101, 48 candidates 8.7 -> 5.8; 3
        // tables of 74 x 8, 43 candidates 10.0 -> 6.8; 500 tables of 29 x 8, 5 candidates 13.0 -> 10.1, 2000 of 19 x 6, 4 candidates
        // 38.4 -> 24.6.  Past the line: 16 tables of 100 x 30, 20 candidates 8.0 -> 9.3, 128 of 63 x 16, 8 candidates 9.0 -> 10.3.  Tables of
        // more than 64 sizes, which each CTA stages and searches, only where there are many tables or hardly any CTAs: 21 of 51 x 43, 13
        // candidates, 16 / 64 / 128 / 200 sizes 7.3 7.7 8.7 10.5 -> 5.5 7.3 9.2 11.2, 500 of 29 x 8 12.0 13.1 14.4 15.5 -> 9.0 10.3 11.5 12.6.
        // And not where the launch of both halves would be lost.
        // Predictions, beside whose other planes' CTAs those of few tables are too many (21 of 51 x 43 7.1 -> 8.0, 100 of 60 x 12, 6
        // candidates 10.7 -> 8.5, 128 of 63 x 16 13.3 -> 11.9; 12 of 44 x 30, 41 candidates 7.9 -> 7.2; 511 x 64, 32 candidates 8.1 -> 9.0).
        const long long ctas = ((long long)n_P * n_m + kDecThreads - 1) / kDecThreads * h->T.n_tables;
        const long long cost = std::max(ctas, (long long)h->sm_count * 4) * (250 + 30 * n_s);
        const int npad = h->T.npad, sms = h->sm_count;
        const bool launch_more = both && fits(pl.ln) && ctas + scatter_ctas > sms * 6;  // 9 tables of 668 x 19, 7 candidates 8.0 -> 10.8
        pl.dr_decide = ((!launch_more && (npad <= 64 || h->T.n_tables >= 256)) && (npad <= 32 ? 5 * cost < 3 * best : 2 * cost < best)) ||
                       (npad <= 128 && cost < best && 2 * ctas <= sms * (npad <= 64 ? 4 : 3));
        pl.dr_predict = (h->T.n_tables >= 64 && 5 * cost < 3 * best) || (npad <= 128 && cost < best && ctas * (npad <= 64 ? 1 : 2) <= sms);
        pl.dr_ptiles = int(ctas / h->T.n_tables);
        // All message sizes in a CTA (STAGED, lines.cuh), for rows off the sectors: threads for as many groups as leave the fewest
        // idle.  Worth it where a CTA's process counts make up for its set-up, on grids of several CTAs per SM.
        if (n_m > 32 && n_m <= kLineThreads) {
            double busy = 0.0;
            for (int t = 128; t <= kLineThreads; t += 32) {
                const double b = double(t / n_m * n_m) / t;
                if (b >= busy) { busy = b; pl.all_threads = t; }
            }
            const double busy_lines = double(n_m) / (pl.ln.mgroups * pl.ln.width);
            const long long d_ctas = (long long)pl.ln.ptiles * h->T.n_tables, p_ctas = (long long)pl.lp.ptiles * h->T.n_tables;
            // Decision, odd rows only: with half the bytes of a plane the waits weigh more.  Time with row segments = 1, 8 / 16 / 29 candidates:
            //   223 tables of 1832 process counts, 33 message sizes 0.82 0.85 0.92, 65 0.93 0.98 1.11, 99 0.79 0.83 0.94, 137 0.74 0.95 1.09
            //   1200 of 511                         33 0.90 0.92 1.04, 65 1.05 1.08 1.27, 99 0.88 0.93 1.08, 161 0.91 0.96 1.10
            //   1200 of 172                         33 1.04 1.01 0.98, 65 1.14 1.15 1.15, 99 1.14 1.15 1.19, 195 1.14 1.18 1.23
            //   2048 of 100 (8 / 20 / 32)           33 0.93 0.89 0.84, 65 0.97 0.97 0.96, 99 0.95 0.96 0.98, 201 0.92 0.95 0.97, 127 1.04 1.05 1.06
            //   2048 of 28                          33 1.07 1.00 0.91, 65 0.95 0.95 0.91, 99 0.84 0.85 0.85, 161 0.81 0.85 0.88, 47 1.08 1.04 1.03
            //   2048 of 14                          33 1.14 1.04 0.95, 65 0.83 0.83 0.82, 99 0.75 0.76 0.78, 161 0.68 0.73 0.78
            // and 600 tables of 511, 127 message sizes 0.97 1.01 1.12, 320 of 199 1.58 1.57 1.53; fewer CTAs for the longest and the shortest
            // ranges only (100 of 2097, 109 message sizes, 16 candidates 0.92; 303 of 31, 189 message sizes, 4 candidates 0.91).
            const int d_least = n_P >= 1024 && n_s <= 16 ? 3 : n_P <= 48 && n_m >= 128 ? 2 : 6;
            pl.all_decide = n_m % 2 != 0 && d_ctas >= (long long)h->sm_count * d_least &&
                            (n_P <= 48   ? n_m >= 64
                             : n_P < 256 ? (n_P >= 96 && busy >= 1.1 * busy_lines) || (n_P <= 128 && n_m >= 192 && n_s <= 16)
                                         : n_s <= (n_P >= 700 ? 32 : 24) && (n_m >= 72 || busy >= 0.88));
            // Predictions, rows off the sectors of the sizes, or of times and sizes.  The same:
            //   1200 tables of 511                  33 0.57 0.58 0.63, 65 0.62 0.65 0.72, 99 0.57 0.60 0.66, 161 0.64 0.66 0.74, 100 (whole sectors of
            //                                       times; 8 / 20 / 32) 0.70 0.77 0.85
            //   1200 of 172                         33 0.99 1.03 1.13, 47 0.83 0.86 0.97, 99 0.67 0.71 0.81, 161 0.72 0.76 0.87
            //   2048 of 100 (8 / 20 / 32)           33 1.07 1.04 1.00, 65 0.91 1.07 1.14, 99 0.76 0.87 0.98, 201 0.70 0.81 0.91, 100 1.21 1.26 1.27
            //   2048 of 28                          65 1.08 1.10 1.09, 99 1.01 1.01 1.03, 137 0.89 0.95 1.00, 255 0.87 0.91
            //   2048 of 14                          33 1.30 1.18 1.10, 65 0.99 0.98 0.96, 99 0.86 0.86 0.88, 161 0.82 0.86 0.90
            // and 4000 of 59, 99 1.11 1.14 1.22, 255 0.86 0.93; 320 of 199, 99 1.01 1.02 1.15; 112 of 1776, 117 message sizes, 31 candidates 0.91.
            const bool rows_long = n_m % 4 == 0 ? n_P >= 256 && n_s <= 32 : n_P >= (n_m >= 96 ? 96 : n_m >= 44 ? 160 : 192);
            const bool rows_few = n_m % 4 != 0 && ((n_P <= 20 && n_m >= 64) || (n_s <= 16 && n_m >= (n_P <= 48 ? 128 : 192)));
            pl.all_predict = n_m % 8 != 0 && p_ctas >= (long long)h->sm_count * (n_P >= 1024 ? 2 : 4) && (rows_long || rows_few);
            // One CTA per SM: 1200 tables of 511 process counts, 20 / 32 / 48 candidates: 255 0.79 0.87 0.99, 250 0.83 0.94 1.07, 201 at 32
            // 0.96, at 48 1.13; 173 at 32 1.10, 127 at 48 1.05; 148 of 2999, 48 candidates 255 0.89, 250 0.98; 2048 of 200, 255 0.80 0.92 1.09;
            // 1200 of 172, 255 at 16 0.90, at 29 1.06.
            pl.all_alone = n_m % 4 != 0 && n_m > 192 && n_s <= (n_P >= 1024 ? 48 : n_P >= 192 ? 32 : 16) && n_P >= 160;
        }
    }
    // One launch for both halves where the GPU holds all their CTAs at once (four per SM, six with a cell per thread; its Scatter CTAs
    // have four warps)
    if (pl.ln.mgroups > 0 && both) {
        const long long base = (long long)pl.n_mtiles * h->T.n_tables, hold = (long long)h->sm_count * (pl.dr_decide ? 6 : 4);
        const long long decide = (pl.dr_decide ? (long long)pl.dr_ptiles : (long long)pl.ln.mgroups * pl.ln.ptiles) * h->T.n_tables, room = hold - decide;
        pl.select = room >= scatter_ctas;
        if (pl.select) {
            pl.sel_run = int(std::max<long long>(4, (n_P + kDecWarps * (room / base) - 1) / (kDecWarps * (room / base))));
            pl.sel_ptiles = (n_P + kDecWarps * pl.sel_run - 1) / (kDecWarps * pl.sel_run);
        }
    }
    // Knots: the ends of up to kLineSegs segments of a CTA's process counts, by the ratio of process counts, on the last one of
    // a step of eight
    auto knots_of = [&](Plan::Tiling &tiling) {
        std::vector<int32_t> knots;
        for (int t = 0; t < tiling.ptiles; ++t) {
            const int first = t * tiling.np, n = std::min(n_P, first + tiling.np) - first;
            auto P_at = [&](int i) { return g->P ? int64_t(g->P[first + i]) : int64_t(g->P_lo) + first + i; };
            tiling.pairs = std::max(tiling.pairs, log2_pair(P_at(n - 1)) - log2_pair(P_at(0)) + 1);
            const size_t at = knots.size();
            knots.resize(at + kLineSegs + 2, n - 1);
            int n_segs = 0, end = 0;
            knots[at] = 0;
            while (end < n - 1) {
                const int left = kLineSegs - n_segs;
                const double ratio = std::max(2.0, std::pow(double(P_at(n - 1)) / double(P_at(end)), 1.0 / left));
                int next = std::min(n - 1, end == 0 ? 7 : end + 8);
                while (next < n - 1 && (left == 1 || double(P_at(std::min(n - 1, next + 8))) <= ratio * double(P_at(end)))) next = std::min(n - 1, next + 8);
                knots[at + ++n_segs] = end = next;
            }
            if (n_segs == 0) n_segs = 1;  // one process count
            knots[at + kLineSegs + 1] = n_segs;
        }
        return knots;
    };

    // ---- device arrays ----
    std::vector<unsigned char> blob;
    std::vector<uint32_t> m32(n_m);
    for (int i = 0; i < n_m; ++i) m32[i] = uint32_t(g->m[i]);
    const size_t off_m = append_aligned(blob, m32);
    const size_t off_ns = append_aligned(blob, ns_of_m);
    size_t off_P = 0, off_s = 0;
    if (g->P) off_P = append_aligned(blob, std::vector<int32_t>(g->P, g->P + n_P));
    if (pl.n_seg && g->s) {
        std::vector<uint32_t> s32(n_s);
        for (int i = 0; i < n_s; ++i) s32[i] = uint32_t(g->s[i]);
        off_s = append_aligned(blob, s32);
    }

    if (pl.ln.mgroups > 0) {
        pl.ln.off_knots = append_aligned(blob, knots_of(pl.ln));
        pl.lp.off_knots = append_aligned(blob, knots_of(pl.lp));
    }
    // Short candidate lists: Section 2's k for every (candidate, m), as the doubles the kernels multiply with
    const bool short_lists = pl.inline_sweep && pl.n_seg > 0 && n_s > 0;
    if (short_lists) {
        std::vector<double> kt(size_t(n_s) * n_m, 1.0);
        for (int i = 0; i < n_m; ++i) {
            const uint64_t m = g->m[i];
            for (int c = 0; c < ns_of_m[i]; ++c) {
                const uint64_t sv = g->s ? g->s[c] : g->s_lo + uint64_t(c) * g->s_step;
                const uint64_t q = m / sv;
                kt[size_t(c) * n_m + i] = double(q + ((g->k_mode == 0 && q * sv != m) ? 1 : 0));
            }
        }
        pl.off_k = append_aligned(blob, kt);
    }

    // ---- sweep kernel plan: (m, chunk) pairs, heaviest first ----
    if (pl.envelope) {
        // one scratch row per message size
        std::vector<int32_t> pair_base(n_m + 1);
        for (int i = 0; i <= n_m; ++i) pair_base[i] = i;
        pl.n_pairs = n_m;
        pl.off_pair_base = append_aligned(blob, pair_base);
        // short lists: small CTAs; the list of representatives of one message size lives in shared memory
        pl.env_threads = ns_max <= 64 ? 64 : (ns_max <= 4096 ? 256 : 1024);
        pl.env_rep_cap = std::min(std::max(ns_max, 1), 6144);
        pl.env_coarse_log = 5;
        while ((2 << pl.env_coarse_log) < (n_P + 1023) / 1024) ++pl.env_coarse_log;
        pl.env_max_coarse = envelope_coarse_of(n_P - 1, pl.env_coarse_log) + 2;
    } else if (!pl.inline_sweep) {
        const int p_tiles = (n_P + 32 * kSweepR - 1) / (32 * kSweepR);
        pl.sweep_wp = kWarps;
        while (pl.sweep_wp > 1 && pl.sweep_wp / 2 >= p_tiles - 1) pl.sweep_wp >>= 1;
        pl.sweep_ptiles = 1 + (p_tiles - 1 + pl.sweep_wp - 1) / pl.sweep_wp;
        // Chunks: about six CTAs per SM, a CTA's upper bounds cost as much as 25 sub-chunks
        long long cands = 0;
        for (int i = 0; i < n_m; ++i) cands += ns_of_m[i];
        const long long share = cands * pl.sweep_ptiles * h->T.n_tables / ((long long)h->sm_count * 6);
        const auto whole_subs = [](long long n) { return (n + kSweepSub - 1) / kSweepSub * kSweepSub; };
        long long chunk = std::min<long long>(std::max(std::min(std::max<long long>(2048, whole_subs(share)), whole_subs(ns_max)), (long long)kSweepSub), 1 << 20);
        // but no more of them than 32 per message size where a table's partial minima would not fit the scratch of a launch
        const long long longest = whole_subs((ns_max + 31LL) / 32);
        const auto partials = [&]() {
            long long n = 0;
            for (int i = 0; i < n_m; ++i) n += (ns_of_m[i] + chunk - 1) / chunk;
            return double(n) * pl.n_seg * n_P * (sizeof(double) + sizeof(uint32_t));
        };
        while (chunk < longest && partials() > double(kSweepScratchLimit)) chunk = std::min(2 * chunk, longest);
        pl.chunk_len = int(chunk);
        std::vector<int32_t> pair_base(n_m + 1, 0);
        struct Pair { int32_t m, chunk, row, len; };
        std::vector<Pair> pairs;
        for (int i = 0; i < n_m; ++i) {
            pair_base[i] = int32_t(pairs.size());
            for (int c = 0; (long long)c * pl.chunk_len < ns_of_m[i]; ++c)
                pairs.push_back({i, c, int32_t(pairs.size()), std::min(pl.chunk_len, ns_of_m[i] - c * pl.chunk_len)});
        }
        pair_base[n_m] = int32_t(pairs.size());
        pl.n_pairs = int(pairs.size());
        std::stable_sort(pairs.begin(), pairs.end(), [](const Pair &a, const Pair &b) { return a.len > b.len; });
        std::vector<int32_t> pm(pl.n_pairs), pc(pl.n_pairs), pr(pl.n_pairs);
        for (int i = 0; i < pl.n_pairs; ++i) { pm[i] = pairs[i].m; pc[i] = pairs[i].chunk; pr[i] = pairs[i].row; }
        pl.off_pair_m = append_aligned(blob, pm);
        pl.off_pair_chunk = append_aligned(blob, pc);
        pl.off_pair_row = append_aligned(blob, pr);
        pl.off_pair_base = append_aligned(blob, pair_base);
    }

    if (blob.size() > slot.grid_cap) {
        if (slot.d_grid) CK(cudaFree(slot.d_grid));
        slot.d_grid = nullptr;
        slot.grid_cap = 0;
        const size_t cap = std::max<size_t>(blob.size() + blob.size() / 4, 4096);
        const cudaError_t e = cudaMalloc(&slot.d_grid, cap);
        if (e != cudaSuccess) slot.d_grid = nullptr;
        if (e == cudaErrorMemoryAllocation) { cudaGetLastError(); return PLOGP_E_NOMEM; }
        if (e != cudaSuccess) return cuda_fail(e, "cudaMalloc(grid)");
        slot.grid_cap = cap;
    }
    // The source is pageable host memory: the runtime stages it before returning.
    CK(cudaMemcpyAsync(slot.d_grid, blob.data(), blob.size(), cudaMemcpyHostToDevice, st));

    GridDev &G = pl.G;
    G.P_list = g->P ? reinterpret_cast<const int32_t *>(slot.d_grid + off_P) : nullptr;
    G.n_P = n_P;
    G.P_lo = g->P ? 0 : g->P_lo;
    G.m_list = reinterpret_cast<const uint32_t *>(slot.d_grid + off_m);
    G.n_m = n_m;
    G.s_list = (pl.n_seg && g->s) ? reinterpret_cast<const uint32_t *>(slot.d_grid + off_s) : nullptr;
    G.n_s = pl.n_seg ? n_s : 0;
    G.s_lo = uint32_t(g->s_lo);
    G.s_step = uint32_t(g->s_step);
    G.ns_of_m = reinterpret_cast<const int32_t *>(slot.d_grid + off_ns);
    G.k_list = short_lists ? reinterpret_cast<const double *>(slot.d_grid + pl.off_k) : nullptr;
    G.mask = g->strategy_mask;
    G.k_mode = g->k_mode;
    G.lc_max = std::max(1, ceil_log2(P_hi));

    // ---- scratch: sweep partials (per table batch), gap rows ----
    size_t per_table = 0;
    if (!pl.inline_sweep) per_table += size_t(pl.n_seg) * pl.n_pairs * n_P * (sizeof(double) + sizeof(uint32_t)) + 512;
    // The gap pre-pass costs a launch: taken where decide_kernel and segmin_kernel run many CTAs per table and fill the GPU several times over
    // (4096 tables, P = 2..512, 128 m, 32 sizes: 1290 -> 1280 us)
    if (pl.inline_sweep && pl.n_seg > 0) {
        for (Plan::Tiling *tiling : {&pl.ln, &pl.lp}) {
            const long long ctas_per_table = (long long)tiling->mgroups * tiling->ptiles;
            tiling->gaps = ctas_per_table >= 4 && ctas_per_table * h->T.n_tables >= (long long)h->sm_count * 16;
        }
        pl.ln.gaps &= !pl.dr_decide;
        pl.lp.gaps &= !pl.dr_predict;
        if (pl.ln.gaps || pl.lp.gaps) {
            pl.gaps_stride = (1 + n_s + n_m + 1) & ~1;
            pl.gaps_bytes_per_table = size_t(pl.gaps_stride) * sizeof(double);
            per_table += pl.gaps_bytes_per_table;
        }
    }
    pl.tables_per_batch = h->T.n_tables;
    if (!pl.inline_sweep && per_table * h->T.n_tables > kSweepScratchLimit)
        pl.tables_per_batch = int(std::max<size_t>(1, kSweepScratchLimit / per_table));
    pl.tables_per_batch = std::min(pl.tables_per_batch, 65535);
    pl.scratch_bytes = per_table ? per_table * pl.tables_per_batch + 1024 : 0;  // the sections start on 256-byte boundaries
    rc = ensure_scratch(h, pl.scratch_bytes);
    return rc == PLOGP_OK ? keep() : rc;
}

// The same for the C calls, which throw nothing
int prepare(plogp_tables *h, const plogp_grid *g, cudaStream_t st, const Plan **out)
{
    try {
        return find_or_build(h, g, st, out);
    } catch (const std::exception &) { return PLOGP_E_NOMEM; }  // bad_alloc, or a length no vector can have
}

size_t align_up(size_t x, size_t a) { return (x + a - 1) / a * a; }

// plogp_select_best's layout: two planes per table, the ids of Table 1 / Table 2
OutMap default_out_map()
{
    OutMap om{};
    om.planes = 2; om.plane_bcast = 0; om.plane_scat = 1;
    for (int i = 0; i < 16; ++i) om.id_of[i] = uint8_t(i < PLOGP_N_STRATEGIES ? i : 255);
    return om;
}

int run(plogp_tables *h, const plogp_grid *g, bool predict, FusedParams out, cudaStream_t st, int t_begin = 0, int t_end = -1)
{
    int dev = 0;
    CK(cudaGetDevice(&dev));
    if (dev != h->device) return PLOGP_E_INVAL;
    const Plan *plan = nullptr;
    int rc = prepare(h, g, st, &plan);
    if (rc != PLOGP_OK) return rc;
    const Plan &pl = *plan;
    if (pl.empty) return PLOGP_OK;
    rc = ensure_scratch(h, pl.scratch_bytes);
    if (rc != PLOGP_OK) return rc;
    // Decision tables on short candidate lists with segmented strategies: decide_kernel for the Broadcast half
    // (select_kernel for both halves of a small one).  What is left of a decision table, if only Scatter strategies, goes to
    // scatter_kernel or scatter_rows_kernel; predictions to segmin_kernel, then planes_kernel, scatter_rows_kernel and
    // fused_kernel; long lists, reduced by sweep_kernel or envelope_kernel, to fused_kernel.
    const bool use_decide = !predict && pl.inline_sweep && pl.n_seg > 0;
    // the kernel that follows the (optional) Broadcast decision kernel: Scatter strategies only => scatter_kernel
    const bool use_scatter = !predict && ((use_decide ? pl.G.mask & 0x1C00u : pl.G.mask) & 0x3FFu) == 0;

    const bool overlap = !h->profiling;  // the times of overlapping kernels would not add up
    if (t_end < 0) t_end = h->T.n_tables;
    for (int t0 = t_begin; t0 < t_end; t0 += pl.tables_per_batch) {
        const int nt = std::min(pl.tables_per_batch, t_end - t0);
        unsigned char *ws = h->d_ws;
        double *part_time = nullptr;
        uint32_t *part_idx = nullptr;
        if (!pl.inline_sweep) {
            const size_t cells = size_t(nt) * pl.n_seg * pl.n_pairs * pl.G.n_P;
            part_time = reinterpret_cast<double *>(ws);
            ws += align_up(cells * sizeof(double), 256);
            part_idx = reinterpret_cast<uint32_t *>(ws);
            ws += align_up(cells * sizeof(uint32_t), 256);
        }
        double *gaps = nullptr;
        if (predict ? pl.lp.gaps : use_decide && pl.ln.gaps) {
            gaps = reinterpret_cast<double *>(ws);
            GapsParams gp{};
            gp.T = h->T; gp.G = pl.G;
            gp.table0 = t0; gp.n_tables_launch = nt; gp.gaps = gaps; gp.stride = pl.gaps_stride;
            { LaunchTimer lt(h, PLOGP_KERNEL_GAPS, st); CK(launch_gaps(gp, st)); }
            g_launches += 1;
        }

        if (pl.envelope) {
            EnvParams ep{};
            ep.T = h->T; ep.G = pl.G;
            ep.table0 = t0; ep.n_tables_launch = nt;
            ep.part_time = part_time; ep.part_idx = part_idx; ep.n_seg = pl.n_seg;
            ep.rep_cap = pl.env_rep_cap; ep.coarse_log = pl.env_coarse_log; ep.max_coarse = pl.env_max_coarse;
            { LaunchTimer lt(h, PLOGP_KERNEL_ENVELOPE, st); CK(launch_envelope(ep, pl.env_threads, st)); }
            g_launches += 1;
        } else if (!pl.inline_sweep && pl.n_pairs > 0) {
            SweepParams sp{};
            sp.T = h->T; sp.G = pl.G;
            sp.pair_m = reinterpret_cast<const int32_t *>(pl.d_grid + pl.off_pair_m);
            sp.pair_chunk = reinterpret_cast<const int32_t *>(pl.d_grid + pl.off_pair_chunk);
            sp.pair_row = reinterpret_cast<const int32_t *>(pl.d_grid + pl.off_pair_row);
            sp.n_pairs = pl.n_pairs; sp.n_ptiles = pl.sweep_ptiles; sp.chunk_len = pl.chunk_len; sp.wp = pl.sweep_wp;
            sp.part_time = part_time; sp.part_idx = part_idx; sp.n_seg = pl.n_seg; sp.table0 = t0;
            int n_launches = 0;
            { LaunchTimer lt(h, PLOGP_KERNEL_SWEEP, st); CK(launch_sweep(sp, nt, &n_launches, st)); }
            g_launches += unsigned(n_launches);
        }
        GridDev Gf = pl.G;
        auto lines = [&]() {
            LinesParams lp{};
            lp.T = h->T; lp.G = pl.G;
            const Plan::Tiling &t = predict ? pl.lp : pl.ln;
            lp.width = t.width; lp.threads = kDecThreads; lp.n_mgroups = t.mgroups; lp.n_p = t.np; lp.n_ptiles = t.ptiles; lp.n_pairs = t.pairs;
            lp.knots = reinterpret_cast<const int32_t *>(pl.d_grid + t.off_knots);
            lp.gaps = gaps; lp.gaps_stride = pl.gaps_stride;
            lp.table0 = t0; lp.n_tables_launch = nt; lp.out_table0 = out.out_table0; lp.om = out.om;
            if (predict ? pl.dr_predict : pl.dr_decide) { lp.direct = 1; lp.n_mgroups = 1; lp.n_ptiles = pl.dr_ptiles; }
            return lp;
        };
        // All message sizes in a CTA, where two of them fit an SM (228 KB, 1 KB of it each CTA's own): the shared memory grows with
        // message sizes times candidates and times (floor, ceil) pairs, past what a CTA can have.  With one per SM (1200 tables of 511
        // process counts, 48 candidates, 127 / 173 / 255 message sizes) the decision takes 1.80 / 2.02 / 1.56 times as long as row segments.
        auto stage = [&](LinesParams &lp, size_t most) {
            LinesParams whole = lp;
            whole.staged = 1; whole.width = pl.G.n_m; whole.n_mgroups = 1; whole.threads = pl.all_threads;
            if (lines_smem_bytes(whole) <= most) lp = whole;
        };
        constexpr size_t kHalf = 113 * 1024;
        if (predict && pl.inline_sweep && pl.n_seg > 0) {
            // Predictions on short candidate lists: the segmented minima (planes 2, 5, 9 and the best segment sizes)
            // come from segmin_kernel; the kernels behind it write the other planes.
            LinesParams sp = lines();
            sp.p_time = out.p_time; sp.p_best_s = out.p_best_s;
            if (!sp.direct && pl.all_predict && reinterpret_cast<uintptr_t>(out.p_time) % 32 == 0 && reinterpret_cast<uintptr_t>(out.p_best_s) % 16 == 0)
                stage(sp, pl.all_alone ? size_t(kMaxSmem) : kHalf);
            { LaunchTimer lt(h, PLOGP_KERNEL_SEGMIN, st); CK(launch_segmin(sp, overlap && gaps, st)); }
            g_launches += 1;
            Gf.mask &= ~kSegBits;
            Gf.n_s = 0;
            if (!Gf.mask) continue;
        }
        if (use_decide) {
            // Broadcast half; the Scatter half (no candidate lists) beside it or in the kernel behind it
            LinesParams dp = lines();
            dp.G.mask &= 0x3FFu;
            dp.d_strategy = out.d_strategy; dp.d_sbytes = out.d_sbytes; dp.d_time = out.d_time;
            if (pl.select && !gaps && overlap) {
                SelectParams sl{};
                sl.decide = dp;
                ScatterParams &sc = sl.scatter;
                sc.T = h->T; sc.G = pl.G;
                sc.vec = 1; sc.n_mtiles = pl.n_mtiles; sc.n_ptiles = pl.sel_ptiles; sc.run_len = pl.sel_run;
                sc.table0 = t0; sc.n_tables_launch = nt; sc.out_table0 = out.out_table0; sc.om = out.om;
                sc.d_strategy = out.d_strategy; sc.d_sbytes = out.d_sbytes; sc.d_time = out.d_time;
                CK(launch_select(sl, st));
                g_launches += 1;
                continue;
            }
            if (!dp.direct && pl.all_decide && reinterpret_cast<uintptr_t>(out.d_time) % 32 == 0 && reinterpret_cast<uintptr_t>(out.d_sbytes) % 16 == 0 &&
                reinterpret_cast<uintptr_t>(out.d_strategy) % 4 == 0) stage(dp, kHalf);
            { LaunchTimer lt(h, PLOGP_KERNEL_DECIDE, st); CK(launch_decide(dp, overlap && gaps, st)); }
            g_launches += 1;
            Gf.mask &= 0x1C00u;
            Gf.n_s = 0;
            if (!Gf.mask) continue;
        }
        // Rows of message sizes that are no multiple of a 32-byte sector: the Scatter sums go out as one piece per CTA (rows.cu).
        // Decision tables, 32 sizes, without -> with: 2048 tables, P = 2..513, n_m = 127 1.83 -> 1.45 ms, 130 1.88 -> 1.58, 145
        // 2.16 -> 1.74, 66 0.98 -> 0.83, whole sectors 132 1.64 -> 1.56, 136 1.52 -> 1.59 and 72 0.84 -> 0.87.  A warp more for
        // a few message sizes past 32 costs what it gains (42: 0.525 -> 0.546 ms, 46 of 4096 tables 560 -> 552 us); what the L2
        // takes gains nothing (200 tables 207 -> 205 us); a CTA sums up in front of its run what eight warps did elsewhere, so
        // its run is at least as long as the table (1024 tables of 200 sizes 947 -> 818 us, 512 of 256 497 -> 451, of 1000 sizes
        // 1104 -> 1202) and at most 256, split until there are 16 CTAs per SM.  Listed process counts are summed up by intervals,
        // which is most of a cell there (1000 tables, 203 process counts, 101 m: 339 -> 370 us).
        const size_t cells = size_t(pl.G.n_P) * pl.G.n_m;
        const bool rows_off = !pl.G.P_list && pl.G.n_m % 4 != 0 && pl.G.n_m >= 44 && pl.G.n_m <= kRowsMaxM && h->T.npad <= 256 && cells * nt >= (size_t(1) << 23);
        RowsParams rp{};
        rp.T = h->T; rp.G = Gf;
        rp.run_len = std::min(pl.G.n_P, std::max(h->T.n_bp, int(std::min<long long>(256, (long long)pl.G.n_P * nt / (h->sm_count * 16LL)))));
        rp.n_ptiles = (pl.G.n_P + rp.run_len - 1) / rp.run_len;
        rp.table0 = t0; rp.n_tables_launch = nt; rp.out_table0 = out.out_table0;
        if (use_scatter && rows_off && reinterpret_cast<uintptr_t>(out.d_time) % 32 == 0 && reinterpret_cast<uintptr_t>(out.d_sbytes) % 16 == 0 &&
            reinterpret_cast<uintptr_t>(out.d_strategy) % 4 == 0) {
            rp.om = out.om;
            rp.d_strategy = out.d_strategy; rp.d_sbytes = out.d_sbytes; rp.d_time = out.d_time;
            { LaunchTimer lt(h, PLOGP_KERNEL_SCATTER, st); CK(launch_rows(rp, false, overlap && use_decide, st)); }
            g_launches += 1;
            continue;
        }
        if (use_scatter) {
            ScatterParams sc{};
            sc.T = h->T; sc.G = Gf;
            const bool aligned = reinterpret_cast<uintptr_t>(out.d_time) % 16 == 0 && reinterpret_cast<uintptr_t>(out.d_sbytes) % 8 == 0 &&
                                 reinterpret_cast<uintptr_t>(out.d_strategy) % 2 == 0;
            // The table of sums is built by every CTA and takes 512 bytes per interval: 1000 tables, 200 process counts, 128 m,
            // closed forms along the run -> table: 64 sizes 449 -> 429 us, 128 468 -> 471, 200 486 -> 542.
            sc.chain_table = pl.G.P_list && h->T.n_bp <= 96;
            sc.vec = aligned && !sc.chain_table ? pl.sc_vec : 1;
            sc.n_mtiles = (pl.G.n_m + 32 * sc.vec - 1) / (32 * sc.vec);
            sc.n_ptiles = pl.sc_ptiles; sc.run_len = pl.sc_run;
            sc.table0 = t0; sc.n_tables_launch = nt; sc.out_table0 = out.out_table0; sc.om = out.om;
            sc.d_strategy = out.d_strategy; sc.d_sbytes = out.d_sbytes; sc.d_time = out.d_time;
            { LaunchTimer lt(h, PLOGP_KERNEL_SCATTER, st); CK(launch_scatter(sc, overlap && use_decide, st)); }
            g_launches += 1;
            continue;
        }
        bool behind = pl.n_seg > 0 && (!pl.inline_sweep ? pl.envelope || pl.n_pairs > 0 : predict);  // a kernel of this call is in front
        // Rows that are no multiple of a 32-byte sector: the planes that need no sum along P are written cell by cell as they
        // lie in memory (planes.cu).  Whole calls, all ids, 32 sizes, without -> with: 1024 tables, P = 2..513, n_m = 127 3.34 ->
        // 2.36 ms, 33 1.05 -> 0.86, whole sectors 136 2.05 -> 1.98 and 72 1.07 -> 1.10.  It is one launch more, so the line is
        // where it starts to gain: rows of one warp are written one after another anyhow (n_m = 17: 0.40 -> 0.46 ms), planes of
        // few rows spend it on their set-up (P = 2..101, 145 m, 4000 tables 2.37 -> 2.40, P = 2..201, 2000 tables 2.64 -> 2.14),
        // and the L2 takes what is smaller than it (P = 2..512, 99 m: 32 tables 92 -> 93 us, 100 300 -> 277).
        if (predict && pl.inline_sweep && pl.G.n_m % 4 != 0 && pl.G.n_m > 32 && pl.G.n_m <= kPlanesMaxM && pl.G.n_P >= 160 && cells * nt >= (size_t(1) << 22)) {
            PlanesParams pp{};
            pp.T = h->T; pp.G = pl.G; pp.mask = Gf.mask & kPlanesMask;
            // whole planes per CTA, split while that leaves fewer than eight CTAs per SM
            const size_t split = std::max<size_t>(1, (size_t(h->sm_count) * 8 + nt - 1) / nt);
            pp.seg_cells = (long long)std::max<size_t>(2048, ((cells + 31 + split - 1) / split + 255) / 256 * 256);
            pp.table0 = t0; pp.n_tables_launch = nt; pp.out_table0 = out.out_table0; pp.p_time = out.p_time;
            if (pp.mask) {
                { LaunchTimer lt(h, PLOGP_KERNEL_FUSED, st); CK(launch_planes(pp, overlap && behind, st)); }
                g_launches += 1;
                behind = true;
                Gf.mask &= ~kPlanesMask;
                if (!Gf.mask) continue;
            }
            if (rows_off && !(Gf.mask & ~0x1800u) && reinterpret_cast<uintptr_t>(out.p_time) % 32 == 0) {
                rp.G = Gf;
                rp.om.planes = 13;
                rp.d_time = out.p_time;
                { LaunchTimer lt(h, PLOGP_KERNEL_FUSED, st); CK(launch_rows(rp, true, overlap && behind, st)); }
                g_launches += 1;
                continue;
            }
        }
        FusedParams fp = out;
        fp.T = h->T; fp.G = Gf;
        fp.n_mtiles = pl.n_mtiles; fp.n_ptiles = pl.n_ptiles; fp.passes_per_tile = pl.passes_per_tile;
        fp.table0 = t0; fp.n_tables_launch = nt;
        // part_time doubles as the "segmented minima come from the sweep kernel" switch
        fp.part_time = pl.inline_sweep ? nullptr : part_time;
        fp.part_idx = part_idx;
        fp.pair_base = pl.inline_sweep ? nullptr : reinterpret_cast<const int32_t *>(pl.d_grid + pl.off_pair_base);
        fp.n_pairs = pl.n_pairs; fp.n_seg = pl.n_seg;
        { LaunchTimer lt(h, PLOGP_KERNEL_FUSED, st); CK(launch_fused(fp, predict, overlap && behind, st)); }
        g_launches += 1;
    }
    return PLOGP_OK;
}

}  // namespace

extern "C" {

// Checks host tables; on success packs them as [latency][gap][sizes] for one copy to the device.
static int check_tables(int n_tables, int n_bp, const uint64_t *sizes_bytes, int sizes_shared, const double *gap, const double *latency,
                        std::vector<unsigned char> &pack, bool *monotone)
{
    const double most = std::numeric_limits<double>::max();
    bool falls = false;
    for (int t = 0; t < n_tables; ++t) {
        const uint64_t *sz = sizes_bytes + (sizes_shared ? 0 : size_t(t) * n_bp);
        const double *gp = gap + size_t(t) * n_bp;
        if (!(latency[t] >= 0.0 && latency[t] <= most)) return PLOGP_E_INVAL;
        // all values first, without a branch per value; which error it is, only where there is one
        unsigned bad = 0, down = 0;
        for (int i = 0; i < n_bp; ++i) bad |= unsigned(!(gp[i] >= 0.0)) | unsigned(!(gp[i] <= most));
        for (int i = 1; i < n_bp; ++i) down |= unsigned(gp[i] < gp[i - 1]);
        if (t == 0 || !sizes_shared) {
            for (int i = 1; i < n_bp; ++i) bad |= unsigned(sz[i] <= sz[i - 1]);
            bad |= unsigned(double(sz[n_bp - 1]) >= kTwo53);
        }
        if (bad)
            for (int i = 0; i < n_bp; ++i) {
                if (!std::isfinite(gp[i]) || gp[i] < 0.0) return PLOGP_E_INVAL;
                if (i && sz[i] <= sz[i - 1]) return PLOGP_E_INVAL;
                if (double(sz[i]) >= kTwo53) return PLOGP_E_RANGE;
            }
        // Above the last size the last interval's line is continued: a falling line would turn g negative for
        // large arguments, and the kernels' lower bounds and comparisons rely on times that are not.
        if (gp[n_bp - 1] < gp[n_bp - 2]) return PLOGP_E_RANGE;
        falls |= down != 0;
    }
    *monotone = !falls;
    const size_t lat = size_t(n_tables) * 8, gaps = size_t(n_tables) * n_bp * 8, sizes = (sizes_shared ? size_t(1) : size_t(n_tables)) * n_bp * 8;
    try {
        pack.resize(lat + gaps + sizes);
    } catch (const std::exception &) { return PLOGP_E_NOMEM; }
    std::memcpy(pack.data(), latency, lat);
    std::memcpy(pack.data() + lat, gap, gaps);
    std::memcpy(pack.data() + lat + gaps, sizes_bytes, sizes);
    return PLOGP_OK;
}

// Enqueues the packed tables' copy and their layout.
static int upload_tables(plogp_tables *h, int sizes_shared, cudaStream_t st)
{
    // pageable source: the runtime stages it before returning
    CK(cudaMemcpyAsync(h->d_raw, h->pack.data(), h->pack.size(), cudaMemcpyHostToDevice, st));
    LayoutParams lp{};
    lp.gap = reinterpret_cast<const double *>(h->d_raw) + h->T.n_tables;
    lp.sizes = reinterpret_cast<const uint64_t *>(lp.gap + size_t(h->T.n_tables) * h->T.n_bp);
    lp.tab = h->d_tab;
    lp.n_tables = h->T.n_tables; lp.n_bp = h->T.n_bp; lp.npad = h->T.npad; lp.sizes_shared = sizes_shared;
    CK(launch_layout(lp, st));
    g_launches += 1;
    return PLOGP_OK;
}

int plogp_table_load(int n_tables, int n_bp, const uint64_t *sizes_bytes, int sizes_shared,
                     const double *gap, const double *latency, plogp_tables **out)
{
    if (!sizes_bytes || !gap || !latency || !out) return PLOGP_E_INVAL;
    if (n_tables < 1 || n_bp < 2) return PLOGP_E_INVAL;
    if (n_bp > PLOGP_MAX_BREAKPOINTS) return PLOGP_E_RANGE;
    int npad = 2;
    while (npad < n_bp) npad <<= 1;  // >= n_bp: at least one +inf key follows the last interval

    std::vector<unsigned char> pack;
    bool monotone = false;
    const int brc = check_tables(n_tables, n_bp, sizes_bytes, sizes_shared, gap, latency, pack, &monotone);
    if (brc != PLOGP_OK) return brc;

    plogp_tables *h = new (std::nothrow) plogp_tables();
    if (!h) return PLOGP_E_NOMEM;
    auto fail = [&](int rc) { plogp_table_free(h); return rc; };
    cudaError_t e;
    if ((e = cudaGetDevice(&h->device)) != cudaSuccess) return fail(cuda_fail(e, "cudaGetDevice"));
    if ((e = cudaDeviceGetAttribute(&h->sm_count, cudaDevAttrMultiProcessorCount, h->device)) != cudaSuccess)
        return fail(cuda_fail(e, "cudaDeviceGetAttribute"));
    // one allocation: the kernels' layout, then room for the caller's arrays [latency][gap][sizes per table]
    const size_t tab = size_t(n_tables) * 3 * npad * sizeof(double), raw = size_t(n_tables) * (1 + 2 * size_t(n_bp)) * 8;
    if ((e = cudaMalloc(&h->d_tab, tab + raw)) != cudaSuccess)
        return fail(e == cudaErrorMemoryAllocation ? (cudaGetLastError(), PLOGP_E_NOMEM) : cuda_fail(e, "cudaMalloc(tables)"));
    h->d_raw = reinterpret_cast<unsigned char *>(h->d_tab) + tab;
    h->pack.swap(pack);
    h->T.tab = h->d_tab;
    h->T.lat = reinterpret_cast<const double *>(h->d_raw);
    h->T.n_tables = n_tables;
    h->T.n_bp = n_bp;
    h->T.npad = npad;
    h->monotone = monotone;
    const int urc = upload_tables(h, sizes_shared, nullptr);
    if (urc != PLOGP_OK) return fail(urc);
    if ((e = cudaStreamSynchronize(nullptr)) != cudaSuccess) return fail(cuda_fail(e, "cudaStreamSynchronize(tables)"));
    *out = h;
    return PLOGP_OK;
}

int plogp_table_update(plogp_tables *h, const uint64_t *sizes_bytes, int sizes_shared, const double *gap,
                       const double *latency, void *stream)
{
    if (!h || !sizes_bytes || !gap || !latency) return PLOGP_E_INVAL;
    int dev = 0;
    CK(cudaGetDevice(&dev));
    if (dev != h->device) return PLOGP_E_INVAL;
    bool monotone = false;
    const int brc = check_tables(h->T.n_tables, h->T.n_bp, sizes_bytes, sizes_shared, gap, latency, h->pack, &monotone);
    if (brc != PLOGP_OK) return brc;  // the tables on the device are untouched
    h->monotone = monotone;
    return upload_tables(h, sizes_shared, static_cast<cudaStream_t>(stream));
}

int plogp_table_free(plogp_tables *h)
{
    if (!h) return PLOGP_OK;
    int rc = PLOGP_OK;
    for (int i = 0; i < 2; ++i) {
        if (h->ev_done[i]) cudaEventDestroy(h->ev_done[i]);
        if (h->ev_copied[i]) cudaEventDestroy(h->ev_copied[i]);
    }
    if (h->copy_stream) cudaStreamDestroy(h->copy_stream);
    auto release = [&](void *b) {
        const cudaError_t e = b ? cudaFree(b) : cudaSuccess;
        if (e != cudaSuccess) rc = cuda_fail(e, "cudaFree");
    };
    for (void *b : {static_cast<void *>(h->d_tab), static_cast<void *>(h->d_ws), static_cast<void *>(h->d_stage[0]), static_cast<void *>(h->d_stage[1])}) release(b);
    for (const Plan &c : h->plans) release(c.d_grid);
    for (auto &t : h->timed) { cudaEventDestroy(t.a); cudaEventDestroy(t.b); }
    delete h;
    return rc;
}

int plogp_profile_enable(plogp_tables *h, int enable)
{
    if (!h) return PLOGP_E_INVAL;
    h->profiling = enable != 0;
    return PLOGP_OK;
}

int plogp_profile_read(plogp_tables *h, double *ms, int32_t *launches)
{
    if (!h || !ms || !launches) return PLOGP_E_INVAL;
    for (int k = 0; k < PLOGP_N_KERNEL_KINDS; ++k) { ms[k] = 0.0; launches[k] = 0; }
    int rc = PLOGP_OK;
    for (auto &t : h->timed) {
        float v = 0.f;
        cudaError_t e = cudaEventSynchronize(t.b);
        if (e == cudaSuccess) e = cudaEventElapsedTime(&v, t.a, t.b);
        if (e == cudaSuccess) { ms[t.kind] += v; launches[t.kind] += 1; }
        else rc = cuda_fail(e, "cudaEventElapsedTime");
        cudaEventDestroy(t.a);
        cudaEventDestroy(t.b);
    }
    h->timed.clear();
    return rc;
}

int plogp_predict(plogp_tables *tables, const plogp_grid *grid, double *d_time, uint32_t *d_best_s, void *stream)
{
    if (!tables || !grid || !d_time) return PLOGP_E_INVAL;
    FusedParams out{};
    out.om = default_out_map();
    out.p_time = d_time;
    out.p_best_s = d_best_s;
    return run(tables, grid, true, out, static_cast<cudaStream_t>(stream));
}

int plogp_select_best(plogp_tables *tables, const plogp_grid *grid, uint8_t *d_strategy, uint32_t *d_s_bytes,
                      double *d_time, void *stream)
{
    if (!tables || !grid || !d_strategy || !d_s_bytes || !d_time) return PLOGP_E_INVAL;
    FusedParams out{};
    out.om = default_out_map();
    out.d_strategy = d_strategy;
    out.d_sbytes = d_s_bytes;
    out.d_time = d_time;
    return run(tables, grid, false, out, static_cast<cudaStream_t>(stream));
}

int plogp_select_best_host(plogp_tables *h, const plogp_grid *grid, uint8_t *h_strategy, uint32_t *h_s_bytes,
                           double *h_time, void *stream)
{
    if (!h || !grid || !h_strategy || !h_s_bytes || !h_time) return PLOGP_E_INVAL;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    int dev = 0;
    CK(cudaGetDevice(&dev));
    if (dev != h->device) return PLOGP_E_INVAL;
    const Plan *plan = nullptr;
    int rc = prepare(h, grid, st, &plan);
    if (rc != PLOGP_OK) return rc;
    if (plan->empty) return PLOGP_OK;
    const size_t cells = size_t(2) * plan->G.n_P * plan->G.n_m;  // per table
    const size_t per_table = cells * 13 + 3 * 256;
    // Tables per staging set: at most 512 MiB, at least one table.  The first set is an eighth of the whole (4 MiB or more),
    // so that the first copy starts early and its kernels are all that the copies do not hide.
    const int batch = int(std::min<size_t>(h->T.n_tables, std::max<size_t>(1, (size_t(512) << 20) / per_table)));
    const int first = int(std::min<size_t>(batch, std::max<size_t>((h->T.n_tables + 7) / 8, (size_t(4) << 20) / per_table + 1)));
    const size_t need = per_table * batch;
    if (need > h->stage_cap) {
        for (int i = 0; i < 2; ++i) {
            if (h->d_stage[i]) CK(cudaFree(h->d_stage[i]));
            h->d_stage[i] = nullptr;
        }
        h->stage_cap = 0;
        for (int i = 0; i < 2; ++i) {
            cudaError_t e = cudaMalloc(&h->d_stage[i], need);
            if (e == cudaErrorMemoryAllocation) { cudaGetLastError(); return PLOGP_E_NOMEM; }
            if (e != cudaSuccess) return cuda_fail(e, "cudaMalloc(staging)");
        }
        h->stage_cap = need;
    }
    if (!h->copy_stream) {
        CK(cudaStreamCreateWithFlags(&h->copy_stream, cudaStreamNonBlocking));
        for (int i = 0; i < 2; ++i) {
            CK(cudaEventCreateWithFlags(&h->ev_done[i], cudaEventDisableTiming));
            CK(cudaEventCreateWithFlags(&h->ev_copied[i], cudaEventDisableTiming));
        }
    }
    auto align = [](size_t x) { return (x + 255) / 256 * 256; };
    int slot = 0;
    for (int t0 = 0, nt; t0 < h->T.n_tables; t0 += nt, slot ^= 1) {
        nt = std::min(t0 == 0 ? first : batch, h->T.n_tables - t0);
        // layout of a staging set: time | segment size | strategy, each for nt tables
        double *s_time = reinterpret_cast<double *>(h->d_stage[slot]);
        uint32_t *s_sb = reinterpret_cast<uint32_t *>(h->d_stage[slot] + align(cells * 8 * batch));
        uint8_t *s_id = h->d_stage[slot] + align(cells * 8 * batch) + align(cells * 4 * batch);
        if (t0 >= first + batch) {  // the set's previous copy has left
            cudaError_t ew = cudaStreamWaitEvent(st, h->ev_copied[slot], 0);
            if (ew != cudaSuccess) { rc = cuda_fail(ew, "cudaStreamWaitEvent"); break; }
        }
        FusedParams out{};
        out.om = default_out_map();
        out.d_time = s_time;
        out.d_sbytes = s_sb;
        out.d_strategy = s_id;
        out.out_table0 = t0;  // the staging set holds tables t0 .. t0 + nt - 1
        rc = run(h, grid, false, out, st, t0, t0 + nt);
        // On any failure the loop ends here, and both streams are drained below before the call returns: no
        // copy into the caller's arrays is left in flight.
        cudaError_t e = cudaSuccess;
        if (rc == PLOGP_OK) e = cudaEventRecord(h->ev_done[slot], st);
        if (rc == PLOGP_OK && e == cudaSuccess) e = cudaStreamWaitEvent(h->copy_stream, h->ev_done[slot], 0);
        if (rc == PLOGP_OK && e == cudaSuccess)
            e = cudaMemcpyAsync(h_time + size_t(t0) * cells, s_time, cells * 8 * nt, cudaMemcpyDeviceToHost, h->copy_stream);
        if (rc == PLOGP_OK && e == cudaSuccess)
            e = cudaMemcpyAsync(h_s_bytes + size_t(t0) * cells, s_sb, cells * 4 * nt, cudaMemcpyDeviceToHost, h->copy_stream);
        if (rc == PLOGP_OK && e == cudaSuccess)
            e = cudaMemcpyAsync(h_strategy + size_t(t0) * cells, s_id, cells * nt, cudaMemcpyDeviceToHost, h->copy_stream);
        if (rc == PLOGP_OK && e == cudaSuccess) e = cudaEventRecord(h->ev_copied[slot], h->copy_stream);
        if (rc == PLOGP_OK && e != cudaSuccess) rc = cuda_fail(e, "plogp_select_best_host: copy pipeline");
        if (rc != PLOGP_OK) break;
    }
    cudaError_t e1 = cudaStreamSynchronize(h->copy_stream), e2 = cudaStreamSynchronize(st);
    if (rc != PLOGP_OK) { cudaGetLastError(); return rc; }
    if (e1 != cudaSuccess) return cuda_fail(e1, "cudaStreamSynchronize(copy)");
    if (e2 != cudaSuccess) return cuda_fail(e2, "cudaStreamSynchronize");
    return PLOGP_OK;
}

int plogp_select_best_collective(plogp_tables *h, const plogp_grid *grid, int collective, uint8_t *d_strategy,
                                 uint32_t *d_s_bytes, double *d_time, void *stream)
{
    if (!h || !grid || !d_strategy || !d_s_bytes || !d_time) return PLOGP_E_INVAL;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    plogp_grid g = *grid;
    FusedParams out{};
    out.om = default_out_map();
    out.om.planes = 1; out.om.plane_bcast = 0; out.om.plane_scat = 0;
    out.d_strategy = d_strategy; out.d_sbytes = d_s_bytes; out.d_time = d_time;
    switch (collective) {
    case PLOGP_GATHER:  // the Scatter strategies run backwards: ids 10, 11, 12 -> 13, 14, 15
        g.strategy_mask &= 0x1C00u;
        for (int i = 10; i <= 12; ++i) out.om.id_of[i] = uint8_t(i + 3);
        return run(h, &g, false, out, st);
    case PLOGP_REDUCE: {  // the Broadcast strategies without a handshake run backwards: 0 2 3 5 6 7 9 -> 16 .. 22
        g.strategy_mask &= 0x2EDu;
        static const int from[7] = {0, 2, 3, 5, 6, 7, 9};
        for (int i = 0; i < 7; ++i) out.om.id_of[from[i]] = uint8_t(16 + i);
        return run(h, &g, false, out, st);
    }
    case PLOGP_BARRIER: {  // one decision per (table, P); the message sizes play no part
        g.strategy_mask &= 0xC9u;
        int dev = 0;
        CK(cudaGetDevice(&dev));
        if (dev != h->device) return PLOGP_E_INVAL;
        const Plan *plan = nullptr;
        const int rc = prepare(h, &g, st, &plan);
        if (rc != PLOGP_OK) return rc;
        if (plan->empty) return PLOGP_OK;  // no process count, no message size to carry the plan, or no strategy
        CK(launch_barrier(h->T, plan->G, 0, h->T.n_tables, d_strategy, d_s_bytes, d_time, st));
        g_launches += 1;
        return PLOGP_OK;
    }
    default:
        return PLOGP_E_INVAL;
    }
}

int plogp_segment_surface(plogp_tables *h, const plogp_grid *grid, double *d_surface, void *stream)
{
    if (!h || !grid || !d_surface) return PLOGP_E_INVAL;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    int dev = 0;
    CK(cudaGetDevice(&dev));
    if (dev != h->device) return PLOGP_E_INVAL;
    const Plan *plan = nullptr;
    const int rc = prepare(h, grid, st, &plan);
    if (rc != PLOGP_OK) return rc;
    const Plan &pl = *plan;
    if (pl.empty || pl.n_seg == 0 || pl.G.n_s == 0) return PLOGP_OK;
    // up to four message sizes per warp, while that leaves eight CTAs per SM
    int surf_m = 32;
    while (surf_m > 8 && (long long)((pl.G.n_m + surf_m - 1) / surf_m) * ((pl.G.n_P + 7) / 8) * h->T.n_tables < (long long)h->sm_count * 8) surf_m >>= 1;
    for (int t0 = 0; t0 < h->T.n_tables; t0 += 65535) {
        SensParams sp{};
        sp.T = h->T; sp.G = pl.G;
        sp.table0 = t0; sp.n_tables_launch = std::min(65535, h->T.n_tables - t0); sp.out_table0 = 0;
        sp.surface = d_surface; sp.surf_m = surf_m;
        CK(launch_surface(sp, st));
        g_launches += 1;
    }
    return PLOGP_OK;
}

int plogp_segment_sensitivity(plogp_tables *h, const plogp_grid *grid, uint64_t s_fixed, const double *d_pred_time,
                              double *d_time_fixed, double *d_ratio, void *stream)
{
    if (!h || !grid || !d_time_fixed) return PLOGP_E_INVAL;
    if ((d_ratio == nullptr) != (d_pred_time == nullptr)) return PLOGP_E_INVAL;
    if (s_fixed == 0 || grid->dtype_bytes == 0 || s_fixed % grid->dtype_bytes) return PLOGP_E_INVAL;
    if (s_fixed >= kTwo32) return PLOGP_E_RANGE;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    int dev = 0;
    CK(cudaGetDevice(&dev));
    if (dev != h->device) return PLOGP_E_INVAL;
    const Plan *plan = nullptr;
    const int rc = prepare(h, grid, st, &plan);
    if (rc != PLOGP_OK) return rc;
    const Plan &pl = *plan;
    if (pl.empty || pl.n_seg == 0) return PLOGP_OK;
    // enough CTAs to fill the GPU, each with a run of process counts per warp
    const bool aligned = (reinterpret_cast<uintptr_t>(d_pred_time) | reinterpret_cast<uintptr_t>(d_time_fixed) | reinterpret_cast<uintptr_t>(d_ratio)) % 16 == 0;
    const int vec = pl.G.n_m % 2 == 0 && aligned && (pl.G.n_m + 63) / 64 * 2 == (pl.G.n_m + 31) / 32 ? 2 : 1;
    const long long base_blocks = (long long)((pl.G.n_m + 32 * vec - 1) / (32 * vec)) * h->T.n_tables;
    int p_per_cta = pl.G.n_P;
    while (p_per_cta > 8 && base_blocks * ((pl.G.n_P + p_per_cta - 1) / p_per_cta) < (long long)h->sm_count * 8) p_per_cta = (p_per_cta + 1) / 2;
    for (int t0 = 0; t0 < h->T.n_tables; t0 += 65535) {
        SensParams sp{};
        sp.T = h->T; sp.G = pl.G;
        sp.table0 = t0; sp.n_tables_launch = std::min(65535, h->T.n_tables - t0); sp.out_table0 = 0;
        sp.s_fixed = uint32_t(s_fixed); sp.p_per_cta = p_per_cta; sp.vec = vec;
        sp.pred_time = d_pred_time; sp.time_fixed = d_time_fixed; sp.ratio = d_ratio;
        CK(launch_fixed(sp, st));
        g_launches += 1;
    }
    return PLOGP_OK;
}

int plogp_decision_boundaries(int n_tables, int n_P, int n_m, const uint8_t *d_strategy, uint8_t *d_boundary, void *stream)
{
    if (n_tables < 0 || n_P < 0 || n_m < 0) return PLOGP_E_INVAL;
    if (n_tables == 0 || n_P == 0 || n_m == 0) return PLOGP_OK;
    if (!d_strategy || !d_boundary) return PLOGP_E_INVAL;
    int dev = 0, sms = 0;
    CK(cudaGetDevice(&dev));
    CK(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
    CK(launch_boundaries(d_strategy, d_boundary, 2LL * n_tables, n_P, n_m, sms, static_cast<cudaStream_t>(stream)));
    g_launches += 1;
    return PLOGP_OK;
}

const char *plogp_status_string(int status)
{
    switch (status) {
    case PLOGP_OK: return "ok";
    case PLOGP_E_INVAL: return "invalid argument";
    case PLOGP_E_NOMEM: return "out of memory";
    case PLOGP_E_CUDA: return "CUDA runtime error";
    case PLOGP_E_RANGE: return "value out of the supported range";
    default: return "unknown status";
    }
}

const char *plogp_last_cuda_error(void) { return g_cuda_error.c_str(); }

uint64_t plogp_kernel_launches(void) { return g_launches.load(); }

double plogp_fp64_fma_rate(double milliseconds)
{
    if (!(milliseconds > 0.0)) return double(PLOGP_E_INVAL);
    int dev = 0, sms = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
        return double(PLOGP_E_CUDA);
    double *sink = nullptr;
    cudaEvent_t e0 = nullptr, e1 = nullptr;
    double rate = double(PLOGP_E_CUDA);
    const int blocks = sms * 4;
    const double fma_per_iter = double(blocks) * kThreads * 32.0;
    do {
        if (cudaMalloc(&sink, sizeof(double)) != cudaSuccess) break;
        if (cudaEventCreate(&e0) != cudaSuccess || cudaEventCreate(&e1) != cudaSuccess) break;
        int iters = 2000;
        float ms = 0.f;
        bool ok = true;
        for (int round = 0; round < 3 && ok; ++round) {  // warm-up, calibration, measurement
            ok = cudaEventRecord(e0) == cudaSuccess && launch_fp64_probe(sink, iters, blocks, nullptr) == cudaSuccess &&
                 (g_launches += 1, true) &&
                 cudaEventRecord(e1) == cudaSuccess && cudaEventSynchronize(e1) == cudaSuccess &&
                 cudaEventElapsedTime(&ms, e0, e1) == cudaSuccess;
            if (ok && round == 1 && ms > 0.f) iters = int(std::min(2e8, std::max(2000.0, iters * milliseconds / ms)));
        }
        if (ok && ms > 0.f) rate = fma_per_iter * iters / (ms * 1e-3);
    } while (0);
    if (e0) cudaEventDestroy(e0);
    if (e1) cudaEventDestroy(e1);
    if (sink) cudaFree(sink);
    return rate;
}

}  // extern "C"
