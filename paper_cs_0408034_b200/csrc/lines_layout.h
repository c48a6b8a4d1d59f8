// Shared memory of lines_block (lines.cuh), for the kernel and for the host, which chooses a CTA's message sizes by it.
#pragma once

#include "internal.h"

namespace plogp {

namespace lines {

constexpr int kSegs = kLineSegs, kKnots = kSegs + 1;
constexpr int kBars = kKnots + 3 * kSegs;  // what a line's times are compared with
constexpr int kRows = 8;  // process counts per thread and step

struct __align__(16) Row {  // a process count
    double x;  // P - 1
    int pair;  // first entry of its (floor, ceil) pair in the pairs' arrays
    int unused;
};

struct Smem {
    double *tab, *gs;
    double *k;         // [n_s][width]: Section 2's k
    int *knot;         // [kKnots + 1]: indices of the knots, then the number of segments
    Row *row;          // [n_p]
    double *pair_t;    // [n_pairs][width]: smallest time of ids 6 to 9
    uint32_t *pair_s;  // the same: segment size, id
    uint8_t *pair_id;
    unsigned *key;     // [groups][kKnots + 1][width] and behind them
    unsigned *bar;     // [kBars][width]; both in the place of the pairs, which come later
    uint32_t *live;    // [kSegs][2][width]: candidates of id 5 that can win in a segment, a bit each
    uint32_t *near;    // [2][width]: candidates of ids 2 and 9 beside the best one
    uint8_t *flat;     // [kSegs][width]: the same for the flat tree (1), id 2's best candidate (2) and the chain (4)
    uint32_t *sval;    // [n_s]
    double *out_t;     // STAGED: a step's cells, [groups * kRows][width] and room for a shift of up to three cells
    uint32_t *out_s;
    uint8_t *out_id;
};

__host__ __device__ inline size_t layout(int npad, int n_s, int n_pairs, int n_p, int width, int threads, int staged, unsigned char *base, Smem *o)
{
    const int nsv = n_s > 0 ? n_s : 1, groups = threads / width;
    size_t off = 0;
    auto take = [&](size_t bytes) { size_t at = off; off += (bytes + 15) & ~size_t(15); return at; };
    const size_t o_tab = take(3 * size_t(npad) * 8), o_gs = take(size_t(nsv) * 8), o_k = take(size_t(nsv) * width * 8), o_knot = take((kKnots + 1) * 4), o_row = take(size_t(n_p) * sizeof(Row)),
                 o_live = take(size_t(kSegs) * 2 * width * 4), o_near = take(size_t(2) * width * 4), o_flat = take(size_t(kSegs) * width), o_sv = take(size_t(nsv) * 4);
    const size_t o_key = off;
    const size_t o_pt = take(size_t(n_pairs) * width * 8), o_ps = take(size_t(n_pairs) * width * 4), o_pi = take(size_t(n_pairs) * width);
    const size_t keys = size_t(groups) * (kKnots + 1) * width * 4, bars = size_t(kBars) * width * 4;
    if (off < o_key + keys + bars) off = o_key + keys + bars;
    const size_t cells = staged ? size_t(groups) * kRows * width + 4 : 0;
    off = (off + 31) & ~size_t(31);
    const size_t o_t = take(cells * 8), o_s = take(cells * 4), o_id = take(cells);
    if (o) {
        o->out_t = reinterpret_cast<double *>(base + o_t); o->out_s = reinterpret_cast<uint32_t *>(base + o_s); o->out_id = base + o_id;
        o->tab = reinterpret_cast<double *>(base + o_tab); o->gs = reinterpret_cast<double *>(base + o_gs);
        o->k = reinterpret_cast<double *>(base + o_k); o->knot = reinterpret_cast<int *>(base + o_knot); o->row = reinterpret_cast<Row *>(base + o_row);
        o->pair_t = reinterpret_cast<double *>(base + o_pt); o->pair_s = reinterpret_cast<uint32_t *>(base + o_ps); o->pair_id = base + o_pi;
        o->key = reinterpret_cast<unsigned *>(base + o_key); o->bar = reinterpret_cast<unsigned *>(base + o_key + keys); o->live = reinterpret_cast<uint32_t *>(base + o_live);
        o->near = reinterpret_cast<uint32_t *>(base + o_near); o->flat = base + o_flat; o->sval = reinterpret_cast<uint32_t *>(base + o_sv);
    }
    return off;
}

}  // namespace lines

inline size_t lines_smem_bytes(const LinesParams &p)
{
    if (p.direct) return (3 * static_cast<size_t>(p.T.npad) + 3 * static_cast<size_t>(p.G.n_s)) * sizeof(double);
    return lines::layout(p.gaps ? 0 : p.T.npad, p.G.n_s, p.n_pairs, p.n_p, p.width, p.threads, p.staged, nullptr, nullptr);
}

}  // namespace plogp
