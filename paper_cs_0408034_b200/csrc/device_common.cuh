// Device helpers shared by the kernels: table staging into shared memory, g(x), grid accessors.
#pragma once

#include "internal.h"

#include <math_constants.h>

namespace plogp {

// ------------------------------------------------------------------------------------------
// Overlap of the kernels of one call
// ------------------------------------------------------------------------------------------
//
// The first kernel of a call is launched as usual; the ones behind it may start once every CTA of the kernel in front
// has called dependents_may_start.  A kernel that reads what the one in front writes waits for its end first.  Each kernel's
// last CTA waits for the end of the kernel in front before it ends itself, so that the end of a call's last kernel is the
// end of the call.  Nothing here spins: the waits are the hardware's, and a kernel's CTAs only start when all CTAs of the
// kernel in front have their place.  A kernel launched with `overlap` must therefore not end thread 0 of its last CTA anywhere but
// behind last_block_waits; envelope_kernel, which returns early, is only ever the first of a call.
__device__ __forceinline__ void dependents_may_start() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void wait_for_kernel_in_front() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void last_block_waits(int tid)  // call at the end; thread 0 of a kernel's last CTA must get here
{
    if (tid == 0 && blockIdx.x == gridDim.x - 1 && blockIdx.y == gridDim.y - 1) wait_for_kernel_in_front();
}

// ------------------------------------------------------------------------------------------
// Table staging and g(x)
// ------------------------------------------------------------------------------------------

__device__ __forceinline__ void cp_async16(void *smem_dst, const void *gmem_src)
{
    unsigned s = static_cast<unsigned>(__cvta_generic_to_shared(smem_dst));
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(s), "l"(gmem_src));
}

__device__ __forceinline__ void cp_async_wait_all()
{
    asm volatile("cp.async.commit_group;\n" ::: "memory");
    asm volatile("cp.async.wait_group 0;\n" ::: "memory");
}

// Copies one table (key | gap | slope, 3*npad doubles) into shared memory with 16-byte
// asynchronous copies.  The caller synchronises the CTA afterwards.
__device__ __forceinline__ void stage_table(double *s_tab, const TableDev &T, int table)
{
    const double *src = T.tab + static_cast<size_t>(table) * 3 * T.npad;
    const int n16 = (3 * T.npad) >> 1;
    for (int i = threadIdx.x; i < n16; i += blockDim.x) cp_async16(s_tab + 2 * i, src + 2 * i);
    cp_async_wait_all();
}

// g(x) of Section 2 on the staged table: branch-free search of the interval that starts at or
// below x (keys beyond the last interval are +inf), then one fused multiply-add along that
// interval's line.  x below the first size is held at the first gap (dx clamped to 0); x above
// the last size continues the last interval's line.
__device__ __forceinline__ double gap_at(const double *s_tab, int npad, double x)
{
    int i = 0;
#pragma unroll 1
    for (int step = npad >> 1; step > 0; step >>= 1) {
        const int j = i + step;
        i = (s_tab[j] <= x) ? j : i;
    }
    const double dx = fmax(x - s_tab[i], 0.0);
    return fma(dx, s_tab[2 * npad + i], s_tab[npad + i]);
}

// g(1): sizes are whole numbers, so 1 lies below the table or in one of its first two intervals
__device__ __forceinline__ double gap_at_one(const double *s_tab, int npad)
{
    const int i = s_tab[1] <= 1.0 ? 1 : 0;
    return fma(fmax(1.0 - s_tab[i], 0.0), s_tab[2 * npad + i], s_tab[npad + i]);
}

__device__ __forceinline__ int P_at(const GridDev &G, int pidx)
{
    return G.P_list ? G.P_list[pidx] : G.P_lo + pidx;
}

__device__ __forceinline__ uint32_t s_at(const GridDev &G, int si)
{
    return G.s_list ? G.s_list[si] : G.s_lo + static_cast<uint32_t>(si) * G.s_step;
}

// (floor, ceil) of log2 P as one number that grows with P: 2 floor + (P is no power of two)
__device__ __forceinline__ int pair_of(int P) { return 2 * (31 - __clz(P)) + ((P & (P - 1)) != 0 ? 1 : 0); }

// k of Section 2: number of segments of size s in a message of m bytes.
__device__ __forceinline__ uint32_t segments(uint32_t m, uint32_t s, int k_mode)
{
    const uint32_t q = m / s;
    return q + ((k_mode == 0 && q * s != m) ? 1u : 0u);
}

// Lower bounds in FP32: two fused multiply-adds at a time, rounded towards minus infinity.  With operands that are
// rounded down themselves and non-negative, a result is never above the FP64 value of the same expression.
using f32x2 = unsigned long long;
struct __align__(16) f32x2x2 { f32x2 x, y; };
__device__ __forceinline__ f32x2 splat2(float a)
{
    f32x2 r;
    asm("mov.b64 %0, {%1, %1};" : "=l"(r) : "f"(a));
    return r;
}
__device__ __forceinline__ f32x2 fma2_down(f32x2 a, f32x2 b, f32x2 c)
{
    f32x2 r;
    asm("fma.rm.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
    return r;
}
// the smallest of a and the two values of t (one three-input minimum)
__device__ __forceinline__ float min_with2(float a, f32x2 t)
{
    float r;
    asm("{.reg .f32 lo, hi;\n\tmov.b64 {lo, hi}, %2;\n\tmin.f32 %0, %1, lo, hi;}" : "=f"(r) : "f"(a), "l"(t));
    return r;
}

// Four doubles from shared to global memory, both 32-byte aligned
__device__ __forceinline__ void store4(double *out, const double *s)
{
    const double2 a = *reinterpret_cast<const double2 *>(s), b = *reinterpret_cast<const double2 *>(s + 2);
    asm volatile("st.global.v4.f64 [%0], {%1, %2, %3, %4};" ::"l"(out), "d"(a.x), "d"(a.y), "d"(b.x), "d"(b.y) : "memory");
}

// Interval search alone: largest i with key[i] <= x (0 when x is below the table).
__device__ __forceinline__ int interval_of(const double *s_tab, int npad, double x)
{
    int i = 0;
#pragma unroll 1
    for (int step = npad >> 1; step > 0; step >>= 1) {
        const int j = i + step;
        i = (s_tab[j] <= x) ? j : i;
    }
    return i;
}

// x rounded to a whole number, for 0 <= x < 2^51 (two additions; the rounding instruction has a quarter of their rate).
// Of the two whole numbers around a quotient's true value the caller takes the right one by the sign of the remainder:
// a product with the reciprocal is off by far less than one half, as j m < 2^53 and j <= 2^30.
__device__ __forceinline__ double round_whole(double x)
{
    const double big = 6755399441055744.0;  // 1.5 * 2^52
    return (x + big) - big;
}

// g(x) for a caller whose arguments never decrease (the Scatter Chain's j m): the current interval's line is kept in
// registers and shared memory is touched only when x crosses into the next interval (keys past the last interval are
// +inf, and npad >= n_bp leaves at least one such key, so the walk stops inside the array).  Below the table a
// pseudo-interval with slope 0 holds g at its first value.
struct ChainWalk {
    int i;
    double key, next, slope, gap;

    __device__ __forceinline__ void start(const double *s_tab, int npad, double x)
    {
        if (x < s_tab[0]) {
            i = -1; key = 0.0; next = s_tab[0]; slope = 0.0; gap = s_tab[npad];
        } else {
            i = interval_of(s_tab, npad, x);
            load(s_tab, npad);
        }
    }
    __device__ __forceinline__ void load(const double *s_tab, int npad)
    {
        key = s_tab[i]; next = s_tab[i + 1]; slope = s_tab[2 * npad + i]; gap = s_tab[npad + i];
    }
    __device__ __forceinline__ void advance(const double *s_tab, int npad, double x)
    {
        while (x >= next) {
            // rare: keep it a branch (the barrier stops the compiler from turning the reload into
            // loads and selects that would run at every step)
            asm volatile("" ::: "memory");
            ++i;
            load(s_tab, npad);
        }
    }
    __device__ __forceinline__ double at(const double *s_tab, int npad, double x)
    {
        advance(s_tab, npad, x);
        return fma(x - key, slope, gap);
    }
    // Sum of g(j m) for j = j0 .. j1 (whole numbers, j0 <= j1) in closed form: inside one interval g is a line, so its
    // terms are an arithmetic series, n times g at their mean argument.  The loop runs over the intervals that the
    // arguments cross (at most n_bp), not over j.
    __device__ __forceinline__ double range(const double *s_tab, int npad, double md, double j0, double j1)
    {
        const double x1 = j1 * md;
        double sum = 0.0;
        advance(s_tab, npad, j0 * md);
        if (x1 >= next) {
            const double inv_m = 1.0 / md;
            do {
                // last j of the interval: the largest with j m < next (next <= x1 < 2^53: the products are exact)
                double q = round_whole(next * inv_m);
                if (fma(-q, md, next) <= 0.0) q -= 1.0;
                sum = fma(q - j0 + 1.0, fma(0.5 * ((j0 + q) * md) - key, slope, gap), sum);
                j0 = q + 1.0;
                advance(s_tab, npad, j0 * md);
            } while (x1 >= next);
        }
        return fma(j1 - j0 + 1.0, fma(0.5 * ((j0 + j1) * md) - key, slope, gap), sum);
    }
};

// Scatter Chain sum in front of each warp's run of process counts, for one message size per lane.  A CTA's n_warps warps
// own the runs [e0, e1) of process-count indices, one after another from index c0 on.  The terms j <= P(c0) - 2, which
// lie in front of the whole CTA, are split over its warps by table intervals (front); each warp adds the closed form of
// its own run (own), which the warps behind it need.  A handful of intervals per warp instead of a pass over the process
// counts, and nothing is carried between CTAs.  The caller puts a barrier between the two calls.
static __device__ __noinline__ void chain_front_parts(const double *s_tab, int npad, int n_bp, const int32_t *P_list, int P_lo, double md, int c0, int e0,
                                                      int e1, int warp, int n_warps, double *s_front, double *s_own, int stride)
{
    auto P_of = [&](int e) { return P_list ? P_list[e] : P_lo + e; };
    double front = 0.0, own = 0.0;
    if (c0 < e1) {  // the CTA has process counts (a warp without any still takes its share of the front)
        const int P0 = P_of(c0);
        const double jc = static_cast<double>(P0 - 2);
        ChainWalk w;
        if (jc >= 1.0) {
            const double inv_m = 1.0 / md, x_end = jc * md;
            const int n_int = n_bp - 1, i0 = n_int * warp / n_warps, i1 = n_int * (warp + 1) / n_warps;
            auto first_j = [&](int i) {  // smallest j with j m >= key i; jc + 1 when that lies behind jc
                const double key = s_tab[i];
                const double q = round_whole(key * inv_m), j = fmax(fma(-q, md, key) > 0.0 ? q + 1.0 : q, 1.0);
                return key > x_end ? jc + 1.0 : j;
            };
            double ja = first_j(i0);
            if (warp == 0) front = (ja - 1.0) * s_tab[npad];  // below the table
            // no branch depends on the lane, and the intervals do not wait for one another
#pragma unroll 4
            for (int i = i0; i < i1; ++i) {
                const double jb = i + 1 < n_int ? first_j(i + 1) : jc + 1.0;
                front = fma(jb - ja, fma(0.5 * ((ja + jb - 1.0) * md) - s_tab[i], s_tab[2 * npad + i], s_tab[npad + i]), front);
                ja = jb;
            }
        }
        if (e0 < e1 && warp < n_warps - 1) {
            const double j0 = e0 == c0 ? jc + 1.0 : static_cast<double>(P_of(e0 - 1)), j1 = static_cast<double>(P_of(e1 - 1) - 1);
            w.start(s_tab, npad, j0 * md);
            own = w.range(s_tab, npad, md, j0, j1);
        }
    }
    s_front[warp * stride] = front;
    s_own[warp * stride] = own;
}
__device__ __forceinline__ double chain_front_sum(const double *s_front, const double *s_own, int stride, int warp, int n_warps)
{
    double run = 0.0;
#pragma unroll
    for (int w = 0; w < n_warps; ++w) run += s_front[w * stride];
    for (int w = 0; w < warp; ++w) run += s_own[w * stride];
    return run;
}

// The same sums for listed process counts, from a table per message size (lane) of the CTA: s_ja[i] = the first j whose
// argument j m lies in interval i or behind it, s_before[i] = the sum of g(j m) over all j in front of it.  The sum up to any
// j is then one arithmetic series, whatever the distance to the process count before it.  Built by all warps, each a chunk
// of the intervals; a barrier of the caller's goes between the calls and one behind them.
struct ChainTable {
    double *ja, *before, *tot;  // [n_bp - 1][32], the same, [warps][32]; at the lane's column

    __device__ __forceinline__ void build(const double *s_tab, int npad, int n_bp, double md, double j_max, int warp, int warps) const
    {
        const double inv_m = 1.0 / md, x_max = j_max * md;
        const int n_int = n_bp - 1, i0 = n_int * warp / warps, i1 = n_int * (warp + 1) / warps;
        auto first_j = [&](int i) {  // smallest j with j m >= key i; j_max + 1 when that lies behind j_max
            const double key = s_tab[i];
            const double q = round_whole(key * inv_m), j = fmax(fma(-q, md, key) > 0.0 ? q + 1.0 : q, 1.0);
            return key > x_max ? j_max + 1.0 : j;
        };
        double j = first_j(i0), sum = warp == 0 ? (j - 1.0) * s_tab[npad] : 0.0;  // below the table
#pragma unroll 4
        for (int i = i0; i < i1; ++i) {
            const double jb = i + 1 < n_int ? first_j(i + 1) : j_max + 1.0;
            ja[32 * i] = j;
            before[32 * i] = sum;
            sum = fma(jb - j, fma(0.5 * ((j + jb - 1.0) * md) - s_tab[i], s_tab[2 * npad + i], s_tab[npad + i]), sum);
            j = jb;
        }
        tot[32 * warp] = sum;
    }
    __device__ __forceinline__ void add_up(int n_bp, int warp, int warps) const
    {
        const int n_int = n_bp - 1, i0 = n_int * warp / warps, i1 = n_int * (warp + 1) / warps;
        double front = 0.0;
        for (int w = 0; w < warp; ++w) front += tot[32 * w];
#pragma unroll 4
        for (int i = i0; i < i1; ++i) before[32 * i] += front;
    }
};
struct ChainAt {  // a lane's place in it; arguments never decrease
    int i;
    double key, next, slope, gap, ja, before;

    __device__ __forceinline__ void start(const double *s_tab, int npad, const ChainTable &c, double x)
    {
        if (x < s_tab[0]) {
            i = -1; key = 0.0; next = s_tab[0]; slope = 0.0; gap = s_tab[npad]; ja = 1.0; before = 0.0;
        } else {
            i = interval_of(s_tab, npad, x);
            load(s_tab, npad, c);
        }
    }
    __device__ __forceinline__ void load(const double *s_tab, int npad, const ChainTable &c)
    {
        key = s_tab[i]; next = s_tab[i + 1]; slope = s_tab[2 * npad + i]; gap = s_tab[npad + i];
        ja = c.ja[32 * i]; before = c.before[32 * i];
    }
    __device__ __forceinline__ double sum(const double *s_tab, int npad, const ChainTable &c, double md, double j)
    {
        const double x = j * md;
        if (x >= next) {
            do { ++i; next = s_tab[i + 1]; } while (x >= next);
            load(s_tab, npad, c);
        }
        return fma(j - ja + 1.0, fma(0.5 * ((ja + j) * md) - key, slope, gap), before);
    }
};

// Lexicographic minimum of (t, e) over a warp (all lanes receive it), t >= 0 and e >= 0: three integer warp reductions,
// of the high word, the low word where it ties, and e where both do.
__device__ __forceinline__ void warp_min_pair(double &t, int &e)
{
    const int h = __reduce_min_sync(0xffffffffu, __double2hiint(t));
    const bool on_h = __double2hiint(t) == h;
    const unsigned l = __reduce_min_sync(0xffffffffu, on_h ? static_cast<unsigned>(__double2loint(t)) : 0xffffffffu);
    e = __reduce_min_sync(0xffffffffu, on_h && static_cast<unsigned>(__double2loint(t)) == l ? e : 0x7fffffff);
    t = __hiloint2double(h, static_cast<int>(l));
}
__device__ __forceinline__ double warp_min(double t)  // t >= 0
{
    const int h = __reduce_min_sync(0xffffffffu, __double2hiint(t));
    return __hiloint2double(h, static_cast<int>(__reduce_min_sync(0xffffffffu, __double2hiint(t) == h ? static_cast<unsigned>(__double2loint(t)) : 0xffffffffu)));
}

// The lower envelope of the lines t_e(x) = fma(x, B_e, C_e) of the Segmented Chain, slopes ascending with the candidate e: the
// best line's index does not grow with x.  For the computed, rounded times that holds up to lines that differ by rounding,
// which may be any number of entries apart (a latency far above the gaps makes almost all slopes equal).  With u = 2^-53:
// slopes ascend up to 5 u (g is interpolated), a time is off by u.  An entry below every one whose time at x2 is within
// (1 + e) of the best there loses at all x <= x2 if e > 12 u: its distance does not shrink towards smaller x.  One above
// every such entry at x1 loses at all x in x1 .. r x1 if e > 4 u + 8 u r: its distance does not shrink, the best time grows by r
// at most.  So the winners between x1 and x2 lie between the smallest entry within envelope_near at x2 and the largest within
// envelope_near(x2 / x1) at x1.
__device__ __forceinline__ double envelope_near(double r) { return 0x1p-49 * r; }

}  // namespace plogp
