// Sensitivity of the segmented strategies of Table 1 to the segment size (Section 3.1 searches the size that
// minimises the model; the measured Segmented Chain of the paper's Fig. 1(b) used a fixed 8 kB):
//   surface_kernel   the model of ids 2, 5, 9 for every candidate segment size, [table][3][P][m][s]
//   fixed_kernel     the model with one fixed segment size (the whole message where it does not fit) and its
//                    ratio to the minimum over the candidates that plogp_predict found
//   boundary_kernel  where the selected strategy changes between neighbouring P or neighbouring m
// The three are plain streaming kernels (one model evaluation or one comparison per output element).
#include "device_common.cuh"

#include <algorithm>

namespace plogp {

// One CTA: one table, p.surf_m message sizes (its warps stride over them), kSurfP consecutive process counts; lanes <->
// candidate sizes, so g(s) is computed once per CTA, k and the line coefficients once per (m, s), and every store is a
// run of consecutive s.
constexpr int kSurfP = 8, kSurfW = 8, kSurfS = 32 * kSurfW;

__global__ void __launch_bounds__(kSurfS) surface_kernel(const SensParams p)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    double *s_tab = reinterpret_cast<double *>(smem_raw);
    double *s_gs = s_tab + 3 * p.T.npad;  // [kSurfS]
    const int n_s = p.G.n_s, n_P = p.G.n_P, n_m = p.G.n_m;
    const int n_mg = (n_m + p.surf_m - 1) / p.surf_m;
    const int mgroup = blockIdx.x % n_mg, pchunk = blockIdx.x / n_mg, trel = blockIdx.y;
    const int table = p.table0 + trel;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    stage_table(s_tab, p.T, table);
    __syncthreads();
    const double L = p.T.lat[table];
    const bool on2 = (p.G.mask >> 2) & 1u, on5 = (p.G.mask >> 5) & 1u, on9 = (p.G.mask >> 9) & 1u;
    const int p0 = pchunk * kSurfP, p1 = min(p0 + kSurfP, n_P);
    const double nan = CUDART_NAN;
    const size_t plane = static_cast<size_t>(n_P) * n_m * n_s, step = static_cast<size_t>(n_m) * n_s;
    for (int s0 = 0; s0 < n_s; s0 += kSurfS) {
        const int si_t = s0 + threadIdx.x;
        if (s0 > 0) __syncthreads();  // the previous chunk's gaps have been read
        if (si_t < n_s) s_gs[threadIdx.x] = gap_at(s_tab, p.T.npad, static_cast<double>(s_at(p.G, si_t)));
        __syncthreads();
        for (int midx = mgroup * p.surf_m + warp; midx < min((mgroup + 1) * p.surf_m, n_m); midx += kSurfW) {
        const uint32_t m_u = p.G.m_list[midx];
        for (int c = lane; c < min(kSurfS, n_s - s0); c += 32) {
            const uint32_t s = s_at(p.G, s0 + c);
            const bool fits = s <= m_u;
            double B = nan, C = nan, Q = nan;
            if (fits) {
                const double gs = s_gs[c], k = static_cast<double>(segments(m_u, s, p.G.k_mode));
                B = gs + L;
                C = gs * (k - 1.0);
                Q = gs * k;
            }
            double *out = p.surface + (static_cast<size_t>(table - p.out_table0) * 3 * n_P + p0) * step + static_cast<size_t>(midx) * n_s + s0 + c;
            for (int pi = p0; pi < p1; ++pi, out += step) {
                const int P = P_at(p.G, pi);
                const double pm1 = static_cast<double>(P - 1);
                if (on2) out[0] = fits ? fma(pm1, Q, L) : nan;      // (P-1) (g(s) k) + L
                if (on5) out[plane] = fits ? fma(pm1, B, C) : nan;  // (P-1) (g(s)+L) + g(s)(k-1)
                if (on9)                                            // floor(log2 P) g(s) k + ceil(log2 P) L
                    out[2 * plane] = fits ? fma(static_cast<double>(31 - __clz(P)), Q, static_cast<double>(32 - __clz(P - 1)) * L) : nan;
            }
        }
        }
    }
}

// One CTA: one table, 32 V consecutive message sizes (V per lane), a chunk of process counts (warps stride over it).
// Bound by HBM: three planes read, six written.  256 tables, P = 2..512, 128 m (1.2 GB): 257 us with one size per lane
// and 64-bit index arithmetic per store, 207 us (5.8 TB/s) with two, running pointers and the loads first.
template <int V> struct FixedVec;
template <> struct FixedVec<1> {
    static __device__ __forceinline__ void load(double *v, const double *p) { v[0] = __ldcs(p); }
    static __device__ __forceinline__ void store(double *p, const double *v) { __stcs(p, v[0]); }
};
template <> struct FixedVec<2> {
    static __device__ __forceinline__ void load(double *v, const double *p)
    {
        const double2 t = __ldcs(reinterpret_cast<const double2 *>(p));
        v[0] = t.x; v[1] = t.y;
    }
    static __device__ __forceinline__ void store(double *p, const double *v) { __stcs(reinterpret_cast<double2 *>(p), make_double2(v[0], v[1])); }
};

template <int V>
__global__ void __launch_bounds__(256) fixed_kernel(const SensParams p)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    double *s_tab = reinterpret_cast<double *>(smem_raw);
    const int n_mtiles = (p.G.n_m + 32 * V - 1) / (32 * V);
    const int mtile = blockIdx.x % n_mtiles, pchunk = blockIdx.x / n_mtiles, trel = blockIdx.y;
    const int table = p.table0 + trel;
    stage_table(s_tab, p.T, table);
    __syncthreads();
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, n_warps = blockDim.x >> 5;
    const int midx = mtile * 32 * V + lane * V;
    if (midx >= p.G.n_m) return;  // no barriers below; V = 2 is taken for even n_m only
    const double L = p.T.lat[table];
    double B[V], C[V], Q[V];
#pragma unroll
    for (int v = 0; v < V; ++v) {
        const uint32_t m_u = p.G.m_list[midx + v];
        // the fixed size where it fits, else the whole message in one segment (Section 3.1)
        const uint32_t s_eff = p.s_fixed <= m_u ? p.s_fixed : m_u;
        const double gs = gap_at(s_tab, p.T.npad, static_cast<double>(s_eff));
        const double k = static_cast<double>(segments(m_u, s_eff, p.G.k_mode));
        B[v] = gs + L; C[v] = gs * (k - 1.0); Q[v] = gs * k;
    }
    const uint32_t mask = p.G.mask;
    const bool on[3] = {((mask >> 2) & 1u) != 0, ((mask >> 5) & 1u) != 0, ((mask >> 9) & 1u) != 0};
    const int ids[3] = {2, 5, 9};
    const int n_P = p.G.n_P, n_m = p.G.n_m;
    const size_t plane = static_cast<size_t>(n_P) * n_m;
    const int p0 = pchunk * p.p_per_cta, p1 = min(p0 + p.p_per_cta, n_P);
    const size_t cell = static_cast<size_t>(p0 + warp) * n_m + midx, step = static_cast<size_t>(n_warps) * n_m;
    double *out = p.time_fixed + static_cast<size_t>(table - p.out_table0) * 3 * plane + cell;
    double *rat = p.ratio ? p.ratio + static_cast<size_t>(table - p.out_table0) * 3 * plane + cell : nullptr;
    const double *in = p.pred_time ? p.pred_time + static_cast<size_t>(table - p.out_table0) * 13 * plane + cell : nullptr;
    for (int pi = p0 + warp; pi < p1; pi += n_warps) {
        double best[3][V];
        if (rat) {
#pragma unroll
            for (int q = 0; q < 3; ++q)
                if (on[q]) FixedVec<V>::load(best[q], in + ids[q] * plane);
            in += step;
        }
        const int P = P_at(p.G, pi);
        const double pm1 = static_cast<double>(P - 1), lf = static_cast<double>(31 - __clz(P)), lcL = static_cast<double>(32 - __clz(P - 1)) * L;
        double t[3][V];
#pragma unroll
        for (int v = 0; v < V; ++v) {
            t[0][v] = fma(pm1, Q[v], L);
            t[1][v] = fma(pm1, B[v], C[v]);
            t[2][v] = fma(lf, Q[v], lcL);
        }
#pragma unroll
        for (int q = 0; q < 3; ++q)
            if (on[q]) FixedVec<V>::store(out + q * plane, t[q]);
        out += step;
        if (rat) {
#pragma unroll
            for (int q = 0; q < 3; ++q) {
                if (!on[q]) continue;
#pragma unroll
                for (int v = 0; v < V; ++v) t[q][v] /= best[q][v];
                FixedVec<V>::store(rat + q * plane, t[q]);
            }
            rat += step;
        }
    }
}

__global__ void boundary_kernel(const uint8_t *strategy, uint8_t *boundary, long long n_planes, int n_P, int n_m)
{
    const long long total = n_planes * n_P * n_m;
    for (long long i = blockIdx.x * static_cast<long long>(blockDim.x) + threadIdx.x; i < total;
         i += static_cast<long long>(gridDim.x) * blockDim.x) {
        const int im = static_cast<int>(i % n_m), ip = static_cast<int>((i / n_m) % n_P);
        const uint8_t s = strategy[i];
        uint8_t b = 0;
        if (ip + 1 < n_P && strategy[i + n_m] != s) b |= 1;  // the next larger process count selects another strategy
        if (im + 1 < n_m && strategy[i + 1] != s) b |= 2;    // the next larger message size does
        boundary[i] = b;
    }
}

// The same, 4 W consecutive message sizes per thread (n_m a multiple of that, arrays aligned for it), walking down
// kBndRows process counts, so that every row is read once and the index arithmetic is shared (256 tables, P = 2..512,
// 128 m, 67 MB: 29 us with one row of 8 sizes per thread, 17 us so).
constexpr int kBndRows = 8;
template <int W>
__global__ void __launch_bounds__(256) boundary_rows_kernel(const uint8_t *strategy, uint8_t *boundary, long long n_planes, int n_P, int n_m)
{
    struct __align__(4 * W) Words { unsigned w[W]; };
    const int groups = n_m / (4 * W), chunks = (n_P + kBndRows - 1) / kBndRows;
    const long long total = n_planes * chunks * groups;
    for (long long idx = blockIdx.x * static_cast<long long>(blockDim.x) + threadIdx.x; idx < total; idx += static_cast<long long>(gridDim.x) * blockDim.x) {
        const long long rest = idx / groups;
        const int g = static_cast<int>(idx - rest * groups);
        const long long pl = rest / chunks;
        const int ip0 = static_cast<int>(rest - pl * chunks) * kBndRows, ip1 = min(ip0 + kBndRows, n_P);
        const uint8_t *in = strategy + (pl * n_P + ip0) * n_m + 4LL * W * g;
        uint8_t *out = boundary + (in - strategy);
        Words row = *reinterpret_cast<const Words *>(in);
        for (int ip = ip0; ip < ip1; ++ip, in += n_m, out += n_m) {
            const Words below = ip + 1 < n_P ? *reinterpret_cast<const Words *>(in + n_m) : row;
            // the right neighbours: this group shifted by one byte, its last byte taken from the next group (or itself
            // at the end of the row, which has no neighbour)
            const unsigned last = g + 1 < groups ? in[4 * W] : row.w[W - 1] >> 24;
            Words o;
#pragma unroll
            for (int w = 0; w < W; ++w) {
                const unsigned right = __funnelshift_r(row.w[w], w + 1 < W ? row.w[w + 1] : last, 8);
                o.w[w] = __vsetne4(row.w[w], below.w[w]) | __vsetne4(row.w[w], right) << 1;
            }
            *reinterpret_cast<Words *>(out) = o;
            row = below;
        }
    }
}

cudaError_t launch_surface(const SensParams &p, cudaStream_t st)
{
    const size_t smem = (3 * static_cast<size_t>(p.T.npad) + kSurfS) * sizeof(double);
    const long long bx = static_cast<long long>((p.G.n_m + p.surf_m - 1) / p.surf_m) * ((p.G.n_P + kSurfP - 1) / kSurfP);
    if (bx <= 0 || bx > 0x7FFFFFFFLL || p.n_tables_launch <= 0 || p.n_tables_launch > 65535) return cudaErrorInvalidConfiguration;
    return launch(surface_kernel, static_cast<unsigned>(bx), static_cast<unsigned>(p.n_tables_launch), kSurfS, smem, st, false, p);
}

cudaError_t launch_fixed(const SensParams &p, cudaStream_t st)
{
    const size_t smem = 3 * static_cast<size_t>(p.T.npad) * sizeof(double);
    const int per_cta = 32 * p.vec;
    const long long bx = static_cast<long long>((p.G.n_m + per_cta - 1) / per_cta) * ((p.G.n_P + p.p_per_cta - 1) / p.p_per_cta);
    if (bx <= 0 || bx > 0x7FFFFFFFLL || p.n_tables_launch <= 0 || p.n_tables_launch > 65535) return cudaErrorInvalidConfiguration;
    return launch(p.vec == 2 ? fixed_kernel<2> : fixed_kernel<1>, static_cast<unsigned>(bx), static_cast<unsigned>(p.n_tables_launch), 256, smem, st, false, p);
}

cudaError_t launch_boundaries(const uint8_t *d_strategy, uint8_t *d_boundary, long long n_planes, int n_P, int n_m, int sm_count, cudaStream_t st)
{
    const long long total = n_planes * n_P * n_m;
    if (total <= 0) return cudaSuccess;
    const uintptr_t both = reinterpret_cast<uintptr_t>(d_strategy) | reinterpret_cast<uintptr_t>(d_boundary);
    const int w = n_m % 16 == 0 && both % 16 == 0 ? 4 : (n_m % 8 == 0 && both % 8 == 0 ? 2 : 0);
    const long long items = w ? n_planes * ((n_P + kBndRows - 1) / kBndRows) * (n_m / (4 * w)) : total;
    const unsigned blocks = static_cast<unsigned>(std::min<long long>((items + 255) / 256, static_cast<long long>(sm_count) * 32));
    if (w == 4) boundary_rows_kernel<4><<<blocks, 256, 0, st>>>(d_strategy, d_boundary, n_planes, n_P, n_m);
    else if (w == 2) boundary_rows_kernel<2><<<blocks, 256, 0, st>>>(d_strategy, d_boundary, n_planes, n_P, n_m);
    else boundary_kernel<<<blocks, 256, 0, st>>>(d_strategy, d_boundary, n_planes, n_P, n_m);
    return cudaGetLastError();
}

}  // namespace plogp
