// Internal declarations shared by the host side (api.cu) and the kernels (kernels.cu).
// Nothing here is part of the public ABI.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

namespace plogp {

constexpr int kMaxSmem = 227 * 1024;  // shared memory of a CTA, at most

// Launches a kernel on a stream; overlap: it may start before the kernel in front of it has ended (device_common.cuh).
template <typename P>
inline cudaError_t launch(void (*kernel)(P), unsigned gx, unsigned gy, unsigned threads, size_t smem, cudaStream_t st, bool overlap, const P &params)
{
    // The limit is the kernel's, for all threads: it is only ever raised to what an SM has, or a thread with a smaller call could
    // lower it between another's two lines here.
    if (smem > 48 * 1024) {
        const cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kMaxSmem);
        if (e != cudaSuccess) return e;
    }
    cudaLaunchAttribute attr{};
    attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(gx, gy); cfg.blockDim = dim3(threads); cfg.dynamicSmemBytes = smem; cfg.stream = st;
    cfg.attrs = &attr; cfg.numAttrs = overlap ? 1u : 0u;
    return cudaLaunchKernelEx(&cfg, kernel, params);
}

// Where a decision kernel puts its results and how it names the strategies.  plogp_select_best writes two planes
// per table (Broadcast, Scatter) with the ids of Table 1 / Table 2; the derived collectives (Gather, Reduce) reuse
// the same kernels with one plane per table and the ids of the mirrored strategies.
struct OutMap {
    int planes;       // decision planes per table in the output arrays
    int plane_bcast;  // plane that receives the Broadcast-type decision
    int plane_scat;   // plane that receives the Scatter-type decision
    uint8_t id_of[16];  // output id of internal strategy id 0..12 (255 beyond)
};

// Tables as they live in device memory.  Per table: three runs of `npad` doubles
//   key[npad]   breakpoint sizes usable as interval starts (index <= n_bp-2), +inf beyond
//   gap[npad]   g at the interval start
//   slope[npad] (g[i+1]-g[i]) / (size[i+1]-size[i])
// npad is a power of two >= n_bp, so the interval search needs no bounds checks and an upward
// walk always meets a +inf key.
struct TableDev {
    const double *tab;  // [n_tables][3*npad]
    const double *lat;  // [n_tables]
    int n_tables, n_bp, npad;
};

struct GridDev {
    const int32_t *P_list;  // device [n_P] or nullptr => P = P_lo + index
    int n_P, P_lo;
    const uint32_t *m_list;  // device [n_m]
    int n_m;
    const uint32_t *s_list;  // device [n_s] or nullptr => s = s_lo + index * s_step
    int n_s;
    uint32_t s_lo, s_step;
    const int32_t *ns_of_m;  // device [n_m]: number of candidates s <= m (0 => unsegmented fallback)
    const double *k_list;    // device [n_s][n_m]: Section 2's k for every (m, candidate s <= m), short candidate lists only
    uint32_t mask;
    int k_mode;
    int lc_max;  // ceil(log2 P_hi)
};

// Segment-sweep kernel (large candidate lists): partial minima per (table, segmented strategy,
// (m, chunk) pair, P).
struct SweepParams {
    TableDev T;
    GridDev G;
    const int32_t *pair_m;      // device [n_pairs] in launch order (heaviest first)
    const int32_t *pair_chunk;  // device [n_pairs]
    const int32_t *pair_row;    // device [n_pairs]: row id of the pair (= pair_base[m] + chunk)
    int n_pairs, n_ptiles, chunk_len;
    int wp;  // tiles of 256 process counts per CTA behind the first tile (1, 2, 4 or 8); its 8 warps split the candidates 8 / wp ways
    double *part_time;   // [n_tables_batch][n_seg][n_pairs][n_P]
    uint32_t *part_idx;  // same shape: index of s in the candidate list
    int n_seg;           // enabled segmented strategies (slots in id order)
    int table0;          // first table of this launch (blockIdx.y is relative to it)
};

// Envelope kernel (exact fast path of the segment-size search): same scratch layout as the sweep kernel with
// one row per message size.
struct EnvParams {
    TableDev T;
    GridDev G;
    int table0, n_tables_launch;
    double *part_time;   // [n_tables_batch][n_seg][n_m][n_P]
    uint32_t *part_idx;  // same shape: index of s in the candidate list
    int n_seg;
    int rep_cap;     // entries of the shared-memory list of representatives (longer lists go through it in windows)
    int coarse_log;  // the coarse process-count indices are at most 2 << coarse_log apart
    int max_coarse;  // capacity of the coarse-winner array (>= number of coarse indices)
};

// Segment-size sensitivity kernels (sensitivity.cu)
struct SensParams {
    TableDev T;
    GridDev G;
    int table0, n_tables_launch, out_table0;
    int surf_m;                // message sizes per CTA (surface_kernel)
    double *surface;           // [n_tables][3][n_P][n_m][n_s]
    uint32_t s_fixed;          // the fixed segment size (fixed_kernel)
    int p_per_cta;             // process counts per CTA (fixed_kernel)
    int vec;                   // message sizes per lane (fixed_kernel): 2 where n_m is even and the arrays are 16-byte aligned
    const double *pred_time;   // [n_tables][13][n_P][n_m] from plogp_predict, or nullptr together with ratio
    double *time_fixed, *ratio;  // [n_tables][3][n_P][n_m]
};

struct FusedParams {
    TableDev T;
    GridDev G;
    int n_mtiles, n_ptiles, passes_per_tile;  // a pass covers kWarps*R process counts
    int table0, n_tables_launch;
    int out_table0;  // table whose results sit at the start of the output arrays (0 unless the caller passes a window)
    OutMap om;
    // segmented minima from the sweep or envelope kernel (nullptr: no segmented strategy in the mask)
    const double *part_time;
    const uint32_t *part_idx;
    const int32_t *pair_base;  // device [n_m+1]
    int n_pairs, n_seg;
    // outputs: decision table
    uint8_t *d_strategy;
    uint32_t *d_sbytes;
    double *d_time;
    // outputs: predicted planes
    double *p_time;
    uint32_t *p_best_s;
};

// Closed-form prediction planes cell by cell as they lie in memory: see planes.cu
struct PlanesParams {
    TableDev T;
    GridDev G;
    uint32_t mask;        // of kPlanesMask
    long long seg_cells;  // cells of a plane per CTA, a multiple of 256
    int table0, n_tables_launch, out_table0;
    double *p_time;       // [n_tables][13][n_P][n_m]
};
constexpr uint32_t kPlanesMask = 0x5DBu;  // ids 0 1 3 4 6 7 8 10
constexpr int kPlanesMaxM = 4096;         // g(m) of all message sizes in shared memory
cudaError_t launch_planes(const PlanesParams &p, bool overlap, cudaStream_t st);

// Scatter half of the decision table: see scatter.cuh
struct ScatterParams {
    TableDev T;
    GridDev G;
    int vec;  // message sizes per lane, 1 or 2 (2: n_m even and the outputs aligned for it)
    int chain_table;  // listed process counts: sums per interval in shared memory (vec 1)
    int n_mtiles, n_ptiles, run_len;  // CTAs along m (32 vec sizes each) and along P (kWarps runs of run_len process counts each)
    int table0, n_tables_launch, out_table0;
    OutMap om;
    uint8_t *d_strategy;
    uint32_t *d_sbytes;
    double *d_time;
};

// Scatter half of the decision table, or the predictions of ids 11 and 12, for a range of process counts and rows off the
// sectors: see rows.cu
struct RowsParams {
    TableDev T;
    GridDev G;
    int n_ptiles, run_len;  // CTAs along P and process counts of each
    int table0, n_tables_launch, out_table0;
    OutMap om;  // predictions: 13 planes per table, nothing else is read
    uint8_t *d_strategy;  // aligned for four cells per store: 4,
    uint32_t *d_sbytes;   // 16 and
    double *d_time;       // 32 bytes
};
constexpr int kRowsMaxM = 256;
cudaError_t launch_rows(const RowsParams &p, bool predict, bool overlap, cudaStream_t st);

// Tables as the caller has them -> TableDev's layout: see layout.cu
struct LayoutParams {
    const uint64_t *sizes;  // [n_bp] (shared) or [n_tables][n_bp]
    const double *gap;      // [n_tables][n_bp]
    double *tab;            // [n_tables][3 * npad]
    int n_tables, n_bp, npad, sizes_shared;
};
cudaError_t launch_layout(const LayoutParams &p, cudaStream_t st);

// Gap pre-pass (gaps.cu): g at every distinct argument of decide_kernel and segmin_kernel, once per table.
// Row of a table: [0] = g(1), [1 .. n_s] = g(s_i), [1 + n_s .. 1 + n_s + n_m) = g(m_j).
struct GapsParams {
    TableDev T;
    GridDev G;
    int table0, n_tables_launch;
    double *gaps;  // [n_tables_launch][stride]
    int stride;
};

// Broadcast half of the decision table, or the segmented planes of the predictions (ids 2, 5, 9), for short candidate lists:
// see lines.cuh
struct LinesParams {
    TableDev T;
    GridDev G;
    const double *gaps;  // rows of the gap pre-pass for this launch's tables, or nullptr: the kernel interpolates itself
    int gaps_stride;
    int threads;    // per CTA, at most kLineThreads
    int width;      // message sizes of a CTA, side by side: 32, 16 or 8, or all of them (staged)
    int staged;     // outputs aligned for four cells per store (times 32, sizes 16, ids 4 bytes), all message sizes in a CTA
    int n_p;        // process counts per CTA
    int direct;     // a cell per thread (direct.cuh): only gaps, outputs and n_ptiles, CTAs of kDecThreads cells per table, count
    int n_mgroups, n_ptiles;
    int n_pairs;    // (floor, ceil) pairs of log2 P in a CTA's range of process counts, at most
    const int32_t *knots;  // device [n_ptiles][kLineSegs + 2]: indices inside the CTA's process counts, number of segments
    int table0, n_tables_launch;
    int out_table0;  // table whose results sit at the start of the output arrays
    OutMap om;
    uint8_t *d_strategy;  // decision
    uint32_t *d_sbytes;
    double *d_time;
    double *p_time;      // predictions: [n_tables][13][n_P][n_m]
    uint32_t *p_best_s;  // [n_tables][3][n_P][n_m], or nullptr
};
constexpr int kLineThreads = 256;
constexpr int kLineSegs = 4;  // segments of a CTA's process counts, at most
using DecideParams = LinesParams;  // as decide_kernel takes them,
using SegminParams = LinesParams;  // and segmin_kernel

constexpr int kDecThreads = 128;
constexpr int kDecWarps = kDecThreads / 32;
constexpr int kThreads = 256;
constexpr int kWarps = kThreads / 32;
constexpr int kFusedR = 4;   // process counts per thread and pass in the fused kernel
constexpr int kSweepR = 8;   // process counts per thread in the sweep kernel
constexpr int kSweepSub = 256;  // candidates staged per sub-chunk
constexpr int kSweepGroups = kSweepSub / 32;  // groups of a sub-chunk
constexpr int kSweepSeeds = 128;  // log-spaced candidates that the upper bounds start from
constexpr int kMaxInlineS = 64;

cudaError_t launch_fused(const FusedParams &p, bool predict, bool overlap, cudaStream_t st);
cudaError_t launch_scatter(const ScatterParams &p, bool overlap, cudaStream_t st);  // decision table, Scatter strategies only
cudaError_t launch_sweep(const SweepParams &p, int n_tables_launch, int *launches, cudaStream_t st);
cudaError_t launch_decide(const DecideParams &p, bool overlap, cudaStream_t st);
// both halves of a decision table in one launch: see select.cu (launch_select fills in n_decide)
struct SelectParams {
    DecideParams decide;
    ScatterParams scatter;
    int n_decide;
};
size_t scatter_smem_bytes(const ScatterParams &p, int warps);
cudaError_t launch_select(SelectParams &p, cudaStream_t st);
cudaError_t launch_fp64_probe(double *d_sink, int iters, int blocks, cudaStream_t st);
cudaError_t launch_segmin(const SegminParams &p, bool overlap, cudaStream_t st);
cudaError_t launch_gaps(const GapsParams &p, cudaStream_t st);
cudaError_t launch_barrier(const TableDev &T, const GridDev &G, int table0, int n_tables_launch, uint8_t *d_strategy, uint32_t *d_sbytes,
                           double *d_time, cudaStream_t st);
cudaError_t launch_surface(const SensParams &p, cudaStream_t st);
cudaError_t launch_fixed(const SensParams &p, cudaStream_t st);
cudaError_t launch_boundaries(const uint8_t *d_strategy, uint8_t *d_boundary, long long n_planes, int n_P, int n_m, int sm_count, cudaStream_t st);
size_t envelope_smem_bytes(const TableDev &T, int threads, int rep_cap, int max_coarse);
__host__ __device__ int envelope_coarse_of(int pidx, int g_max);  // number of the last coarse index at or below pidx
cudaError_t launch_envelope(const EnvParams &p, int threads, cudaStream_t st);

}  // namespace plogp
