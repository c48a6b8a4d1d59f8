// A CUDA runtime and kernels made of host memory, for csrc/api.cu on a machine without a GPU: allocations are counted and can
// be refused, every launch checks that the scratch it is given lies inside a live allocation, and nothing is computed.
#include <cuda_runtime.h>

template <typename F>  // as nvcc has it
static cudaError_t cudaFuncSetAttribute(F *f, cudaFuncAttribute a, int v) { return cudaFuncSetAttribute(reinterpret_cast<const void *>(f), a, v); }

#include "../paper_cs_0408034_b200/csrc/internal.h"
#include "../paper_cs_0408034_b200/csrc/lines_layout.h"

#include <cstdlib>
#include <cstring>
#include <map>
#include <new>

namespace {
std::map<const unsigned char *, size_t> live;
long long refuse_at = -1, bad = 0, launches = 0;  // refuse_at: allocations from that size on fail (-1: none)
long long too_large = 0, staged = 0, direct = 0;  // launches with more shared memory than an SM has; with all message sizes in a CTA; a cell per thread

void inside(const void *p, size_t bytes)
{
    auto it = live.upper_bound(static_cast<const unsigned char *>(p));
    if (it == live.begin()) { ++bad; return; }
    --it;
    if (static_cast<const unsigned char *>(p) + bytes > it->first + it->second) ++bad;
}
long long refuse_host_at = -1;  // likewise for operator new, api.cu's own
cudaError_t launched() { ++launches; return cudaSuccess; }
}  // namespace

void *operator new(size_t n)
{
    if (refuse_host_at >= 0 && static_cast<long long>(n) >= refuse_host_at) throw std::bad_alloc();
    if (void *p = std::malloc(n ? n : 1)) return p;
    throw std::bad_alloc();
}
void operator delete(void *p) noexcept { std::free(p); }
void operator delete(void *p, size_t) noexcept { std::free(p); }

extern "C" {
void fake_refuse_host_from(long long bytes) { refuse_host_at = bytes; }
void fake_refuse_from(long long bytes) { refuse_at = bytes; }
long long fake_bad_accesses() { return bad; }
long long fake_launches() { return launches; }
long long fake_too_large() { return too_large; }
long long fake_staged() { return staged; }
long long fake_direct() { return direct; }
long long fake_live_bytes() { long long n = 0; for (auto &a : live) n += static_cast<long long>(a.second); return n; }

cudaError_t cudaMalloc(void **p, size_t n)
{
    if (refuse_at >= 0 && static_cast<long long>(n) >= refuse_at) return cudaErrorMemoryAllocation;
    *p = std::aligned_alloc(256, (n + 255) / 256 * 256);
    live[static_cast<unsigned char *>(*p)] = n;
    return cudaSuccess;
}
cudaError_t cudaFree(void *p)
{
    if (!live.erase(static_cast<unsigned char *>(p))) { ++bad; return cudaErrorInvalidValue; }
    std::free(p);
    return cudaSuccess;
}
cudaError_t cudaMemcpyAsync(void *d, const void *s, size_t n, cudaMemcpyKind kind, cudaStream_t)
{
    inside(kind == cudaMemcpyHostToDevice ? d : s, n);
    if (!bad) std::memcpy(d, s, n);
    return cudaSuccess;
}
cudaError_t cudaGetDevice(int *d) { *d = 0; return cudaSuccess; }
cudaError_t cudaDeviceGetAttribute(int *v, cudaDeviceAttr, int) { *v = 148; return cudaSuccess; }
cudaError_t cudaGetLastError() { return cudaSuccess; }
const char *cudaGetErrorName(cudaError_t) { return "fake"; }
const char *cudaGetErrorString(cudaError_t) { return "fake"; }
cudaError_t cudaStreamSynchronize(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamCreateWithFlags(cudaStream_t *s, unsigned) { *s = nullptr; return cudaSuccess; }
cudaError_t cudaStreamDestroy(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamWaitEvent(cudaStream_t, cudaEvent_t, unsigned) { return cudaSuccess; }
cudaError_t cudaEventCreate(cudaEvent_t *e) { *e = reinterpret_cast<cudaEvent_t>(1); return cudaSuccess; }
cudaError_t cudaEventCreateWithFlags(cudaEvent_t *e, unsigned) { *e = reinterpret_cast<cudaEvent_t>(1); return cudaSuccess; }
cudaError_t cudaEventDestroy(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaEventSynchronize(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventElapsedTime(float *ms, cudaEvent_t, cudaEvent_t) { *ms = 0.f; return cudaSuccess; }
}

// A kernel's limit on dynamic shared memory, for all threads; another thread's call may come in between any two of a call's own.
namespace {
int limit = 48 * 1024;
void (*other_thread)() = nullptr;
void kernel(int) {}
}  // namespace
extern "C" {
cudaError_t cudaFuncSetAttribute(const void *, cudaFuncAttribute, int v)
{
    limit = v;
    if (auto f = other_thread) { other_thread = nullptr; f(); }
    return cudaSuccess;
}
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t *c, const void *, void **)
{
    return static_cast<int>(c->dynamicSmemBytes) <= limit ? cudaSuccess : cudaErrorInvalidValue;
}
// a launch with `mine` bytes while another thread launches the same kernel with `theirs`
int fake_launch_beside(int mine, int theirs_)
{
    static int theirs;
    static cudaError_t e;
    theirs = theirs_;
    e = cudaSuccess;
    other_thread = [] { e = plogp::launch(kernel, 1, 1, 32, theirs, nullptr, false, 0); };
    const cudaError_t own = plogp::launch(kernel, 1, 1, 32, mine, nullptr, false, 0);
    if (other_thread) { auto f = other_thread; other_thread = nullptr; f(); }
    return own == cudaSuccess && e == cudaSuccess;
}
}

namespace plogp {

static void check_parts(const double *t, const uint32_t *i, size_t rows, int n_P)
{
    inside(t, rows * n_P * sizeof(double));
    inside(i, rows * n_P * sizeof(uint32_t));
}
static void check_gaps(const double *g, size_t stride, int nt)
{
    if (g) inside(g, stride * nt * sizeof(double));
}
cudaError_t launch_gaps(const GapsParams &p, cudaStream_t)
{
    inside(p.gaps, sizeof(double) * p.stride * p.n_tables_launch);
    return launched();
}
cudaError_t launch_sweep(const SweepParams &p, int nt, int *n, cudaStream_t)
{
    check_parts(p.part_time, p.part_idx, size_t(nt) * p.n_seg * p.n_pairs, p.G.n_P);
    *n = 1;
    return launched();
}
cudaError_t launch_envelope(const EnvParams &p, int, cudaStream_t)
{
    check_parts(p.part_time, p.part_idx, size_t(p.n_tables_launch) * p.n_seg * p.G.n_m, p.G.n_P);
    return launched();
}
cudaError_t launch_fused(const FusedParams &p, bool, bool, cudaStream_t)
{
    if (p.part_time) check_parts(p.part_time, p.part_idx, size_t(p.n_tables_launch) * p.n_seg * p.n_pairs, p.G.n_P);
    return launched();
}
static cudaError_t check_lines(const LinesParams &p)
{
    check_gaps(p.gaps, p.gaps_stride, p.n_tables_launch);
    staged += p.staged != 0;
    direct += p.direct != 0;
    if (lines_smem_bytes(p) > size_t(kMaxSmem)) { ++too_large; return cudaErrorInvalidValue; }
    return launched();
}
cudaError_t launch_decide(const LinesParams &p, bool, cudaStream_t) { return check_lines(p); }
cudaError_t launch_segmin(const LinesParams &p, bool, cudaStream_t) { return check_lines(p); }
cudaError_t launch_scatter(const ScatterParams &, bool, cudaStream_t) { return launched(); }
cudaError_t launch_select(SelectParams &p, cudaStream_t) { return check_lines(p.decide); }
cudaError_t launch_planes(const PlanesParams &, bool, cudaStream_t) { return launched(); }
cudaError_t launch_rows(const RowsParams &, bool, bool, cudaStream_t) { return launched(); }
cudaError_t launch_layout(const LayoutParams &p, cudaStream_t)
{
    inside(p.tab, sizeof(double) * 3 * p.npad * p.n_tables);
    return launched();
}
cudaError_t launch_barrier(const TableDev &, const GridDev &, int, int, uint8_t *, uint32_t *, double *, cudaStream_t) { return launched(); }
cudaError_t launch_surface(const SensParams &, cudaStream_t) { return launched(); }
cudaError_t launch_fixed(const SensParams &, cudaStream_t) { return launched(); }
cudaError_t launch_boundaries(const uint8_t *, uint8_t *, long long, int, int, int, cudaStream_t) { return launched(); }
cudaError_t launch_fp64_probe(double *, int, int, cudaStream_t) { return launched(); }
int envelope_coarse_of(int pidx, int) { return pidx; }

}  // namespace plogp
