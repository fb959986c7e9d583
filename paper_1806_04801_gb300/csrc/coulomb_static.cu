// hsma_coulomb_sum_static: the direct Coulomb sum of hsma_coulomb_sum, for
// callers that must not allocate device memory at call time.
//
// Some callers cannot let a library call cudaMalloc/cudaFree while they run:
// a host application whose memory manager owns the whole device and forbids
// outside allocations after start-up, or a time-critical loop for which the
// implicit device-wide synchronisation of cudaFree is unacceptable.  This
// entry point takes all of its working memory from one array of
// kStaticScratchBytes that lives in this file as a static __device__ object:
// the driver reserves it when it loads this part of the library, every GPU
// that loads it keeps it until the process exits, and no call allocates.
//
// The array is shared by every call on a device and keeps the contents the
// last call left; each call first clears what must start at zero (work
// counter, status word) with a kernel.  Calls whose device work overlaps --
// on two streams, or from two host threads -- race on the array and give
// wrong results: serialise them.
//
// The first call on each device looks up the array's device address with
// cudaGetSymbolAddress (host code cannot use the symbol itself as a device
// pointer) and caches it with the identity of the current context; make that
// first call before any stream capture.  A later call in a different context
// (the device was reset, and the module loaded again) looks it up anew.
#include <cuda.h>
#include <limits.h>
#include <math.h>
#include <string.h>

#include <algorithm>
#include <mutex>

#include "common.cuh"

namespace hsma {

// Process-unique id of the current context (cuCtxGetId), reached through the
// runtime's driver entry-point table so that the library needs no link
// against the driver library.  Returns false where the driver lacks it.
bool current_context_id(unsigned long long *id)
{
    using GetCurrent = CUresult (*)(CUcontext *);
    using GetId = CUresult (*)(CUcontext, unsigned long long *);
    static GetCurrent get_current = nullptr;
    static GetId get_id = nullptr;
    static std::once_flag once;
    std::call_once(once, [] {
        void *f = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuCtxGetCurrent", &f, 12000, cudaEnableDefault, &q) == cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            get_current = reinterpret_cast<GetCurrent>(f);
        f = nullptr;
        if (cudaGetDriverEntryPointByVersion("cuCtxGetId", &f, 12000, cudaEnableDefault, &q) == cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            get_id = reinterpret_cast<GetId>(f);
        cudaGetLastError();
    });
    CUcontext c = nullptr;
    if (!get_current || !get_id || get_current(&c) != CUDA_SUCCESS || !c) return false;
    return get_id(c, id) == CUDA_SUCCESS;
}

namespace {

constexpr size_t kStaticScratchBytes = (size_t)HSMA_STATIC_SCRATCH_BYTES;
static __device__ __align__(256) unsigned char g_static_scratch[kStaticScratchBytes];

constexpr int kMaxDevices = 64;
std::mutex g_static_mu;
void *g_scratch_addr[kMaxDevices] = {};
unsigned long long g_scratch_ctx[kMaxDevices] = {};  // context id the address belongs to
int g_num_sms[kMaxDevices] = {};

size_t up256(size_t v) { return (v + 255) / 256 * 256; }

struct StaticLayout {
    size_t shi, slo, s64, thi, tlo, t64, partials, ns, ctrl, status, sys, end;
};

// Byte offsets of every buffer inside the static array for one call.
StaticLayout layout_for(long long ns, long long nt, int nchunks, int precision)
{
    StaticLayout L;
    size_t o = 0;
    auto put = [&](size_t bytes) {
        size_t at = o;
        o = up256(o + bytes);
        return at;
    };
    const bool f64 = precision == HSMA_FP64;
    L.shi = put(f64 ? 0 : (size_t)ns * sizeof(float4));
    L.slo = put(f64 ? 0 : (size_t)ns * sizeof(float4));
    L.s64 = put(f64 ? (size_t)ns * sizeof(double4_32a) : 0);
    L.thi = put((size_t)nt * sizeof(float4));
    L.tlo = put((size_t)nt * sizeof(float4));
    L.t64 = put((size_t)nt * sizeof(double4_32a));
    L.partials = put((size_t)nchunks * nt * 2 * sizeof(float4));
    put((size_t)nt * 4 * sizeof(double));  // not used: keeps the sizes that fit what they were
    L.ns = put(sizeof(long long));
    L.ctrl = put(16 * sizeof(int));
    L.status = put(sizeof(int));
    L.sys = put(sizeof(SysDesc));
    L.end = o;
    return L;
}

// Writes the work description, clears the counters and status and empties the
// boxes of the coordinates.
__global__ void coulomb_init_kernel(SysDesc d, long long ns, SysDesc *dsys, long long *dns, int *ctrl, int *status)
{
    if (threadIdx.x == 0) {
        *dsys = d;
        *dns = ns;
        *status = 0;
    }
    if (threadIdx.x < 2) ctrl[threadIdx.x] = 0;
    if (threadIdx.x >= 2 && threadIdx.x < 14) ctrl[threadIdx.x] = (threadIdx.x - 2) % 6 < 3 ? INT_MAX : INT_MIN;
}

// Slot of source i of n for the packed FP32 loop, whose two lanes take the even
// and the odd slots of a run of kPackedFold: the first half of a run's sources
// in order to the one, the second half to the other.  In the caller's order the
// lanes would take every other source, which sums charges of alternating sign
// (a salt listed pair by pair) as two long sums of one sign each.
__device__ __forceinline__ long long lane_run_slot(long long i, long long n)
{
    const int o = (int)(i % kPackedFold), m = (int)min((long long)kPackedFold, n - (i - o)), half = (m + 1) / 2;
    return i - o + (o < half ? 2 * o : 2 * (o - half) + 1);
}

// Sources and targets into the pair kernels' records: FP32 word pairs, or FP64
// records and the boxes of both (one pass over each; the first
// `sblocks` blocks take the sources).
constexpr int kSplitThreads = 256;
__global__ void __launch_bounds__(kSplitThreads) coulomb_split_kernel(long long ns, const double *src, long long nt,
                                                                      const double *tgt, unsigned sblocks, bool f64,
                                                                      CoulombBuffers b)
{
    __shared__ int red[6][kSplitThreads / 32];
    const bool is_src = blockIdx.x < sblocks;
    const long long i = (long long)(is_src ? blockIdx.x : blockIdx.x - sblocks) * kSplitThreads + threadIdx.x;
    const bool live = i < (is_src ? ns : nt);
    const double *p = is_src ? src + 4 * i : tgt + 3 * i;
    const double x = live ? p[0] : 0.0, y = live ? p[1] : 0.0, z = live ? p[2] : 0.0;
    const double q = live && is_src ? p[3] : 0.0;
    if (!f64) {
        if (!live) return;
        float hx, lx, hy, ly, hz, lz;
        split_f64(x, hx, lx);
        split_f64(y, hy, ly);
        split_f64(z, hz, lz);
        const long long k = is_src ? lane_run_slot(i, ns) : i;
        (is_src ? b.shi : b.thi)[k] = make_float4(hx, hy, hz, (float)q);
        (is_src ? b.slo : b.tlo)[k] = make_float4(lx, ly, lz, 0.f);
        return;
    }
    if (live) (is_src ? b.s64 : b.t64)[i] = make_double4_32a(x, y, z, q);
    const double v[3] = {x, y, z};
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        const int lo = live ? box_key(__float_as_int(__double2float_rd(v[a]))) : INT_MAX;
        const int hi = live ? box_key(__float_as_int(__double2float_ru(v[a]))) : INT_MIN;
        const int wl = __reduce_min_sync(0xffffffffu, lo), wh = __reduce_max_sync(0xffffffffu, hi);
        if (lane == 0) {
            red[a][wid] = wl;
            red[3 + a][wid] = wh;
        }
    }
    __syncthreads();
    if (threadIdx.x < 6) {
        int m = red[threadIdx.x][0];
        for (int w = 1; w < kSplitThreads / 32; ++w)
            m = threadIdx.x < 3 ? min(m, red[threadIdx.x][w]) : max(m, red[threadIdx.x][w]);
        int *key = &b.ctrl[(is_src ? 2 : 8) + threadIdx.x];
        if (threadIdx.x < 3)
            atomicMin(key, m);
        else
            atomicMax(key, m);
    }
}

// Once per device and context: the static array's device address and the
// SM count, looked up with the device current (the lookup itself makes the
// runtime's context current on a first call).  Without a context id from the
// driver, the address is looked up on every call.
int static_setup(int dev, void **addr, int *sms)
{
    std::lock_guard<std::mutex> lk(g_static_mu);
    if (dev < 0 || dev >= kMaxDevices) return HSMA_E_ARG;
    unsigned long long ctx = 0;
    bool have_ctx = current_context_id(&ctx);
    if (!g_scratch_addr[dev] || !have_ctx || g_scratch_ctx[dev] != ctx) {
        void *p = nullptr;
        HSMA_CUDA_TRY(cudaGetSymbolAddress(&p, g_static_scratch));
        int n = 0;
        HSMA_CUDA_TRY(cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev));
        have_ctx = current_context_id(&ctx);
        g_num_sms[dev] = n;
        g_scratch_addr[dev] = p;
        g_scratch_ctx[dev] = have_ctx ? ctx : 0;
    }
    *addr = g_scratch_addr[dev];
    *sms = g_num_sms[dev];
    return HSMA_OK;
}

}  // namespace

// Targets of a block, chunks of the sources: items of four tiles, of fewer --
// down to one -- where four would leave less than eight items per CTA slot
// (two -> eight: FP64 20011 sources x 3001 targets 562 -> 531 us, 1e5 x 1000 880
// -> 782; FP32 2e4 x 2e4 348 -> 322).
SysDesc coulomb_shape(long long ns, long long nt, int precision, int slots)
{
    const int TB = pair_targets_per_block(precision, kCoulombVariant);
    const double tile = pair_sources_per_tile(precision, kCoulombVariant);
    SysDesc d{};
    d.ntb = (int)((nt + TB - 1) / TB);
    const double work = (double)d.ntb * ns;
    const double chunk =
        std::max(std::min(4.0 * tile, std::max(tile, work / (8.0 * slots))), work / (24.0 * slots));
    const long long most = std::max(1LL, (long long)std::ceil(ns / tile));
    d.nchunks = (int)std::max(1LL, std::min(most, (long long)llround(ns / chunk)));
    return d;
}

// Four launches and no copy: the records are made and the results written by
// the kernels themselves.
int launch_coulomb(const CoulombBuffers &b, const SysDesc &d, long long ns, const double *src, long long nt,
                   const double *tgt, double *pot, double *field, int precision, long long items, int slots,
                   cudaStream_t st)
{
    const bool f64 = precision == HSMA_FP64;
    coulomb_init_kernel<<<1, 32, 0, st>>>(d, ns, b.sys, b.ns, b.ctrl, b.status);
    HSMA_LAUNCHED();
    const unsigned sb = (unsigned)((ns + kSplitThreads - 1) / kSplitThreads);
    const unsigned tb = (unsigned)((nt + kSplitThreads - 1) / kSplitThreads);
    coulomb_split_kernel<<<sb + tb, kSplitThreads, 0, st>>>(ns, src, nt, tgt, sb, f64, b);
    HSMA_LAUNCHED();
    PairArgs pa;
    pa.sys = b.sys;
    pa.nsys = 1;
    pa.total_items = (int)items;
    pa.ns = b.ns;
    pa.src_hi = b.shi;
    pa.src_lo = b.slo;
    pa.src64 = b.s64;
    pa.ext_hi = b.thi;
    pa.ext_lo = b.tlo;
    pa.ext64 = b.t64;
    pa.n_ext = (int)nt;
    pa.ext_field = field ? 1 : 0;
    pa.ext_skip_zero = 1;
    pa.fx_box = b.ctrl + 2;
    pa.partials = b.partials;
    pa.next_item = b.ctrl;
    pa.status = b.status;
    const int grid = (int)std::max(1LL, std::min(items, (long long)slots));
    int rc = launch_pair(pa, precision, kCoulombVariant, grid, st);
    if (rc) return rc;
    return launch_partial_reduce(b.sys, 1, nt, (int)nt, b.partials, precision, pot, field, st);
}

}  // namespace hsma

using namespace hsma;

extern "C" int hsma_coulomb_sum_static(int64_t ns, const double *src, int64_t nt, const double *tgt, double *pot,
                                       double *field, int precision, void *stream)
{
    if (ns < 1 || nt < 1 || !src || !tgt || !pot) return HSMA_E_ARG;
    if (precision != HSMA_FP64 && precision != HSMA_FP32_ACC64) return HSMA_E_ARG;
    if (((uintptr_t)src | (uintptr_t)tgt | (uintptr_t)pot | (uintptr_t)field) & 7) return HSMA_E_ARG;
    if (ns > (1LL << 31) || nt > (1LL << 30)) return HSMA_E_CAPACITY;
    int dev = 0;
    HSMA_CUDA_TRY(cudaGetDevice(&dev));
    void *base = nullptr;
    int sms = 0;
    int rc = static_setup(dev, &base, &sms);
    if (rc) return rc;

    // work decomposition as in hsma_coulomb_sum, with the chunk count lowered
    // until the call fits in the static array
    const int slots = sms * pair_max_ctas_per_sm(precision, kCoulombVariant);
    SysDesc d = coulomb_shape(ns, nt, precision, slots);
    int nchunks = d.nchunks;
    while (nchunks > 1 && layout_for(ns, nt, nchunks, precision).end > kStaticScratchBytes) nchunks = nchunks / 2;
    StaticLayout L = layout_for(ns, nt, nchunks, precision);
    if (L.end > kStaticScratchBytes) return HSMA_E_CAPACITY;
    d.nchunks = nchunks;
    const long long items = (long long)d.ntb * d.nchunks;
    if (items > (1LL << 30)) return HSMA_E_CAPACITY;

    char *b = (char *)base;
    CoulombBuffers w;
    w.shi = (float4 *)(b + L.shi);
    w.slo = (float4 *)(b + L.slo);
    w.s64 = (double4_32a *)(b + L.s64);
    w.thi = (float4 *)(b + L.thi);
    w.tlo = (float4 *)(b + L.tlo);
    w.t64 = (double4_32a *)(b + L.t64);
    w.partials = (float4 *)(b + L.partials);
    w.ns = (long long *)(b + L.ns);
    w.ctrl = (int *)(b + L.ctrl);
    w.status = (int *)(b + L.status);
    w.sys = (SysDesc *)(b + L.sys);
    cudaStream_t st = (cudaStream_t)stream;
    if ((rc = launch_coulomb(w, d, ns, src, nt, tgt, pot, field, precision, items, slots, st))) return rc;
    int hst = 0;
    HSMA_CUDA_TRY(cudaMemcpyAsync(&hst, w.status, sizeof(int), cudaMemcpyDeviceToHost, st));
    HSMA_CUDA_TRY(cudaStreamSynchronize(st));
    if (hst & ST_TIMEOUT) return HSMA_E_TIMEOUT;
    return HSMA_OK;
}
