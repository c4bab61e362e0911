// Allocation-free global update (opf_global_update_static, see include/opf.h).
//
// The same computation as the global update behind opf_get_solution, for
// callers that cannot allocate device memory: control loops that forbid
// allocation once they run (an allocation may block or fail at any time), and
// hosts whose device memory is handed out only by their own allocator (a
// framework's caching allocator that owns the whole device).  Its scratch (one
// FP64 objective partial per block) is a file-scope __device__
// array instead of memory from a handle, so the call allocates nothing.
#include <cooperative_groups.h>
#include <cuda.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstring>
#include <map>
#include <mutex>
#include <string>

#include "opf_internal.h"

namespace {

namespace cg = cooperative_groups;

constexpr int kThreads = 256;
// Launch forms by the number of globals: one block, which sums the objective
// itself; one cluster of blocks; a grid and a second launch that sums the
// blocks' shares.  us per call in a graph and from a host that enqueues calls
// back to back (the host is the bound there: a second launch costs it 1.9 us):
//   globals        65       256       400       520      2000      4096      8192
//   one block   2.5, 7.8  3.5, 7.8  4.5, 7.9  5.1, 7.8    -         -         -
//   cluster     3.5, 7.7  3.6, 7.7  3.4, 7.7  3.5, 7.7  4.4, 7.8  5.9, 8.2  7.9, 10.2
//   two launches   -         -         -      4.8, 9.8  5.0, 9.6  5.1, 9.7  4.9, 9.6
constexpr int kOneBlock = 256;       // up to so many globals: one block
constexpr int kOneCluster = 4096;    // up to so many: one cluster
constexpr int kCluster = 8;          // its blocks, of up to kClusterThreads
constexpr int kClusterThreads = 512;
constexpr int kBlocks = 8 * 152;     // most blocks of the grid (a few per SM of the whole GPU): more globals than
                                     // threads go round by round
constexpr int kRecip = 16;           // 1 / (rho N) by copy count below this

// Per-block partial sums of c^T x.  Shared by every call in a CUDA context and
// kept between calls; each call writes the entries it later reads.
static __device__ __align__(256) double g_static_partials[OPF_STATIC_MAX_BLOCKS];

struct Recips {
    double r[kRecip];                // 1 / (rho N), 0 where that is not a normal number (then the division is done)
};

// What bounds these kernels: the FP64 pipe (a warp's FP64 instruction occupies
// its sub-partition's for about 64 cycles; 2 million globals in 15 us of memory
// traffic), so the forms below count FP64 instructions.

// num / den: one multiply by den's reciprocal and one correction step (the
// quotient's residual by FMA) instead of the 20-odd instructions of a division;
// the same to the last bit but one.  Infinite and NaN quotients are the
// multiply's.
__device__ __forceinline__ double quotient(double num, double den, double rcp) {
    const double q = num * rcp;
    if ((__double2hiint(q) & 0x7ff00000) == 0x7ff00000) return q;
    return fma(fma(-q, den, num), rcp, q);
}

// Order-preserving integer of a double that is not NaN.
__device__ __forceinline__ long long ordered(double x) {
    const long long b = __double_as_longlong(x);
    return b ^ ((b >> 63) & 0x7fffffffffffffffll);
}
__device__ __forceinline__ bool is_nan(double x) {
    return (unsigned long long)(__double_as_longlong(x) << 1) > 0xffe0000000000000ull;
}

// x_i = clip((sum of u over the copies of global i - c_i) / (rho N_i), lb_i, ub_i)
__device__ __forceinline__ double global_update(int a, int b, const double *u, double c, double lb, double ub,
                                                double rho, const Recips &rc) {
    const int cnt = b - a;
    double sigma = cnt > 0 ? u[a] : 0.0;
    for (int q = a + 1; q < b; ++q) sigma += u[q];
    const double num = sigma - c;
    const double rcp = cnt > 0 && cnt < kRecip ? rc.r[cnt] : 0.0;
    double x = rcp != 0.0 ? quotient(num, rho * (double)cnt, rcp) : num / (rho * (double)cnt);
    if (!is_nan(x)) {                        // NaN stays NaN; a bound that is NaN bounds nothing
        if (ordered(x) < ordered(lb) && !is_nan(lb)) x = lb;
        if (ordered(x) > ordered(ub) && !is_nan(ub)) x = ub;
    }
    return x;
}

// Sum over a block in a fixed order, in thread 0.
__device__ __forceinline__ double block_sum(double v) {
    __shared__ double red[32];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, nw = (int)(blockDim.x + 31) >> 5;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    if (lane == 0) red[w] = v;
    __syncthreads();
    if (w == 0) {
        v = lane < nw ? red[lane] : 0.0;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    }
    return v;
}

// The update of this thread's globals (round by round when there are more than
// threads) and its share of c^T x.
__device__ __forceinline__ double update_share(int n, const int *seg_off, const double *u, const double *c,
                                               const double *lb, const double *ub, double rho, const Recips &rc,
                                               double *x) {
    double o = 0.0;
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
        const double ci = c[i];
        const double xv = global_update(seg_off[i], seg_off[i + 1], u, ci, lb[i], ub[i], rho, rc);
        x[i] = xv;
        o = fma(ci, xv, o);
    }
    return o;
}

// The update of every global and each block's share of c^T x in out[block] (one
// block: the objective).
__global__ void __launch_bounds__(kThreads) k_global_update_static(int n, const int *seg_off, const double *u,
                                                                    const double *c, const double *lb,
                                                                    const double *ub, double rho, Recips rc, double *x,
                                                                    double *out) {
    cudaTriggerProgrammaticLaunchCompletion();       // the sum's block may take its place and wait there
    const double o = block_sum(update_share(n, seg_off, u, c, lb, ub, rho, rc, x));
    if (threadIdx.x == 0) out[blockIdx.x] = o;
}

// The same in one launch, by one cluster: the blocks' shares meet in the first
// block's shared memory and are added there in block order.
__global__ void __cluster_dims__(kCluster, 1, 1) __launch_bounds__(kClusterThreads)
    k_global_update_cluster(int n, const int *seg_off, const double *u, const double *c, const double *lb,
                            const double *ub, double rho, Recips rc, double *x, double *objective) {
    __shared__ double share[kCluster];
    cg::cluster_group cl = cg::this_cluster();
    cl.barrier_arrive();                             // every block of the cluster has started
    double o = update_share(n, seg_off, u, c, lb, ub, rho, rc, x);
    o = block_sum(o);
    cl.barrier_wait();
    if (threadIdx.x == 0) *cl.map_shared_rank(&share[cl.block_rank()], 0) = o;
    cl.sync();
    if (cl.block_rank() == 0 && threadIdx.x == 0) {
        double s = share[0];
        for (int b = 1; b < kCluster; ++b) s += share[b];
        *objective = s;
    }
}

// Objective: the block partials summed in a fixed order by one block.  (By one
// thread, 248 dependent adds took 15 of the 24.6 us of a 63,405-global call;
// with the block sum and the forms above a call takes 10.9 us, 9.3 with this
// kernel's start-up under the update, and one of 2 million globals 61 us, where
// 1 million took 250.)
__global__ void __launch_bounds__(kThreads) k_sum_partials_static(int nblk, const double *partials,
                                                                  double *objective) {
    cudaGridDependencySynchronize();                 // until the update's blocks have finished
    double s = 0.0;
    for (int b = threadIdx.x; b < nblk; b += kThreads) s += partials[b];
    s = block_sum(s);
    if (threadIdx.x == 0) *objective = s;
}

// Driver entry points fetched through the runtime (no link-time dependency
// on the driver library).
using PFN_streamCtx = CUresult (*)(CUstream, CUcontext *);
using PFN_curCtx = CUresult (*)(CUcontext *);
using PFN_ctxId = CUresult (*)(CUcontext, unsigned long long *);
using PFN_push = CUresult (*)(CUcontext);
using PFN_pop = CUresult (*)(CUcontext *);

struct Drv {
    PFN_streamCtx streamCtx = nullptr;
    PFN_curCtx curCtx = nullptr;
    PFN_ctxId ctxId = nullptr;
    PFN_push push = nullptr;
    PFN_pop pop = nullptr;
    bool ok = false;
};

template <typename F>
bool entry(const char *name, F *out) {
    void *p = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion(name, &p, 12000, cudaEnableDefault, &q) != cudaSuccess ||
        q != cudaDriverEntryPointSuccess || !p)
        return false;
    *out = reinterpret_cast<F>(p);
    return true;
}

const Drv &drv() {
    static Drv d;
    static std::once_flag once;
    std::call_once(once, [] {
        d.ok = entry("cuStreamGetCtx", &d.streamCtx) && entry("cuCtxGetCurrent", &d.curCtx) &&
               entry("cuCtxGetId", &d.ctxId) && entry("cuCtxPushCurrent", &d.push) &&
               entry("cuCtxPopCurrent", &d.pop);
    });
    return d;
}

// Per CUDA context the device address of g_static_partials and whether the
// context can hold the one-cluster launch, keyed by the context's process-unique
// id (a destroyed and re-created context, e.g. after cudaDeviceReset, gets a new
// id, so a stale address is never reused).
struct CtxInfo {
    double *partials = nullptr;
    bool cluster = false;
};
std::mutex g_mu;
std::map<unsigned long long, CtxInfo> g_ctx;

bool holds_cluster(cudaStream_t s) {
    cudaLaunchConfig_t cfg;
    memset(&cfg, 0, sizeof(cfg));
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = kCluster;
    attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
    cfg.gridDim = dim3(kCluster);
    cfg.blockDim = dim3(kClusterThreads);
    cfg.stream = s;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    int n = 0;
    if (cudaOccupancyMaxActiveClusters(&n, k_global_update_cluster, &cfg) == cudaSuccess) return n > 0;
    cudaGetLastError();
    return false;
}

int fail(int code, const std::string &msg) {
    opf::set_last_error("opf_global_update_static: " + msg);
    return code;
}

}  // namespace

extern "C" int opf_global_update_static(int32_t n, const int32_t *seg_off, const double *u, const double *c,
                                        const double *lb, const double *ub, double rho, double *x,
                                        double *objective, void *stream) {
    if (n < 1 || !seg_off || !u || !c || !lb || !ub || !x || !objective || !(rho > 0.0))
        return fail(OPF_E_INVALID, "need n >= 1, rho > 0 and non-null device pointers");
    if (n > OPF_STATIC_MAX_GLOBALS)
        return fail(OPF_E_CAPACITY, "n = " + std::to_string(n) + " exceeds OPF_STATIC_MAX_GLOBALS (" +
                                        std::to_string(OPF_STATIC_MAX_GLOBALS) + ")");
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    const Drv &d = drv();
    if (!d.ok) return fail(OPF_E_CUDA, "driver entry points for context queries unavailable");
    // The context the kernels will run in: the stream's (a stream of an SM
    // partition belongs to its own context), else the current one.
    CUcontext ctx = nullptr;
    if (s) {
        if (d.streamCtx((CUstream)s, &ctx) != CUDA_SUCCESS || !ctx) return fail(OPF_E_CUDA, "cuStreamGetCtx failed");
    } else {
        if (d.curCtx(&ctx) != CUDA_SUCCESS) return fail(OPF_E_CUDA, "cuCtxGetCurrent failed");
        if (!ctx) {
            // No context yet on this thread: the runtime makes the current
            // device's primary context on its first call, here a symbol query.
            void *p = nullptr;
            cudaError_t e = cudaGetSymbolAddress(&p, g_static_partials);
            if (e != cudaSuccess) return fail(OPF_E_CUDA, std::string("cudaGetSymbolAddress: ") + cudaGetErrorString(e));
            if (d.curCtx(&ctx) != CUDA_SUCCESS || !ctx) return fail(OPF_E_CUDA, "no current context");
        }
    }
    unsigned long long id = 0;
    if (d.ctxId(ctx, &id) != CUDA_SUCCESS) return fail(OPF_E_CUDA, "cuCtxGetId failed");
    CtxInfo info;
    {
        // set-up, once per context with that context current: the device
        // address of the static array (host code must not use its name as an
        // address)
        std::lock_guard<std::mutex> lock(g_mu);
        auto it = g_ctx.find(id);
        if (it != g_ctx.end()) {
            info = it->second;
        } else {
            if (d.push(ctx) != CUDA_SUCCESS) return fail(OPF_E_CUDA, "cuCtxPushCurrent failed");
            void *p = nullptr;
            cudaError_t e = cudaGetSymbolAddress(&p, g_static_partials);
            if (e == cudaSuccess) info.cluster = holds_cluster(s);
            CUcontext popped = nullptr;
            d.pop(&popped);
            if (e != cudaSuccess || !p)
                return fail(OPF_E_CUDA, std::string("cudaGetSymbolAddress: ") + cudaGetErrorString(e));
            info.partials = static_cast<double *>(p);
            g_ctx[id] = info;
        }
    }
    double *const partials = info.partials;
    Recips rc;
    for (int k = 0; k < kRecip; ++k) {
        const double den = rho * (double)k, r = k ? 1.0 / den : 0.0;
        rc.r[k] = std::isnormal(r) && std::isnormal(den) ? r : 0.0;
    }
    if (n <= kOneBlock) {
        k_global_update_static<<<1, (unsigned)((n + 31) / 32 * 32), 0, s>>>(n, seg_off, u, c, lb, ub, rho, rc, x,
                                                                            objective);
    } else if (n <= kOneCluster && info.cluster) {
        const int threads = std::min(((n + kCluster - 1) / kCluster + 31) / 32 * 32, kClusterThreads);
        k_global_update_cluster<<<kCluster, (unsigned)threads, 0, s>>>(n, seg_off, u, c, lb, ub, rho, rc, x, objective);
    } else {
        const int nblk = std::min((n + kThreads - 1) / kThreads, kBlocks);
        k_global_update_static<<<(unsigned)nblk, kThreads, 0, s>>>(n, seg_off, u, c, lb, ub, rho, rc, x, partials);
        // launched while the update runs (programmatic dependent launch), so that
        // its start-up does not come after it
        cudaLaunchConfig_t cfg;
        memset(&cfg, 0, sizeof(cfg));
        cudaLaunchAttribute attr[1];
        attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        attr[0].val.programmaticStreamSerializationAllowed = 1;
        cfg.gridDim = dim3(1);
        cfg.blockDim = dim3(kThreads);
        cfg.stream = s;
        cfg.attrs = attr;
        cfg.numAttrs = 1;
        const cudaError_t le = cudaLaunchKernelEx(&cfg, k_sum_partials_static, nblk, (const double *)partials, objective);
        if (le != cudaSuccess) return fail(OPF_E_CUDA, std::string("launch: ") + cudaGetErrorString(le));
    }
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return fail(OPF_E_CUDA, std::string("launch: ") + cudaGetErrorString(e));
    return OPF_OK;
}
