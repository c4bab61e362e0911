// Persistent grid engine: one instance spread over every co-resident CTA of a
// cooperative launch, many iterations of Algorithm 1 per launch.
//
// CTA `rank` owns a set of subsystems.  For the whole launch its factor
// columns, the vectors of its subsystems and the FP64 data of the test stay in
// shared memory.  Only u = rho x_s - lambda crosses CTAs.
//
// Exchange of u.  Every entry of the exchange buffer (L2, global-sorted order,
// each global's copies contiguous, double-buffered by iteration parity) carries
// the number of the iteration that reads it in the same 8-byte word as the
// value (FP64: two such words, one per half).  A reader takes the words with
// relaxed loads until their numbers are the current iteration: the data is its
// own flag, so an iteration needs neither a grid barrier nor a fence, and a
// CTA waits only for the copies of its own globals.  A buffer entry is
// overwritten two iterations later by a CTA that has read, one iteration
// later, the u which the entry's readers computed from it; so no reader can
// miss a value.
//
// k_persist_local: parts of a depth-first order (persist_plan.h), one slot and
// one factor column per thread, the slot's state in registers.  Most copies of
// a part's globals are its own, and those travel through an array of u in
// shared memory; the entries of other parts are fetched into the same array,
// one per thread.  Per iteration:
//   the part's remote entries of u polled into the u array;
//   -- CTA barrier --
//   A. per own slot k: sigma = sum of u over the copies of g(k) in copy order,
//      the global update of Eq. closed_1 for g(k) (recomputed for every copy),
//      V = x + lambda / rho (FP64: rho times that);
//   -- CTA barrier --
//   B. per own factor column: t_c = <F_c, V>;
//   -- CTA barrier --
//   C. per own slot: the local update of Eq. closed_2 (V - F t or F t, plus
//      bbar~), the dual update of Eq. ADMM-3, u = rho x_s - lambda
//      into the u array and, when another part reads it, out with the next
//      iteration's number.
// k_persist_engine: the same iteration for parts that do not fit that form
// (several slots per thread): parts are runs of the size-sorted order, slot
// records in shared memory, and every copy of u is read from the exchange.
// On tested iterations each CTA adds the Sec. III-C sums of its slots in FP64
// and stores them; after a grid barrier every CTA sums the P partials in the
// same fixed order and takes the same stopping decision (rank 0 publishes
// the status).  Every wait is bounded: past the limit the CTA records a fault
// in the status and leaves, and the others follow.
//
// What bounds it: FP32, the latency of one iteration (an L2 store and an L2
// load between the CTAs, three CTA barriers, the longest column); FP64, the
// FP64 pipe (a warp instruction occupies a sub-partition's for about 64
// cycles), so the FP64 forms below count FP64 instructions: the clip compares
// integers, the global update is one FMA, a column is one chain over its own
// rows.
// Measured per iteration with a test every 50, before (every copy of u through
// L2 behind a grid barrier, parts of the size-sorted order, FP64 sums of the
// test by butterflies) and now: 8500 buses FP32 4.23 -> 3.10 us, FP64 10.5 ->
// 7.7 us; 123 buses FP64 4.7 -> 3.04 us.  Of the 8500-bus steps: stamped
// entries alone, all copies through L2, 6.1 us FP32 (every slot polls, and the
// polls fill the L1) and 8.4 us FP64; local parts 3.6 and 8.8 us; the copies'
// places in registers, loops unrolled, long warps of co-resident CTAs on
// different sub-partitions, and the test's sums spread over lanes and warps
// 3.1 and 7.7 us (a test cost some 40 us, now 12).
#include <cuda_runtime.h>

#include <algorithm>
#include <cstring>
#include <type_traits>

#include "opf_internal.h"
#include "test_rule.cuh"

namespace opf {
namespace {

constexpr unsigned long long kBarrierLimitNs = 1000000000ull;   // 1 s

__device__ __forceinline__ unsigned long long ld_acquire_gpu(const unsigned long long *p) {
    unsigned long long v;
    asm volatile("ld.acquire.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
    return v;
}

__device__ __forceinline__ unsigned long long global_ns() {
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

__device__ __forceinline__ double warp_sum_d(double v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// Barrier `target / P` of this launch over all P CTAs (the counter is zeroed
// before the launch and gains P per barrier).  Thread 0 arrives with a
// release add (ordering the CTA's writes, made before the __syncthreads,
// before the arrival) and waits with acquire loads; a wait past the limit
// sets *fault.
__device__ __forceinline__ bool grid_barrier(unsigned long long *bar, unsigned long long target,
                                             volatile int *fault) {
    __syncthreads();
    if (threadIdx.x == 0) {
        asm volatile("red.release.gpu.global.add.u64 [%0], 1;" ::"l"(bar) : "memory");
        if (ld_acquire_gpu(bar) < target) {
            const unsigned long long t0 = global_ns();
            unsigned polls = 0;
            while (ld_acquire_gpu(bar) < target) {
                if ((++polls & 63u) == 0 && global_ns() - t0 > kBarrierLimitNs) {
                    *fault = 1;
                    break;
                }
            }
        }
    }
    __syncthreads();
    return *fault == 0;
}

template <typename T>
__device__ __forceinline__ void stage(T *dst, const T *src, int n) {
    for (int i = threadIdx.x; i < n; i += blockDim.x) dst[i] = src[i];
}

// <f, v> over the first n rows of a zero-padded column (FP32: n rounded up to
// 4 rows, two chains; FP64: to 2 rows, one chain, no add at the end).
__device__ __forceinline__ float dot_fv(const float *__restrict__ f, const float *__restrict__ v, int n) {
    float a0 = 0.0f, a1 = 0.0f;
#pragma unroll 4
    for (int r = 0; r < n; r += 4) {
        const float4 a = *reinterpret_cast<const float4 *>(f + r);
        const float4 b = *reinterpret_cast<const float4 *>(v + r);
        a0 = fmaf(a.x, b.x, a0);
        a1 = fmaf(a.y, b.y, a1);
        a0 = fmaf(a.z, b.z, a0);
        a1 = fmaf(a.w, b.w, a1);
    }
    return a0 + a1;
}

__device__ __forceinline__ double dot_fv(const double *__restrict__ f, const double *__restrict__ v, int n) {
    double acc = 0.0;
#pragma unroll 4
    for (int r = 0; r < n; r += 2) {
        const double2 a = *reinterpret_cast<const double2 *>(f + r);
        const double2 b = *reinterpret_cast<const double2 *>(v + r);
        acc = fma(a.x, b.x, acc);
        acc = fma(a.y, b.y, acc);
    }
    return acc;
}

// Part `part` (0..3) of <f, v> over the zero-padded column: 4-row vectors at
// rows 4 part, 4 part + 16, ...
template <typename T>
__device__ __forceinline__ T dot_fv_part(const T *__restrict__ f, const T *__restrict__ v, int npad, int part);

template <>
__device__ __forceinline__ float dot_fv_part<float>(const float *__restrict__ f, const float *__restrict__ v,
                                                    int npad, int part) {
    float a0 = 0.0f, a1 = 0.0f;
    for (int r = 4 * part; r < npad; r += 16) {
        const float4 a = *reinterpret_cast<const float4 *>(f + r);
        const float4 b = *reinterpret_cast<const float4 *>(v + r);
        a0 = fmaf(a.x, b.x, a0);
        a1 = fmaf(a.y, b.y, a1);
        a0 = fmaf(a.z, b.z, a0);
        a1 = fmaf(a.w, b.w, a1);
    }
    return a0 + a1;
}

template <>
__device__ __forceinline__ double dot_fv_part<double>(const double *__restrict__ f, const double *__restrict__ v,
                                                      int npad, int part) {
    double a0 = 0.0, a1 = 0.0;
    for (int r = 4 * part; r < npad; r += 16) {
        const double2 a = *reinterpret_cast<const double2 *>(f + r);
        const double2 b = *reinterpret_cast<const double2 *>(v + r);
        const double2 c = *reinterpret_cast<const double2 *>(f + r + 2);
        const double2 d = *reinterpret_cast<const double2 *>(v + r + 2);
        a0 = fma(a.x, b.x, a0);
        a1 = fma(a.y, b.y, a1);
        a0 = fma(c.x, d.x, a0);
        a1 = fma(c.y, d.y, a1);
    }
    return a0 + a1;
}

// Column stride of a staged factor with npad rows: npad, plus 4 words when
// npad is a multiple of 8, so that the 16-byte column reads of 8 consecutive
// threads (consecutive columns) fall in distinct bank groups.
__host__ __device__ __forceinline__ int fstride(int npad) { return npad + ((npad & 7) == 0 ? 4 : 0); }

// Part ranges: pr[field * (P + 1) + rank].
enum { GR_K = 0, GR_S, GR_J, GR_F, GR_V, GR_R, GR_L, GR_NFIELDS };

// ---- exchange entries: value and iteration number in one word
using u64 = unsigned long long;

struct Word1 { u64 a; };
struct Word2 { u64 a, b; };

__device__ __forceinline__ void xput(u64 *X, int i, float u, unsigned stamp) {
    const u64 w = ((u64)stamp << 32) | __float_as_uint(u);
    asm volatile("st.relaxed.gpu.global.u64 [%0], %1;" ::"l"(X + i), "l"(w) : "memory");
}
__device__ __forceinline__ void xput(u64 *X, int i, double u, unsigned stamp) {
    const u64 s = (u64)stamp << 32;
    const u64 w0 = s | (unsigned)__double2loint(u), w1 = s | (unsigned)__double2hiint(u);
    asm volatile("st.relaxed.gpu.global.v2.u64 [%0], {%1, %2};" ::"l"(X + 2 * (size_t)i), "l"(w0), "l"(w1) : "memory");
}
__device__ __forceinline__ void xget(const u64 *X, int i, Word1 &w) {
    asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(w.a) : "l"(X + i) : "memory");
}
__device__ __forceinline__ void xget(const u64 *X, int i, Word2 &w) {
    asm volatile("ld.relaxed.gpu.global.v2.u64 {%0, %1}, [%2];" : "=l"(w.a), "=l"(w.b) : "l"(X + 2 * (size_t)i) : "memory");
}
__device__ __forceinline__ bool xis(const Word1 &w, unsigned stamp) { return (unsigned)(w.a >> 32) == stamp; }
__device__ __forceinline__ bool xis(const Word2 &w, unsigned stamp) {
    return (unsigned)(w.a >> 32) == stamp && (unsigned)(w.b >> 32) == stamp;
}
__device__ __forceinline__ float xval(const Word1 &w) { return __uint_as_float((unsigned)w.a); }
__device__ __forceinline__ double xval(const Word2 &w) { return __hiloint2double((int)(unsigned)w.b, (int)(unsigned)w.a); }

// One more unsuccessful poll; true when the wait has to end: a fault of this
// CTA, or the limit (which makes it one).
__device__ __forceinline__ bool wait_over(unsigned &polls, u64 &t0, volatile int *fault) {
    if ((++polls & 255u) != 0) return false;
    if (t0 == 0) t0 = global_ns();
    if (!*fault && global_ns() - t0 <= kBarrierLimitNs) return false;
    *fault = 1;
    return true;
}

// The u of entry i that iteration `stamp` reads.
template <typename T>
__device__ __forceinline__ T xwait(const u64 *X, int i, unsigned stamp, volatile int *fault) {
    typename std::conditional<sizeof(T) == 4, Word1, Word2>::type w;
    unsigned polls = 0;
    u64 t0 = 0;
    for (;;) {
        xget(X, i, w);
        if (xis(w, stamp) || wait_over(polls, t0, fault)) break;
    }
    return xval(w);
}

// Sum over the cnt >= 2 copies of a global (entries us .. us + cnt - 1, in
// order) of the u read by iteration `stamp`; copy `own` is the caller's own
// and comes from u.  Up to SEGW copies' loads are in flight together.
template <typename T>
__device__ __forceinline__ T copy_sum(const u64 *X, int us, int cnt, int own, T u, unsigned stamp,
                                      volatile int *fault) {
    using W = typename std::conditional<sizeof(T) == 4, Word1, Word2>::type;
    constexpr int SEGW = 4;
    T sum = T(0);
    for (int q0 = 0; q0 < cnt; q0 += SEGW) {
        W w[SEGW];
        unsigned polls = 0;
        u64 t0 = 0;
        for (;;) {
#pragma unroll
            for (int j = 0; j < SEGW; ++j)
                if (q0 + j < cnt && q0 + j != own) xget(X, us + q0 + j, w[j]);
            bool ok = true;
#pragma unroll
            for (int j = 0; j < SEGW; ++j)
                if (q0 + j < cnt && q0 + j != own) ok = ok && xis(w[j], stamp);
            if (ok || wait_over(polls, t0, fault)) break;
        }
#pragma unroll
        for (int j = 0; j < SEGW; ++j)
            if (q0 + j < cnt) {
                const T v = q0 + j == own ? u : xval(w[j]);
                sum = q0 + j == 0 ? v : sum + v;
            }
    }
    return sum;
}

// The iteration of one slot, by precision.
//   FP32: in the units of x; these forms and their order are the iterates'
//   rounding (over the 15,000 iterations of a loose solve of the 8500-bus
//   feeder another order moves x by 2e-5), so they stay as they are.
//   FP64: in units of rho, V = rho x + lambda, rho x_s = V - y or y plus
//   rho bbar~ (y starts at it), lambda = V - rho x_s, u = rho x_s - lambda: 8
//   FP64 instructions fewer per slot than the FP32 forms.  The global update
//   is one FMA with c~ / N, and the clip compares order-preserving integers (a
//   double's bits, the lower 63 flipped when negative): an FP64 compare costs
//   as much as an FP64 FMA.  NaN stays NaN.
template <typename T>
struct Slot;

template <>
struct Slot<float> {
    float lam, xs, u;                // lambda - lambda_ref, x_s - x_ref, u
    float r, v, w;                   // x of this iteration, v = x + lambda / rho, lambda / rho
    float bt, ct, rn, lo, hi;        // bbar~, c~, 1 / (rho N), bounds - x_ref
    int frow, trow, fcm, pos;        // F offset of the row, t offset, f | column stride << 8 | mode << 20, V position

    __device__ __forceinline__ void load(const IterArgs<float> &g, int kk, int gi, int cnt) {
        bt = g.bt[kk];
        rn = g.recip[cnt];
        ct = g.ct[gi];
        lo = g.lbt[gi];
        hi = g.ubt[gi];
        lam = g.mu[kk];
        xs = g.ds[kk];
        w = __fmul_rn(lam, g.inv_rho);
        u = g.rho * xs - lam;
        r = v = 0.0f;
    }
    __device__ __forceinline__ void global_update(float sigma) {
        float x = (sigma - ct) * rn;
        if (x < lo) x = lo;
        if (x > hi) x = hi;
        r = x;
        v = x + w;
    }
    __device__ __forceinline__ void local_update(const float *F, const float *tb, const IterArgs<float> &g) {
        const float *Fr = F + frow, *tt = tb + trow;
        const int f = fcm & 255, cs = (fcm >> 8) & 0xfff;
        float y0 = 0.0f, y1 = 0.0f;      // two chains for latency
        int c = 0;
#pragma unroll 2
        for (; c + 1 < f; c += 2) {
            y0 += Fr[c * cs] * tt[c];
            y1 += Fr[(c + 1) * cs] * tt[c + 1];
        }
        if (c < f) y0 += Fr[c * cs] * tt[c];
        xs = ((fcm >> 20) ? (y0 + y1) : v - (y0 + y1)) + bt;
        const float res = r - xs;
        lam = lam + g.rho * res;
        w = __fmul_rn(lam, g.inv_rho);
        u = g.rho * xs - lam;
    }
    __device__ __forceinline__ float state() const { return xs; }
    // Sec. III-C terms: of the global x (acc 2, 5) and of the slot (acc 0, 1, 3, 4).
    __device__ __forceinline__ void test_global(double acc[6], const IterArgs<float> &, double xr, double c) const {
        const double xd = xr + (double)r;
        acc[2] += xd * xd;
        acc[5] += c * xd;
    }
    __device__ __forceinline__ void test_slot(double acc[6], const IterArgs<float> &, float old, double xr,
                                              double lr) const {
        const double res = (double)(r - xs), dd = (double)xs - (double)old;
        const double xsd = xr + (double)xs, lamd = lr + (double)lam;
        acc[0] += res * res;
        acc[1] += dd * dd;
        acc[3] += xsd * xsd;
        acc[4] += lamd * lamd;
    }
    __device__ __forceinline__ void save(const IterArgs<float> &g, int kk) const {
        g.mu[kk] = lam;
        g.ds[kk] = xs;
    }
};

template <>
struct Slot<double> {
    double lam, rx, u;               // lambda - lambda_ref, rho (x_s - x_ref), u
    double r, v;                     // rho x of this iteration, V = r + lam
    double rbt, ct, rn;              // +-rho bbar~ (mode 1 / 0), c~ / N, 1 / N
    long long lo, hi;                // rho (bounds - x_ref), order-preserving
    int frow, trow, fcm, pos;

    static __device__ __forceinline__ long long flip(long long b) {
        return b ^ ((b >> 63) & 0x7fffffffffffffffll);
    }
    __device__ __forceinline__ void load(const IterArgs<double> &g, int kk, int gi, int cnt) {
        const double rbar = g.rho * g.bt[kk];
        rbt = (fcm >> 20) ? rbar : -rbar;
        rn = 1.0 / (double)cnt;
        ct = g.ct[gi] * rn;
        lo = flip(__double_as_longlong(g.rho * g.lbt[gi]));
        hi = flip(__double_as_longlong(g.rho * g.ubt[gi]));
        lam = g.mu[kk];
        rx = g.rho * g.ds[kk];
        u = rx - lam;
        r = v = 0.0;
    }
    __device__ __forceinline__ void global_update(double sigma) {
        r = fma(sigma, rn, -ct);
        const long long b = __double_as_longlong(r);
        if (((u64)b << 1) <= 0xffe0000000000000ull) {        // not NaN
            long long k = flip(b);
            k = k < lo ? lo : k;
            k = k > hi ? hi : k;
            r = __longlong_as_double(flip(k));
        }
        v = r + lam;
    }
    __device__ __forceinline__ void local_update(const double *F, const double *tb, const IterArgs<double> &) {
        const double *Fr = F + frow, *tt = tb + trow;
        const int f = fcm & 255, cs = (fcm >> 8) & 0xfff;
        double y = rbt;
#pragma unroll 4
        for (int c = 0; c < f; ++c) y += Fr[c * cs] * tt[c];
        rx = (fcm >> 20) ? y : v - y;
        lam = v - rx;
        u = rx - lam;
    }
    __device__ __forceinline__ double state() const { return rx; }
    __device__ __forceinline__ void test_global(double acc[6], const IterArgs<double> &g, double xr, double c) const {
        const double xd = xr + r * g.inv_rho;
        acc[2] += xd * xd;
        acc[5] += c * xd;
    }
    __device__ __forceinline__ void test_slot(double acc[6], const IterArgs<double> &g, double old, double xr,
                                              double lr) const {
        const double res = (r - rx) * g.inv_rho, dd = (rx - old) * g.inv_rho;
        const double xsd = xr + rx * g.inv_rho, lamd = lr + lam;
        acc[0] += res * res;
        acc[1] += dd * dd;
        acc[3] += xsd * xsd;
        acc[4] += lamd * lamd;
    }
    __device__ __forceinline__ void save(const IterArgs<double> &g, int kk) const {
        g.mu[kk] = lam;
        g.ds[kk] = rx * g.inv_rho;
    }
};

// Geometry of a slot from its part's subsystem record r and its row.
template <typename T>
__device__ __forceinline__ void place(Slot<T> &s, const int4 r, int row) {
    const int f = r.w >> 10, npad = (r.w >> 1) & 0x1ff;
    s.frow = r.x + row;
    s.trow = r.z;
    s.fcm = f | (fstride(npad) << 8) | ((r.w & 1) << 20);
    s.pos = r.y + row;
}

// A slot's record in shared memory (k_persist_engine): the fields of Slot that
// the rest cannot be derived from.
template <typename T>
struct SlotRec {
    T f[6];                          // FP32: lam, xs, bt, ct, lo, hi; FP64: lam, rx, rbt, ct, lo, hi (bits)
    int seg, mo;                     // (first copy's entry << 8) | copies; subsystem << 8 | row, own copy's index << 24
};
static_assert(sizeof(SlotRec<float>) == persist_slot_bytes(4) && sizeof(SlotRec<double>) == persist_slot_bytes(8),
              "the layout reserves this much per slot");

__device__ __forceinline__ void pack(SlotRec<float> &q, const Slot<float> &s) {
    q.f[0] = s.lam; q.f[1] = s.xs; q.f[2] = s.bt; q.f[3] = s.ct; q.f[4] = s.lo; q.f[5] = s.hi;
}
__device__ __forceinline__ void pack(SlotRec<double> &q, const Slot<double> &s) {
    q.f[0] = s.lam; q.f[1] = s.rx; q.f[2] = s.rbt; q.f[3] = s.ct;
    q.f[4] = __longlong_as_double(s.lo); q.f[5] = __longlong_as_double(s.hi);
}
__device__ __forceinline__ void unpack(Slot<float> &s, const SlotRec<float> &q, const IterArgs<float> &g) {
    s.lam = q.f[0]; s.xs = q.f[1]; s.bt = q.f[2]; s.ct = q.f[3]; s.lo = q.f[4]; s.hi = q.f[5];
    s.w = __fmul_rn(s.lam, g.inv_rho);
    s.u = g.rho * s.xs - s.lam;
}
__device__ __forceinline__ void unpack(Slot<double> &s, const SlotRec<double> &q, const IterArgs<double> &) {
    s.lam = q.f[0]; s.rx = q.f[1]; s.rbt = q.f[2]; s.ct = q.f[3];
    s.lo = __double_as_longlong(q.f[4]); s.hi = __double_as_longlong(q.f[5]);
    s.u = s.rx - s.lam;
}

// Shared-memory areas of the test and the flags (offset lay.off_misc).
struct Misc {
    volatile int *flags;             // [0] fault, [1] stop
    DevStatus *loc;
    double (*red)[6];
    __device__ __forceinline__ explicit Misc(unsigned char *m)
        : flags(reinterpret_cast<volatile int *>(m)), loc(reinterpret_cast<DevStatus *>(m + 16)),
          red(reinterpret_cast<double(*)[6]>(m + 16 + ((sizeof(DevStatus) + 15) & ~15))) {}
};

// The test of iteration `it`: the CTA's sums out, grid barrier number nb, the
// P partials summed, the decision.  False: leave the loop (stopped or fault).
__device__ __forceinline__ bool test_iteration(const Misc &m, const PersistPtrs &pp, double acc[6], int it,
                                               int check_every, int P, int bar_extra, unsigned long long nb,
                                               DevStatus *st, double rho_d) {
    const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5, nw = (int)(blockDim.x >> 5), rank = (int)blockIdx.x;
    const double mine = cta_sum6(acc, m.red);
    if (tid < 6) __stcg(pp.part + rank * 6 + tid, mine);
    if (!grid_barrier(pp.sync, nb * (unsigned long long)(P + bar_extra), m.flags)) return false;
    // the partials of one quantity per warp, in the same order in every CTA
    for (int q = w; q < 6; q += nw) {
        double v = 0.0;
        for (int r = lane; r < P; r += 32) v += __ldcg(pp.part + r * 6 + q);
        v = warp_sum_d(v);
        if (lane == 0) m.red[0][q] = v;
    }
    __syncthreads();
    if (w == 0) {
        DevStatus *loc = m.loc;
        const int since = ((it + 1) % check_every) == 0 ? check_every : ((it + 1) % check_every);
        apply_test_warp(loc, m.red[0], rho_d, since);
        if (lane == 0) {
            m.flags[1] = loc->done;
            if (rank == 0) {
                st->iter = loc->iter;
                st->pres = loc->pres;
                st->dres = loc->dres;
                st->eprim = loc->eprim;
                st->edual = loc->edual;
                st->obj = loc->obj;
                st->converged = loc->converged;
                st->numeric = loc->numeric;
                st->done = loc->done;
            }
        }
    }
    __syncthreads();
    return m.flags[1] == 0;
}

__device__ __forceinline__ void leave(const Misc &m, DevStatus *st, cudaGraphConditionalHandle cond, int use_cond) {
    if (threadIdx.x != 0) return;
    if (m.flags[0]) {
        atomicExch(&st->fault, 1);
        atomicExch(&st->done, 1);
    }
    if (use_cond && blockIdx.x == 0) cudaGraphSetConditional(cond, (m.flags[0] || m.flags[1]) ? 0u : 1u);
}

// Factors of the part: one warp per own subsystem, columns re-strided.
template <typename T>
__device__ __forceinline__ void stage_factors(T *F, const IterArgs<T> &g, const int4 *srec, const int *subs, int s0,
                                              int ns) {
    for (int i = threadIdx.x >> 5; i < ns; i += blockDim.x >> 5) {
        const int4 r = srec[i];
        const int f = r.w >> 10, npad = (r.w >> 1) & 0x1ff, cs = fstride(npad);
        const T *src = g.F + g.sub2[subs ? subs[s0 + i] : s0 + i].x;
        for (int e = threadIdx.x & 31; e < f * npad; e += 32) {
            const int c = e / npad;
            F[r.x + c * cs + (e - c * npad)] = src[e];
        }
    }
}

// SPLIT: small CTAs, each factor column on 4 lanes (rows 4 p, 4 p + 16, .. of
// lane p, then a shuffle sum), so the longest column is no longer one lane's
// dependent chain; otherwise one lane per column.
template <typename T, bool SPLIT>
__global__ void __launch_bounds__(kPersistMaxThreads, SPLIT ? 1 : 2)
k_persist_local(IterArgs<T> g, PersistLayout lay, PersistPtrs pp, T *U, int bar_extra, int n_iters, int check_every,
                DevStatus *st, double rho_d, cudaGraphConditionalHandle cond, int use_cond) {
    extern __shared__ __align__(16) unsigned char sm[];
    const int P = lay.P, rank = (int)blockIdx.x, P1 = P + 1, L = lay.L;
    const int nthr = blockDim.x;
    if (st->done) {
        if (use_cond && rank == 0 && threadIdx.x == 0) cudaGraphSetConditional(cond, 0);
        return;
    }
    // A part's first slots and columns are its longest, so work item 0 starts
    // at another warp in CTAs that share an SM (b and b + the number of SMs, or
    // neighbours): their long warps then sit on different sub-partitions.
    const int turn = 32 * (((rank & 1) + (2 * rank >= P ? 2 : 0)) % (nthr >> 5));
    const int tid = (int)threadIdx.x >= turn ? (int)threadIdx.x - turn : (int)threadIdx.x - turn + nthr;
    const int *pr = pp.pr;
    auto range = [&](int f, int &a, int &n) { a = pr[f * P1 + rank]; n = pr[f * P1 + rank + 1] - a; };
    int k0, nk, s0, ns, j0, nj, v0, nv, r0, nrem, l0, nl;
    range(GR_K, k0, nk); range(GR_S, s0, ns); range(GR_J, j0, nj); range(GR_V, v0, nv);
    range(GR_R, r0, nrem); range(GR_L, l0, nl);
    T *F = reinterpret_cast<T *>(sm + lay.off_F);
    int4 *srec = reinterpret_cast<int4 *>(sm + lay.off_srec);
    int *list = reinterpret_cast<int *>(sm + lay.off_list);
    int *rem = reinterpret_cast<int *>(sm + lay.off_rem);
    T *ul = reinterpret_cast<T *>(sm + lay.off_ul);                // u of the own slots, then of the remote entries
    T *vb = reinterpret_cast<T *>(sm + lay.off_vb);
    T *tb = reinterpret_cast<T *>(sm + lay.off_tb);
    double *xrs = reinterpret_cast<double *>(sm + lay.off_xrs);    // x_ref of each slot's global
    double *lrs = reinterpret_cast<double *>(sm + lay.off_lrs);    // lambda_ref of each slot
    double *cobj = reinterpret_cast<double *>(sm + lay.off_cobj);  // c of the global on its first copy, else 0
    const Misc m(sm + lay.off_misc);

    stage<int4>(srec, g.srec + s0, ns);
    stage<int>(list, pp.list + l0, nl);
    stage<int>(rem, pp.rem + r0, nrem);
    for (int i = tid; i < nv; i += nthr) vb[i] = T(0);
    if (tid == 0) {
        m.flags[0] = 0;
        m.flags[1] = 0;
        *m.loc = *st;
    }
    __syncthreads();
    stage_factors<T>(F, g, srec, pp.sub, s0, ns);
    constexpr int XW = sizeof(T) == 4 ? 1 : 2;          // words per exchange entry
    u64 *X0 = pp.xu, *X1 = pp.xu + (size_t)XW * L;      // read by even / odd iterations
    // the thread's slot; its first u out, its entry of iteration 1 marked unwritten
    const bool have = tid < nk;
    Slot<T> s;
    int seg = 0, out = -1, kk = 0;
    if (have) {
        kk = pp.slot[k0 + tid];
        const int mt = g.cmeta[k0 + tid], gi = g.gk[kk];
        seg = pp.seg[k0 + tid];
        out = pp.out[k0 + tid];
        place(s, srec[mt >> 8], mt & 255);
        s.load(g, kk, gi, seg & 255);
        xrs[tid] = g.xr[gi];
        lrs[tid] = g.lamr[kk];
        cobj[tid] = g.pk[kk] == (g.segp[kk] >> 8) ? g.c64[gi] : 0.0;
        ul[tid] = s.u;
        if (out >= 0) {
            xput(X0, out, s.u, 0u);
            xput(X1, out, T(0), 0xffffffffu);
        }
    }
    // the thread's factor column
    const int part4 = SPLIT ? tid & 3 : 0, jcol = SPLIT ? tid >> 2 : tid;
    const T *Fcol = F, *vcol = vb;
    int ncol = 0;
    if (jcol < nj) {
        const int itm = g.citems[j0 + jcol];
        const int4 r = srec[itm >> 8];
        const int npad = (r.w >> 1) & 0x1ff;
        Fcol = F + r.x + (itm & 255) * fstride(npad);
        vcol = vb + r.y;
        ncol = SPLIT || sizeof(T) == 4 ? npad : (g.sub[pp.sub[s0 + (itm >> 8)]].y + 1) & ~1;
    }
    // the first four copies' places in the u array in registers, later ones in the list
    const int cnt = seg & 255, *lst = list + (seg >> 8);
    unsigned at01 = 0, at23 = 0;
    if (cnt > 1) {
        at01 = (unsigned)lst[0] | ((unsigned)lst[1] << 16);
        at23 = (cnt > 2 ? (unsigned)lst[2] : 0u) | ((cnt > 3 ? (unsigned)lst[3] : 0u) << 16);
    }
    unsigned long long nb = 1;
    bool running = grid_barrier(pp.sync, nb * (unsigned long long)(P + bar_extra), m.flags);
    // one iteration (CHK: tested); false: leave the loop
    auto iteration = [&](int it, auto tested) -> bool {
        constexpr bool CHK = decltype(tested)::value;
        const u64 *Xin = (it & 1) ? X1 : X0;
        u64 *Xout = (it & 1) ? X0 : X1;
        double acc[6] = {0, 0, 0, 0, 0, 0};
        // remote entries: the threads of the smallest subsystems first (they
        // finish the previous iteration first)
        for (int i = nthr - 1 - tid; i < nrem; i += nthr) ul[nk + i] = xwait<T>(Xin, rem[i], (unsigned)it, m.flags);
        __syncthreads();
        if (m.flags[0]) return false;       // written in the waits above only, so every thread reads the same
        if (have) {
            T sigma = s.u;
            if (cnt > 1) {
                const T a0 = ul[at01 & 0xffffu], a1 = ul[at01 >> 16], a2 = ul[at23 & 0xffffu], a3 = ul[at23 >> 16];
                sigma = a0 + a1;
                if (cnt > 2) sigma += a2;
                if (cnt > 3) sigma += a3;
#pragma unroll 4
                for (int q = 4; q < cnt; ++q) sigma += ul[lst[q]];
            }
            s.global_update(sigma);
            vb[s.pos] = s.v;
            if constexpr (CHK) {
                s.test_global(acc, g, xrs[tid], cobj[tid]);
                U[(size_t)L + g.pk[kk]] = s.u;      // the u behind this global update, for the solution
            }
        }
        __syncthreads();
        if constexpr (SPLIT) {
            T a = T(0);
            if (jcol < nj) a = dot_fv_part<T>(Fcol, vcol, ncol, part4);
            a += __shfl_xor_sync(0xffffffffu, a, 1);
            a += __shfl_xor_sync(0xffffffffu, a, 2);
            if (jcol < nj && part4 == 0) tb[jcol] = a;
        } else {
            if (jcol < nj) tb[jcol] = dot_fv(Fcol, vcol, ncol);
        }
        __syncthreads();
        if (have) {
            const T old = s.state();
            s.local_update(F, tb, g);
            if (out >= 0) xput(Xout, out, s.u, (unsigned)it + 1u);
            ul[tid] = s.u;
            if constexpr (CHK) {
                s.test_slot(acc, g, old, xrs[tid], lrs[tid]);
                U[g.pk[kk]] = s.u;
            }
        }
        if constexpr (CHK) return test_iteration(m, pp, acc, it, check_every, P, bar_extra, ++nb, st, rho_d);
        return true;
    };
    for (int it = 0; it < n_iters && running; ++it) {
        if (((it + 1) % check_every) == 0 || it == n_iters - 1) running = iteration(it, std::true_type{});
        else running = iteration(it, std::false_type{});
    }
    if (have) s.save(g, kk);
    leave(m, st, cond, use_cond);
}

template <typename T>
__global__ void __launch_bounds__(kPersistMaxThreads, 2)
k_persist_engine(IterArgs<T> g, PersistLayout lay, PersistPtrs pp, T *U, int bar_extra, int n_iters, int check_every,
                 DevStatus *st, double rho_d, cudaGraphConditionalHandle cond, int use_cond) {
    extern __shared__ __align__(16) unsigned char sm[];
    const int P = lay.P, rank = (int)blockIdx.x, P1 = P + 1, L = lay.L;
    const int tid = threadIdx.x, nthr = blockDim.x;
    if (st->done) {
        if (use_cond && rank == 0 && tid == 0) cudaGraphSetConditional(cond, 0);
        return;
    }
    const int *pr = pp.pr;
    auto range = [&](int f, int &a, int &n) { a = pr[f * P1 + rank]; n = pr[f * P1 + rank + 1] - a; };
    int k0, nk, s0, ns, j0, nj, v0, nv;
    range(GR_K, k0, nk); range(GR_S, s0, ns); range(GR_J, j0, nj); range(GR_V, v0, nv);
    T *F = reinterpret_cast<T *>(sm + lay.off_F);
    int4 *srec = reinterpret_cast<int4 *>(sm + lay.off_srec);
    int *items = reinterpret_cast<int *>(sm + lay.off_items);
    SlotRec<T> *slots = reinterpret_cast<SlotRec<T> *>(sm + lay.off_slots);
    T *rb = reinterpret_cast<T *>(sm + lay.off_r);                 // rho x of the slots
    T *rns = reinterpret_cast<T *>(sm + lay.off_rn);               // 1 / (rho N) (FP64: 1 / N) by copy count N
    T *vb = reinterpret_cast<T *>(sm + lay.off_vb);
    T *tb = reinterpret_cast<T *>(sm + lay.off_tb);
    double *xrs = reinterpret_cast<double *>(sm + lay.off_xrs);
    double *lrs = reinterpret_cast<double *>(sm + lay.off_lrs);
    double *cobj = reinterpret_cast<double *>(sm + lay.off_cobj);
    const Misc m(sm + lay.off_misc);

    stage<int4>(srec, g.srec + s0, ns);
    stage<int>(items, g.citems + j0, nj);
    for (int i = tid; i < nv; i += nthr) vb[i] = T(0);
    for (int i = tid; i < 256; i += nthr) rns[i] = sizeof(T) == 4 ? g.recip[i] : i ? (T)(1.0 / (double)i) : T(0);
    if (tid == 0) {
        m.flags[0] = 0;
        m.flags[1] = 0;
        *m.loc = *st;
    }
    __syncthreads();
    stage_factors<T>(F, g, srec, nullptr, s0, ns);
    constexpr int XW = sizeof(T) == 4 ? 1 : 2;
    u64 *X0 = pp.xu, *X1 = pp.xu + (size_t)XW * L;
    for (int k = tid; k < nk; k += nthr) {
        const int kk = k0 + k, gi = g.gk[kk], mt = g.cmeta[kk], seg = g.segp[kk], own = g.pk[kk] - (seg >> 8);
        Slot<T> s;
        place(s, srec[mt >> 8], mt & 255);
        s.load(g, kk, gi, seg & 255);
        pack(slots[k], s);
        slots[k].seg = seg;
        slots[k].mo = (int)((unsigned)mt | ((unsigned)own << 24));
        xrs[k] = g.xr[gi];
        lrs[k] = g.lamr[kk];
        cobj[k] = own == 0 ? g.c64[gi] : 0.0;
        if ((seg & 255) > 1) {
            xput(X0, g.pk[kk], s.u, 0u);
            xput(X1, g.pk[kk], T(0), 0xffffffffu);
        }
    }
    auto fetch = [&](Slot<T> &s, int k, int &seg, int &own) {
        const SlotRec<T> q = slots[k];
        seg = q.seg;
        own = (int)((unsigned)q.mo >> 24);
        place(s, srec[(q.mo & 0xffffff) >> 8], q.mo & 255);
        unpack(s, q, g);
        s.rn = rns[q.seg & 255];
        s.r = rb[k];
        s.v = vb[s.pos];
    };
    unsigned long long nb = 1;
    bool running = grid_barrier(pp.sync, nb * (unsigned long long)(P + bar_extra), m.flags);
    auto iteration = [&](int it, auto tested) -> bool {
        constexpr bool CHK = decltype(tested)::value;
        const u64 *Xin = (it & 1) ? X1 : X0;
        u64 *Xout = (it & 1) ? X0 : X1;
        double acc[6] = {0, 0, 0, 0, 0, 0};
        Slot<T> s;
        int seg, own;
        for (int k = tid; k < nk; k += nthr) {
            fetch(s, k, seg, own);
            const int cnt = seg & 255;
            T sigma = s.u;
            if (cnt > 1) sigma = copy_sum<T>(Xin, seg >> 8, cnt, own, s.u, (unsigned)it, m.flags);
            s.global_update(sigma);
            vb[s.pos] = s.v;
            rb[k] = s.r;
            if constexpr (CHK) {
                s.test_global(acc, g, xrs[k], cobj[k]);
                U[(size_t)L + (seg >> 8) + own] = s.u;
            }
        }
        __syncthreads();
        if (m.flags[0]) return false;       // written in the waits above only, so every thread reads the same
        for (int j = tid; j < nj; j += nthr) {
            const int itm = items[j];
            const int4 r = srec[itm >> 8];
            const int npad = (r.w >> 1) & 0x1ff;
            tb[j] = dot_fv(F + r.x + (itm & 255) * fstride(npad), vb + r.y, npad);
        }
        __syncthreads();
        for (int k = tid; k < nk; k += nthr) {
            fetch(s, k, seg, own);
            const T old = s.state();
            s.local_update(F, tb, g);
            pack(slots[k], s);
            if ((seg & 255) > 1) xput(Xout, (seg >> 8) + own, s.u, (unsigned)it + 1u);
            if constexpr (CHK) {
                s.test_slot(acc, g, old, xrs[k], lrs[k]);
                U[(seg >> 8) + own] = s.u;
            }
        }
        if constexpr (CHK) return test_iteration(m, pp, acc, it, check_every, P, bar_extra, ++nb, st, rho_d);
        return true;
    };
    for (int it = 0; it < n_iters && running; ++it) {
        if (((it + 1) % check_every) == 0 || it == n_iters - 1) running = iteration(it, std::true_type{});
        else running = iteration(it, std::false_type{});
    }
    for (int k = tid; k < nk; k += nthr) {
        Slot<T> s;
        int seg, own;
        fetch(s, k, seg, own);
        s.save(g, k0 + k);
    }
    leave(m, st, cond, use_cond);
}

// The variant of a layout (kernel attributes, occupancy and launch agree on it).
template <typename T>
const void *persist_fn(const PersistLayout &lay) {
    if (!lay.local) return (const void *)k_persist_engine<T>;
    return lay.split ? (const void *)k_persist_local<T, true> : (const void *)k_persist_local<T, false>;
}

}  // namespace

template <typename T>
int prepare_persist_engine(const PersistLayout &lay) {
    return cudaFuncSetAttribute(persist_fn<T>(lay), cudaFuncAttributeMaxDynamicSharedMemorySize, (int)lay.bytes) ==
                   cudaSuccess ? 0 : -1;
}

// CTAs per SM.
template <typename T>
int persist_occupancy(const PersistLayout &lay) {
    int n = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, persist_fn<T>(lay), lay.threads, lay.bytes) != cudaSuccess)
        return 0;
    return n;
}

// Bytes of a plan's exchange buffer: two buffers of L entries.
template <typename T>
size_t persist_exchange_bytes(int L) { return (size_t)2 * L * (sizeof(T) == 4 ? 8 : 16); }

template <typename T>
int launch_persist_engine(const IterArgs<T> &g, const PersistLayout &lay, const PersistPtrs &pp, T *U,
                          int bar_extra, int n_iters, int check_every, DevStatus *st, double rho,
                          cudaGraphConditionalHandle cond, int use_cond, cudaStream_t s) {
    // the barrier counter starts at 0 in every launch
    if (cudaMemsetAsync(pp.sync, 0, sizeof(unsigned long long), s) != cudaSuccess) return -1;
    cudaLaunchConfig_t cfg;
    memset(&cfg, 0, sizeof(cfg));
    cfg.gridDim = dim3(lay.P, 1, 1);
    cfg.blockDim = dim3(lay.threads, 1, 1);
    cfg.dynamicSmemBytes = lay.bytes;
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeCooperative;
    attr[0].val.cooperative = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    IterArgs<T> ga = g;
    PersistLayout la = lay;
    PersistPtrs pa = pp;
    void *args[] = {&ga, &la, &pa, &U, &bar_extra, &n_iters, &check_every, &st, &rho, &cond, &use_cond};
    const cudaError_t e = cudaLaunchKernelExC(&cfg, persist_fn<T>(lay), args);
    return e == cudaSuccess ? 0 : -1;
}

#define OPF_PERSIST_INST(T)                                                                                   \
    template int prepare_persist_engine<T>(const PersistLayout &);                                                        \
    template int persist_occupancy<T>(const PersistLayout &);     template size_t persist_exchange_bytes<T>(int);                                                        \
    template int launch_persist_engine<T>(const IterArgs<T> &, const PersistLayout &, const PersistPtrs &,  \
                                          T *, int, int, int, DevStatus *, double,                            \
                                          cudaGraphConditionalHandle, int, cudaStream_t);
OPF_PERSIST_INST(float)
OPF_PERSIST_INST(double)
#undef OPF_PERSIST_INST

}  // namespace opf
