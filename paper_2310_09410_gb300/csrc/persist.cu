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
// Owner form (OWN, globals with many copies, where a part would read mostly
// other parts' u): every global is updated once, by the CTA that owns it, whose
// copies' u are one run of the exchange buffer, and its x goes out in an
// exchange entry of its own.  Two exchanges per iteration, of one word per slot
// and one per global, instead of one of a word per copy read elsewhere:
//   the owned copies' u polled; -- CTA barrier -- x of the owned globals, a
//   thread each, out; x of the part's globals polled; -- CTA barrier --
//   V per slot, and B and C as above.
// An entry of u is overwritten two iterations later by a CTA that has read, one
// iteration later, the x which its owner computed from it, and one of x by the
// owner after it has read u of every reader from one iteration later.
// 240 blocks of up to 100 slots, 14 copies per global: FP32 3.4 us per iteration
// against 6.5 on the cluster engine (12,000 stores to other CTAs' shared memory
// twice an iteration, each behind a cluster barrier that waits for them), FP64
// 7.4 against 8.7 in the local form.
// Parts that do not fit that form (several slots per thread) are runs of the
// size-sorted order, the slots' data in shared memory, every copy of u read from
// the exchange: k_persist_engine (FP64) by stamped words as above,
// k_persist_slots (FP32) from plain words behind a grid barrier.
// On tested iterations each CTA adds the Sec. III-C sums of its slots in FP64
// and publishes them as stamped words; every CTA sums the P partials in the same
// fixed order and takes the same stopping decision (rank 0 publishes the
// status).  Every wait is bounded: past the limit the CTA records a fault
// in the status and leaves, and the others follow.
//
// What bounds it: FP32, the latency of one iteration (an L2 store and an L2
// load between the CTAs, three CTA barriers, the longest column); FP64, the
// FP64 pipe (a warp instruction occupies a sub-partition's for about 64
// cycles), so the FP64 forms below count FP64 instructions: the clip compares
// integers, the global update is one FMA, a column is one chain over its own
// rows.
// One cluster (CL, instances of the warp engine's size): the stamped words lie
// in the readers' shared memory and the writer stores into them directly
// (distributed shared memory), so an exchange is one remote store.  FP32 keeps
// the warp engine's order of every sum (the iterates are its, bit for bit) with
// the factor rows in registers, columns on one lane each and those of more than
// 32 rows on two.  FP64 (every form) spreads the long columns and rows over lanes.
// us per iteration with a test every 50: 8500 buses FP32 4.4 -> 3.1, FP64 10.7 ->
// 7.3, 123 buses FP64 4.6 -> 2.6 (before: every copy of u through L2 behind a
// grid barrier); one cluster against the warp engine, FP32 13 / 34 / 123 buses
// 1.5 / 1.6 / 2.1 -> 0.93 / 0.93 / 1.06, FP64 13 / 34 buses 2.4 -> 1.8.
#include <cooperative_groups.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cstring>
#include <type_traits>

#include "opf_internal.h"
#include "smem_limit.h"
#include "test_rule.cuh"

namespace opf {
namespace {

namespace cg = cooperative_groups;

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

// <f, v> over the first n rows of a zero-padded column.  FP32: two chains, the
// 16-byte loads of CH row vectors in flight together (vectors past n as zeros,
// which leave the chains as they are).  FP64: rows rounded up to 2, one chain,
// no add at the end.
template <int CH>
__device__ __forceinline__ float dot_fv(const float *__restrict__ f, const float *__restrict__ v, int n) {
    float a0 = 0.0f, a1 = 0.0f;
    for (int r = 0; r < n; r += 4 * CH) {
        float4 a[CH], b[CH];
#pragma unroll
        for (int k = 0; k < CH; ++k) {
            a[k] = b[k] = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
            if (r + 4 * k < n) {
                a[k] = *reinterpret_cast<const float4 *>(f + r + 4 * k);
                b[k] = *reinterpret_cast<const float4 *>(v + r + 4 * k);
            }
        }
#pragma unroll
        for (int k = 0; k < CH; ++k) {
            a0 = fmaf(a[k].x, b[k].x, a0);
            a1 = fmaf(a[k].y, b[k].y, a1);
            a0 = fmaf(a[k].z, b[k].z, a0);
            a1 = fmaf(a[k].w, b[k].w, a1);
        }
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

__device__ __forceinline__ float dot_col(const float *f, const float *v, int n) { return dot_fv<2>(f, v, n); }
__device__ __forceinline__ double dot_col(const double *f, const double *v, int n) { return dot_fv(f, v, n); }

// Rows part, part + lanes, .. of <f, v> (one chain: two chains and their add
// measured slower, 2.24 -> 2.72 us per iteration on the 34-bus feeder).
__device__ __forceinline__ double dot_rows(const double *f, const double *v, int n, int part, int lanes) {
    double acc = 0.0;
#pragma unroll 4
    for (int r = part; r < n; r += lanes) acc = fma(f[r], v[r], acc);
    return acc;
}

// Column stride of a staged factor with npad rows: npad, plus 4 words when
// npad is a multiple of 8, so that the 16-byte column reads of 8 consecutive
// threads (consecutive columns) fall in distinct bank groups.
__host__ __device__ __forceinline__ int fstride(int npad) { return npad + ((npad & 7) == 0 ? 4 : 0); }

// Part ranges: pr[field * (P + 1) + rank].
enum { GR_K = 0, GR_S, GR_J, GR_V, GR_R, GR_L };

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

// The same words in the shared memory of a CTA of the cluster: addr is the
// word's address there (mapa), reads are of the CTA's own.
__device__ __forceinline__ unsigned smem_addr(const void *p) { return (unsigned)__cvta_generic_to_shared(p); }
__device__ __forceinline__ unsigned at_rank(unsigned addr, int rank) {
    unsigned r;
    asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
    return r;
}
__device__ __forceinline__ void sput(unsigned addr, float u, unsigned stamp) {
    const u64 w = ((u64)stamp << 32) | __float_as_uint(u);
    asm volatile("st.relaxed.cluster.shared::cluster.u64 [%0], %1;" ::"r"(addr), "l"(w) : "memory");
}
__device__ __forceinline__ void sput(unsigned addr, double u, unsigned stamp) {
    const u64 s = (u64)stamp << 32;
    const u64 w0 = s | (unsigned)__double2loint(u), w1 = s | (unsigned)__double2hiint(u);
    asm volatile("st.relaxed.cluster.shared::cluster.v2.u64 [%0], {%1, %2};" ::"r"(addr), "l"(w0), "l"(w1) : "memory");
}
__device__ __forceinline__ void sget(unsigned addr, Word1 &w) {
    asm volatile("ld.relaxed.cluster.shared::cta.u64 %0, [%1];" : "=l"(w.a) : "r"(addr) : "memory");
}
__device__ __forceinline__ void sget(unsigned addr, Word2 &w) {
    asm volatile("ld.relaxed.cluster.shared::cta.v2.u64 {%0, %1}, [%2];" : "=l"(w.a), "=l"(w.b) : "r"(addr) : "memory");
}
template <typename T>
using WordOf = typename std::conditional<sizeof(T) == 4, Word1, Word2>::type;

// One more unsuccessful poll; true when the wait has to end: a fault of this
// CTA, or the limit (which makes it one).
__device__ __forceinline__ bool wait_over(unsigned &polls, u64 &t0, volatile int *fault) {
    if ((++polls & 255u) != 0) return false;
    if (t0 == 0) t0 = global_ns();
    if (!*fault && global_ns() - t0 <= kBarrierLimitNs) return false;
    *fault = 1;
    return true;
}

// The values that iteration `stamp` reads of N words, get(j, w) loading word j
// (those with live(j)): the loads of all in flight together, until every
// number is there.
template <typename T, int N, typename Get, typename Live>
__device__ __forceinline__ void wait_words(T (&v)[N], Get get, Live live, unsigned stamp, volatile int *fault) {
    WordOf<T> w[N];
    unsigned polls = 0;
    u64 t0 = 0;
    for (;;) {
#pragma unroll
        for (int j = 0; j < N; ++j)
            if (live(j)) get(j, w[j]);
        bool ok = true;
#pragma unroll
        for (int j = 0; j < N; ++j)
            if (live(j)) ok = ok && xis(w[j], stamp);
        if (ok || wait_over(polls, t0, fault)) break;
    }
#pragma unroll
    for (int j = 0; j < N; ++j) v[j] = live(j) ? xval(w[j]) : T(0);
}

// Sum over the cnt >= 2 copies of a global (entries us .. us + cnt - 1, in
// order) of the u read by iteration `stamp`; copy `own` is the caller's own
// and comes from u.  Up to SEGW copies' loads are in flight together.
template <typename T>
__device__ __forceinline__ T copy_sum(const u64 *X, int us, int cnt, int own, T u, unsigned stamp,
                                      volatile int *fault) {
    constexpr int SEGW = 4;
    T sum = T(0);
    for (int q0 = 0; q0 < cnt; q0 += SEGW) {
        T v[SEGW];
        wait_words<T, SEGW>(v, [&](int j, WordOf<T> &w) { xget(X, us + q0 + j, w); },
                            [&](int j) { return q0 + j < cnt && q0 + j != own; }, stamp, fault);
#pragma unroll
        for (int j = 0; j < SEGW; ++j)
            if (q0 + j < cnt) {
                const T t = q0 + j == own ? u : v[j];
                sum = q0 + j == 0 ? t : sum + t;
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
// CL (one cluster, FP32): the rounding of the warp engine, which ran these
// instances before: v = x + lambda / rho is one FMA.
template <typename T, bool CL>
struct Slot;

template <bool CL>
struct Slot<float, CL> {
    float lam, xs, u;                // lambda - lambda_ref, x_s - x_ref, u
    float r, v, w;                   // x of this iteration, v = x + lambda / rho, lambda / rho (not CL)
    float bt, ct, rn, lo, hi;        // bbar~, c~, 1 / (rho N), bounds - x_ref
    float fr[CL ? 32 : 1];           // CL: the slot's row of the factor (at most 32 columns)
    int frow, trow, fcm, pos;        // F offset of the row, t offset, f | column stride << 8 | mode << 20, V position

    __device__ __forceinline__ void load(const IterArgs<float> &g, int kk, int gi, int cnt) {
        load_global(g, gi, cnt);
        bt = g.bt[kk];
        lam = g.mu[kk];
        xs = g.ds[kk];
        w = CL ? g.inv_rho : __fmul_rn(lam, g.inv_rho);
        u = g.rho * xs - lam;
        r = v = 0.0f;
    }
    __device__ __forceinline__ void load_global(const IterArgs<float> &g, int gi, int cnt) {
        rn = g.recip[cnt];
        ct = g.ct[gi];
        lo = g.lbt[gi];
        hi = g.ubt[gi];
        lam = w = 0.0f;
    }
    __device__ __forceinline__ void global_update(float sigma) {
        float x = (sigma - ct) * rn;
        if (x < lo) x = lo;
        if (x > hi) x = hi;
        r = x;
        v = CL ? fmaf(lam, w, x) : x + w;
    }
    // owner form: x of the slot's global, from its owner
    __device__ __forceinline__ float global_x() const { return r; }
    __device__ __forceinline__ void take_x(float x) {
        r = x;
        v = x + w;
    }
    template <bool PAD4, bool SPLIT>
    __device__ __forceinline__ void local_update(const float *F, const float *tb, const IterArgs<float> &g, int, int) {
        const float *Fr = F + frow, *tt = tb + trow;
        const int f = fcm & 255, cs = (fcm >> 8) & 0xfff;
        float y0 = 0.0f, y1 = 0.0f;      // two chains for latency
        if constexpr (CL) {              // row in registers, the products' loads in flight together
            float4 t[8];
#pragma unroll
            for (int k = 0; k < 8; ++k) {
                t[k] = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
                if (4 * k < f) t[k] = *reinterpret_cast<const float4 *>(tt + 4 * k);
            }
#pragma unroll
            for (int k = 0; k < 8; ++k) {
                y0 += fr[4 * k] * t[k].x;
                y1 += fr[4 * k + 1] * t[k].y;
                y0 += fr[4 * k + 2] * t[k].z;
                y1 += fr[4 * k + 3] * t[k].w;
            }
        } else if constexpr (PAD4) {     // columns and products padded with zeros to a multiple of 4
#pragma unroll 2
            for (int c = 0; c < f; c += 4) {
                const float4 t = *reinterpret_cast<const float4 *>(tt + c);
                const float f0 = Fr[0], f1 = Fr[cs], f2 = Fr[2 * cs], f3 = Fr[3 * cs];
                Fr += 4 * cs;
                y0 += f0 * t.x;
                y1 += f1 * t.y;
                y0 += f2 * t.z;
                y1 += f3 * t.w;
            }
        } else {
            int c = 0;
#pragma unroll 2
            for (; c + 1 < f; c += 2) {
                y0 += Fr[c * cs] * tt[c];
                y1 += Fr[(c + 1) * cs] * tt[c + 1];
            }
            if (c < f) y0 += Fr[c * cs] * tt[c];
        }
        xs = ((fcm >> 20) ? (y0 + y1) : v - (y0 + y1)) + bt;
        const float res = r - xs;
        lam = lam + g.rho * res;
        if constexpr (!CL) w = __fmul_rn(lam, g.inv_rho);
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

template <bool CL>
struct Slot<double, CL> {
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
        load_global(g, gi, cnt);
        lam = g.mu[kk];
        rx = g.rho * g.ds[kk];
        u = rx - lam;
        r = v = 0.0;
    }
    __device__ __forceinline__ void load_global(const IterArgs<double> &g, int gi, int cnt) {
        rn = 1.0 / (double)cnt;
        ct = g.ct[gi] * rn;
        lo = flip(__double_as_longlong(g.rho * g.lbt[gi]));
        hi = flip(__double_as_longlong(g.rho * g.ubt[gi]));
        lam = 0.0;
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
    __device__ __forceinline__ double global_x() const { return r; }
    __device__ __forceinline__ void take_x(double x) {
        r = x;
        v = x + lam;
    }
    // SPLIT: the row on `lanes` lanes (columns part, part + lanes, ..), each of
    // which ends with the whole slot
    template <bool PAD4, bool SPLIT>
    __device__ __forceinline__ void local_update(const double *F, const double *tb, const IterArgs<double> &, int part,
                                                 int lanes) {
        const double *Fr = F + frow, *tt = tb + trow;
        const int f = fcm & 255, cs = (fcm >> 8) & 0xfff;
        double y = part == 0 ? rbt : 0.0;
#pragma unroll 4
        for (int c = part; c < f; c += SPLIT ? lanes : 1) y += Fr[c * cs] * tt[c];
        if constexpr (SPLIT)
            for (int o = 1; o < lanes; o <<= 1) y += __shfl_xor_sync(0xffffffffu, y, o);
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
template <typename S>
__device__ __forceinline__ void place(S &s, const int4 r, int row) {
    const int f = r.w >> 10, npad = (r.w >> 1) & 0x1ff;
    s.frow = r.x + row;
    s.trow = r.z;
    s.fcm = f | (fstride(npad) << 8) | ((r.w & 1) << 20);
    s.pos = r.y + row;
}

// A slot's record in shared memory (k_persist_engine): the fields of Slot that
// the rest cannot be derived from.
struct SlotRec {
    double f[6];                     // lam, rx, rbt, ct, lo, hi (bits)
    int seg, mo;                     // (first copy's entry << 8) | copies; subsystem << 8 | row, own copy's index << 24
};
static_assert(sizeof(SlotRec) == persist_slot_bytes(8), "the layout reserves this much per slot");

__device__ __forceinline__ void pack(SlotRec &q, const Slot<double, false> &s) {
    q.f[0] = s.lam; q.f[1] = s.rx; q.f[2] = s.rbt; q.f[3] = s.ct;
    q.f[4] = __longlong_as_double(s.lo); q.f[5] = __longlong_as_double(s.hi);
}
__device__ __forceinline__ void unpack(Slot<double, false> &s, const SlotRec &q) {
    s.lam = q.f[0]; s.rx = q.f[1]; s.rbt = q.f[2]; s.ct = q.f[3];
    s.lo = __double_as_longlong(q.f[4]); s.hi = __double_as_longlong(q.f[5]);
    s.u = s.rx - s.lam;
}

// Shared-memory areas of the test and the flags (offset lay.off_misc).
struct Misc {
    volatile int *flags;             // [0] fault, [1] stop
    DevStatus *loc;
    double *sum;                     // the six sums over all CTAs
    double (*red)[6];                // per warp
    __device__ __forceinline__ explicit Misc(unsigned char *m)
        : flags(reinterpret_cast<volatile int *>(m)), loc(reinterpret_cast<DevStatus *>(m + 16)),
          sum(reinterpret_cast<double *>(m + 16 + ((sizeof(DevStatus) + 15) & ~15))),
          red(reinterpret_cast<double(*)[6]>(m + 64 + ((sizeof(DevStatus) + 15) & ~15))) {}
};

// The test of iteration `it`, test number nb of the launch: the CTA's six sums
// out as stamped FP64 words, every CTA's taken and added in the same order, the
// decision.  The words of a test are overwritten two tests later, when every
// CTA has published (so read) the one between.  False: leave the loop
// (stopped, or a wait ran out).  CL: the words in every CTA's shared memory at
// tw (2 x P x 6), else in pp.part.
template <bool CL>
__device__ __forceinline__ bool test_iteration(const Misc &m, const PersistPtrs &pp, unsigned tw, double acc[6],
                                               int it, int check_every, int P, unsigned nb, DevStatus *st,
                                               double rho_d) {
    const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5, nw = (int)(blockDim.x >> 5), rank = (int)blockIdx.x;
    const unsigned stamp = (unsigned)it + 1u;
    const int base = (int)(nb & 1u) * P * 6;
    const double mine = cta_sum6(acc, m.red);
    if (tid < 6) {
        if constexpr (CL) {
            for (int r = 0; r < P; ++r) sput(at_rank(tw + 16u * (base + rank * 6 + tid), r), mine, stamp);
        } else {
            xput(pp.part, base + rank * 6 + tid, mine, stamp);
        }
    }
    // one quantity per warp, lane l the CTAs l, l + 32, ..
    for (int q = w; q < 6; q += nw) {
        double v = 0.0;
        for (int r = lane; r < P; r += 32)
        {
            double t[1];
            wait_words<double, 1>(t, [&](int, Word2 &x) {
                if constexpr (CL) sget(tw + 16u * (base + r * 6 + q), x);
                else xget(pp.part, base + r * 6 + q, x);
            }, [](int) { return true; }, stamp, m.flags);
            v += t[0];
        }
        v = warp_sum_d(v);
        if (lane == 0) m.sum[q] = v;
    }
    __syncthreads();
    if (m.flags[0]) return false;
    if (w == 0) {
        DevStatus *loc = m.loc;
        const int since = ((it + 1) % check_every) == 0 ? check_every : ((it + 1) % check_every);
        apply_test_warp(loc, m.sum, rho_d, since);
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

// Factors of the part: one warp per own subsystem, columns re-strided.  The
// local forms keep zero columns up to a multiple of 4 and, where half[i] = hn
// > 0, rows hn and up from the next multiple of 4.
template <typename T, bool LOCAL>
__device__ __forceinline__ void stage_factors(T *F, const IterArgs<T> &g, const int4 *srec, const int *subs,
                                              const int *half, int s0, int ns) {
    for (int i = threadIdx.x >> 5; i < ns; i += blockDim.x >> 5) {
        const int4 r = srec[i];
        const int f = r.w >> 10, npad = (r.w >> 1) & 0x1ff, cs = fstride(npad);
        const int4 q = g.sub2[LOCAL ? subs[s0 + i] : s0 + i];
        const int hn = LOCAL && half ? half[s0 + i] : 0, h4 = (hn + 3) & ~3;
        const T *src = g.F + q.x;
        const int fc = LOCAL ? (f + 3) & ~3 : f;
        for (int e = threadIdx.x & 31; e < fc * npad; e += 32) {
            const int c = e / npad, row = e - c * npad;
            int from = row;                      // row of the packed factor, -1: padding
            if (hn) from = row < hn ? row : row < h4 ? -1 : row - h4 + hn;
            F[r.x + c * cs + row] = c < f && from >= 0 && from < q.y ? src[c * q.y + from] : T(0);
        }
    }
}

// Column products of the one-cluster FP32 form in the warp engine's order
// (rows in two chains up to 32 rows, dot_fv; above, in four chains over the
// column or over each of its halves, the rows past a multiple of 4 last in the
// first chain).
__device__ __forceinline__ float dot_rows4(const float *f, const float *v, int n) {
    float a0 = 0.0f, a1 = 0.0f, a2 = 0.0f, a3 = 0.0f;
    const int full = n & ~3;
    for (int r = 0; r < full; r += 16) {
        float4 a[4], b[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            a[k] = b[k] = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
            if (r + 4 * k < full) {
                a[k] = *reinterpret_cast<const float4 *>(f + r + 4 * k);
                b[k] = *reinterpret_cast<const float4 *>(v + r + 4 * k);
            }
        }
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            a0 = fmaf(a[k].x, b[k].x, a0);
            a1 = fmaf(a[k].y, b[k].y, a1);
            a2 = fmaf(a[k].z, b[k].z, a2);
            a3 = fmaf(a[k].w, b[k].w, a3);
        }
    }
    if (full < n) {                       // the padding rows are zeros: they leave the chain as it is
        const float4 a = *reinterpret_cast<const float4 *>(f + full);
        const float4 b = *reinterpret_cast<const float4 *>(v + full);
        a0 = fmaf(a.x, b.x, a0);
        a0 = fmaf(a.y, b.y, a0);
        a0 = fmaf(a.z, b.z, a0);
    }
    return (a0 + a1) + (a2 + a3);
}

// SPLIT (FP64): the longest factor columns on lay.clanes lanes each and the rows
// of the largest subsystems on lay.rlanes, so that the longest one is no longer
// one lane's dependent chain; how many is the plan's choice (pick in api.cpp).
// CL: the CTAs are one thread-block cluster of at most 16; u goes straight into
// the readers' shared memory (stamped words there, no L2 on the way).
// OWN: the owner form.
// TWO: two CTAs per SM (64 registers).
template <typename T, bool CL, bool OWN, bool TWO>
__global__ void __launch_bounds__(kPersistMaxThreads, TWO ? 2 : 1)
k_persist_local(IterArgs<T> g, PersistLayout lay, PersistPtrs pp, T *U, int bar_extra, int n_iters, int check_every,
                DevStatus *st, double rho_d, cudaGraphConditionalHandle cond, int use_cond) {
    constexpr bool SPLIT = sizeof(T) == 8;
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
    const int turn = CL ? 0 : 32 * (((rank & 1) + (2 * rank >= P ? 2 : 0)) % (nthr >> 5));
    const int tid = (int)threadIdx.x >= turn ? (int)threadIdx.x - turn : (int)threadIdx.x - turn + nthr;
    const int *pr = pp.pr;
    auto range = [&](int f, int &a, int &n) { a = pr[f * P1 + rank]; n = pr[f * P1 + rank + 1] - a; };
    int k0, nk, s0, ns, j0, nj, v0, nv, r0, nrem, l0, nl;
    range(GR_K, k0, nk); range(GR_S, s0, ns); range(GR_J, j0, nj); range(GR_V, v0, nv);
    range(GR_R, r0, nrem); range(GR_L, l0, nl);
    T *F = reinterpret_cast<T *>(sm + lay.off_F);
    int4 *srec = reinterpret_cast<int4 *>(sm + lay.off_srec);
    uint4 *list = reinterpret_cast<uint4 *>(sm + lay.off_list);
    int *rem = reinterpret_cast<int *>(sm + lay.off_rem);          // remote entries (CL: destinations of the exports)
    T *ul = reinterpret_cast<T *>(sm + lay.off_ul);                // u of the own slots, the remote entries, a zero
    T *vb = reinterpret_cast<T *>(sm + lay.off_vb);
    T *tb = reinterpret_cast<T *>(sm + lay.off_tb);
    double *xrs = reinterpret_cast<double *>(sm + lay.off_xrs);    // x_ref of each slot's global
    double *lrs = reinterpret_cast<double *>(sm + lay.off_lrs);    // lambda_ref of each slot
    double *cobj = reinterpret_cast<double *>(sm + lay.off_cobj);  // c of the global on its first copy, else 0
    const Misc m(sm + lay.off_misc);
    // CL: stamped words of the remote entries, two buffers of xcap, and of the tests
    constexpr unsigned XB = sizeof(T) == 4 ? 8 : 16;               // bytes per word
    const unsigned xw = smem_addr(sm + lay.off_xw), xbuf = XB * (unsigned)lay.xcap, tw = smem_addr(sm + lay.off_tw);

    stage<int4>(srec, g.srec + s0, ns);
    stage<uint4>(list, pp.list + l0, nl);
    if constexpr (CL) stage<int>(rem, pp.dst + pp.dr[rank], pp.dr[rank + 1] - pp.dr[rank]);
    else stage<int>(rem, pp.rem + r0, nrem);
    for (int i = tid; i < nv; i += nthr) vb[i] = T(0);
    for (int i = tid; i < lay.tcap; i += nthr) tb[i] = T(0);
    if (tid == 0) {
        ul[nk + nrem] = T(0);
        m.flags[0] = 0;
        m.flags[1] = 0;
        *m.loc = *st;
    }
    if constexpr (CL) {
        for (int i = tid; i < 2 * lay.xcap; i += nthr) sput(xw + XB * i, T(0), 0xffffffffu);
        for (int i = tid; i < 12 * P; i += nthr) sput(tw + 16u * i, 0.0, 0xffffffffu);
    }
    __syncthreads();
    stage_factors<T, true>(F, g, srec, pp.sub, CL ? pp.halves : nullptr, s0, ns);
    constexpr int XW = XB / 8;                          // 8-byte words per exchange entry
    u64 *X0 = pp.xu, *X1 = pp.xu + (size_t)XW * L;      // read by even / odd iterations
    // OWN: this CTA's globals and their copies, a global per thread
    T *ow = reinterpret_cast<T *>(sm + lay.off_ow);                // u of the owned globals' copies
    u64 *XG = pp.xu + (size_t)XW * 2 * L;                          // x, two buffers of G entries
    int og0 = 0, nog = 0, oc0 = 0, noc = 0, ofirst = 0, ocnt = 0;
    Slot<T, false> og;
    if constexpr (OWN) {
        og0 = pp.g0[rank];
        nog = pp.g0[rank + 1] - og0;
        oc0 = pp.gfirst[og0];
        noc = pp.gfirst[og0 + nog] - oc0;
        if (tid < nog) {
            ofirst = pp.gfirst[og0 + tid] - oc0;
            ocnt = pp.gfirst[og0 + tid + 1] - oc0 - ofirst;
            og.load_global(g, og0 + tid, ocnt);
            xput(XG, og0 + tid, T(0), 0xffffffffu);
            xput(XG + (size_t)XW * lay.G, og0 + tid, T(0), 0xffffffffu);
        }
    }
    // the thread's slot (SPLIT: the first ones, of the largest subsystems, on
    // lay.rlanes threads each, in warps of their own)
    int ks = tid, rpart = 0, rl = 1;
    if constexpr (SPLIT) {
        const int nb = pp.wide[2 * rank + 1] * lay.rlanes, wide = (nb + 31) & ~31;
        ks = tid < wide ? (tid < nb ? tid / lay.rlanes : nk) : nb / lay.rlanes + tid - wide;
        if (tid < wide) {
            rl = lay.rlanes;
            rpart = tid & (rl - 1);
        }
    }
    const bool have = ks < nk, lead = have && rpart == 0;
    Slot<T, CL> s;
    int seg = 0, out = -1, kk = 0;
    s.fcm = s.frow = s.trow = s.pos = 0;
    if constexpr (CL) __syncthreads();       // the staged factors are read here
    if (have) {
        kk = pp.slot[k0 + ks];
        const int mt = g.cmeta[k0 + ks], gi = g.gk[kk];
        seg = pp.seg[k0 + ks];
        place(s, srec[mt >> 8], mt & 255);
        s.load(g, kk, gi, seg & 255);
        if constexpr (CL && sizeof(T) == 4) {
            const int f4 = ((s.fcm & 255) + 3) & ~3, cs = (s.fcm >> 8) & 0xfff;
#pragma unroll
            for (int c = 0; c < 32; ++c) s.fr[c] = c < f4 ? F[s.frow + c * cs] : 0.0f;
        }
        if (lead) {
            out = CL ? pp.dseg[k0 + ks] : pp.out[k0 + ks];
            xrs[ks] = g.xr[gi];
            lrs[ks] = g.lamr[kk];
            cobj[ks] = g.pk[kk] == (g.segp[kk] >> 8) ? g.c64[gi] : 0.0;
            if constexpr (!OWN) ul[ks] = s.u;
        }
    }
    // CL: the readers of the slot's u, out = first << 8 | count in the list of
    // destinations (rank << 16 | word, made mapped addresses here); the first
    // two in registers
    unsigned da0 = 0, da1 = 0;
    int nd = 0;
    if constexpr (CL) {
        const int n = pp.dr[rank + 1] - pp.dr[rank];
        for (int i = tid; i < n; i += nthr) rem[i] = (int)at_rank(xw + XB * (rem[i] & 0xffff), rem[i] >> 16);
        __syncthreads();
        nd = lead ? out & 255 : 0;
        if (nd > 0) da0 = (unsigned)rem[out >> 8];
        if (nd > 1) da1 = (unsigned)rem[(out >> 8) + 1];
    }
    auto publish = [&](int it) {         // u for iteration `it`
        if constexpr (CL) {
            const unsigned off = (it & 1) ? xbuf : 0u;
            if (nd > 0) sput(da0 + off, s.u, (unsigned)it);
            if (nd > 1) sput(da1 + off, s.u, (unsigned)it);
            for (int i = 2; i < nd; ++i) sput((unsigned)rem[(out >> 8) + i] + off, s.u, (unsigned)it);
        } else {
            if (out >= 0) xput((it & 1) ? X1 : X0, out, s.u, (unsigned)it);
        }
    };
    // the thread's factor column.  FP32 cluster form: those of more than 32
    // rows first, on two lanes each (a lane per half, the second idle when the
    // column is one piece) and in warps of their own.
    constexpr bool PAIRS = CL && sizeof(T) == 4;
    int jcol, part = 0, nbig = 0, cl = 1;
    if constexpr (PAIRS) {
        for (nbig = 0; nbig < nj && g.sub[pp.sub[s0 + (g.citems[j0 + nbig] >> 8)]].y > 32;) ++nbig;
        const int wide = (2 * nbig + 31) & ~31;
        jcol = tid < wide ? (tid < 2 * nbig ? tid >> 1 : nj) : tid - wide + nbig;
        part = tid < wide ? tid & 1 : 0;
    } else {
        jcol = tid;
        if constexpr (SPLIT) {               // the longest columns on lay.clanes lanes
            const int nb = pp.wide[2 * rank] * lay.clanes, wide = (nb + 31) & ~31;
            jcol = tid < wide ? (tid < nb ? tid / lay.clanes : nj) : nb / lay.clanes + tid - wide;
            if (tid < wide) {
                cl = lay.clanes;
                part = tid & (cl - 1);
            }
        }
    }
    const bool big = PAIRS && tid < ((2 * nbig + 31) & ~31);
    const T *Fcol = F, *vcol = vb;
    int ncol = 0, tcol = 0;
    if (jcol < nj) {
        const int itm = g.citems[j0 + jcol], i = itm >> 8;
        const int4 r = srec[i];
        const int npad = (r.w >> 1) & 0x1ff, n = g.sub[pp.sub[s0 + i]].y;
        Fcol = F + r.x + (itm & 255) * fstride(npad);
        vcol = vb + r.y;
        tcol = r.z + (itm & 255);
        ncol = sizeof(T) == 4 ? npad : SPLIT ? n : (n + 1) & ~1;
        if constexpr (CL) {
            const int hn = pp.halves[s0 + i], h4 = (hn + 3) & ~3;
            if (sizeof(T) == 8 && hn) ncol = npad;
            if (big) {
                ncol = hn ? (part ? n - hn : hn) : (part ? 0 : n);
                if (part) { Fcol += h4; vcol += h4; }
            }
        }
    }
    // the first eight copies' places in the u array in registers, later ones in the list
    const int cnt = seg & 255, wmax = __reduce_max_sync(0xffffffffu, cnt);
    const uint4 *lst = list + (seg >> 8);
    uint4 at = make_uint4(0, 0, 0, 0);
    if (!OWN && cnt > 1) at = lst[0];
    bool running = true;
    if constexpr (CL) {
        cg::this_cluster().sync();           // every CTA's words are marked unwritten
        publish(0);
        // (the test hook of the bounded waits: a word that nobody writes)
        if (bar_extra && tid == 0) {
            double t[1];
            wait_words<double, 1>(t, [&](int, Word2 &x) { sget(tw, x); }, [](int) { return true; }, 0u, m.flags);
        }
        __syncthreads();
        running = m.flags[0] == 0;
    } else {
        if (lead && out >= 0) xput(X1, out, T(0), 0xffffffffu);
        if (tid < 12) xput(pp.part, (tid / 6) * P * 6 + rank * 6 + tid % 6, 0.0, 0xffffffffu);
        publish(0);
        running = grid_barrier(pp.sync, (unsigned long long)(P + bar_extra), m.flags);
    }
    unsigned nb = 0;
    constexpr int WAITS = CL ? 1 : 2;        // remote entries of a thread taken together
    // one iteration (CHK: tested); false: leave the loop
    auto iteration = [&](int it, auto tested) -> bool {
        constexpr bool CHK = decltype(tested)::value;
        double acc[6] = {0, 0, 0, 0, 0, 0};
        if constexpr (OWN) {
            // the owned copies' u, their globals' x out, the x of the part's globals
            // in.  (A wait that ran out is acted on after the second barrier: no
            // thread reads the flag while another may still be setting it.)
            const u64 *XU = (it & 1) ? X1 : X0;
            u64 *XX = XG + ((it & 1) ? (size_t)XW * lay.G : 0);
            for (int i0 = tid; i0 < noc; i0 += nthr) {
                T v[1];
                wait_words<T, 1>(v, [&](int, WordOf<T> &w) { xget(XU, oc0 + i0, w); }, [](int) { return true; },
                                 (unsigned)it, m.flags);
                ow[i0] = v[0];
            }
            __syncthreads();
            if (tid < nog) {
                T sigma = T(0);
                for (int q0 = 0; q0 < ocnt; q0 += 8) {       // copy order, eight loads in flight
                    T v[8];
#pragma unroll
                    for (int q = 0; q < 8; ++q) v[q] = q0 + q < ocnt ? ow[ofirst + q0 + q] : T(0);
#pragma unroll
                    for (int q = 0; q < 8; ++q)
                        if (q0 + q < ocnt) sigma += v[q];
                }
                og.global_update(sigma);
                xput(XX, og0 + tid, og.global_x(), (unsigned)it);
            }
            for (int i0 = nthr - 1 - tid; i0 < nrem; i0 += nthr) {
                T v[1];
                wait_words<T, 1>(v, [&](int, WordOf<T> &w) { xget(XX, rem[i0], w); }, [](int) { return true; },
                                 (unsigned)it, m.flags);
                ul[i0] = v[0];
            }
            __syncthreads();
            if (m.flags[0]) return false;
            if (have) {
                s.take_x(ul[seg >> 8]);
                if (lead) vb[s.pos] = s.v;
                if constexpr (CHK) {
                    if (lead) {
                        s.test_global(acc, g, xrs[ks], cobj[ks]);
                        U[(size_t)L + g.pk[kk]] = s.u;
                    }
                }
            }
        } else {
        // remote entries: the threads of the smallest subsystems first (they
        // finish the previous iteration first)
        for (int i0 = nthr - 1 - tid; i0 < nrem; i0 += WAITS * nthr) {
            T v[WAITS];
            auto live = [&](int j) { return j == 0 || i0 + j * nthr < nrem; };
            wait_words<T, WAITS>(v, [&](int j, WordOf<T> &w) {
                const int i = i0 + j * nthr;
                if constexpr (CL) sget(xw + ((it & 1) ? xbuf : 0u) + XB * i, w);
                else xget((it & 1) ? X1 : X0, rem[i], w);
            }, live, (unsigned)it, m.flags);
#pragma unroll
            for (int j = 0; j < WAITS; ++j)
                if (live(j)) ul[nk + i0 + j * nthr] = v[j];
        }
        __syncthreads();
        if (m.flags[0]) return false;       // written in the waits above only, so every thread reads the same
        if (have) {
            T sigma = s.u;
            if (cnt > 1) {
                if constexpr (sizeof(T) == 8) {      // no add past the last copy
                    const T c0 = ul[at.x & 0xffffu], c1 = ul[at.x >> 16], c2 = ul[at.y & 0xffffu], c3 = ul[at.y >> 16];
                    sigma = c0 + c1;
                    if (cnt > 2) sigma += c2;
                    if (cnt > 3) sigma += c3;
                    const unsigned short *l = reinterpret_cast<const unsigned short *>(lst);
#pragma unroll 4
                    for (int q = 4; q < cnt; ++q) sigma += ul[l[q]];
                } else {                             // the places past the last copy hold zeros
                    T c0 = ul[at.x & 0xffffu], c1 = ul[at.x >> 16], c2 = ul[at.y & 0xffffu], c3 = ul[at.y >> 16];
                    T d0 = T(0), d1 = T(0), d2 = T(0), d3 = T(0);
                    if (wmax > 4) {
                        d0 = ul[at.z & 0xffffu]; d1 = ul[at.z >> 16]; d2 = ul[at.w & 0xffffu]; d3 = ul[at.w >> 16];
                    }
                    if constexpr (CL) {              // four chains
                        c0 += d0; c1 += d1; c2 += d2; c3 += d3;
                        for (int q = 8; q < cnt; q += 8) {
                            const uint4 l = lst[q >> 3];
                            c0 += ul[l.x & 0xffffu]; c1 += ul[l.x >> 16]; c2 += ul[l.y & 0xffffu]; c3 += ul[l.y >> 16];
                            c0 += ul[l.z & 0xffffu]; c1 += ul[l.z >> 16]; c2 += ul[l.w & 0xffffu]; c3 += ul[l.w >> 16];
                        }
                        sigma = (c0 + c1) + (c2 + c3);
                    } else {                         // copy order
                        sigma = ((((((c0 + c1) + c2) + c3) + d0) + d1) + d2) + d3;
                        for (int q = 8; q < cnt; q += 8) {
                            const uint4 l = lst[q >> 3];
                            sigma += ul[l.x & 0xffffu]; sigma += ul[l.x >> 16];
                            sigma += ul[l.y & 0xffffu]; sigma += ul[l.y >> 16];
                            sigma += ul[l.z & 0xffffu]; sigma += ul[l.z >> 16];
                            sigma += ul[l.w & 0xffffu]; sigma += ul[l.w >> 16];
                        }
                    }
                }
            }
            s.global_update(sigma);
            if (lead) vb[s.pos] = s.v;
            if constexpr (CHK) {
                if (lead) {
                    s.test_global(acc, g, xrs[ks], cobj[ks]);
                    U[(size_t)L + g.pk[kk]] = s.u;      // the u behind this global update, for the solution
                }
            }
        }
        }
        __syncthreads();
        if constexpr (SPLIT) {
            T a = T(0);
            if (jcol < nj) a = dot_rows(Fcol, vcol, ncol, part, cl);
            for (int o = 1; o < cl; o <<= 1) a += __shfl_xor_sync(0xffffffffu, a, o);
            if (jcol < nj && part == 0) tb[tcol] = a;
        } else if (big) {
            if constexpr (PAIRS) {
                const float t0 = dot_rows4(Fcol, vcol, ncol), t1 = __shfl_xor_sync(0xffffffffu, t0, 1);
                if (jcol < nj && part == 0) tb[tcol] = t0 + t1;
            }
        } else if (jcol < nj) {
            if constexpr (PAIRS) tb[tcol] = dot_fv<4>(Fcol, vcol, ncol);
            else tb[tcol] = dot_col(Fcol, vcol, ncol);
        }
        __syncthreads();
        if (have || SPLIT) {
            const T old = s.state();
            s.template local_update<true, SPLIT>(F, tb, g, rpart, rl);
            if (lead) {
                publish(it + 1);
                if constexpr (!OWN) ul[ks] = s.u;
                if constexpr (CHK) {
                    s.test_slot(acc, g, old, xrs[ks], lrs[ks]);
                    U[g.pk[kk]] = s.u;
                }
            }
        }
        if constexpr (CHK) return test_iteration<CL>(m, pp, tw, acc, it, check_every, P, nb++, st, rho_d);
        return true;
    };
    for (int it = 0; it < n_iters && running; ++it) {
        if (((it + 1) % check_every) == 0 || it == n_iters - 1) running = iteration(it, std::true_type{});
        else running = iteration(it, std::false_type{});
    }
    if (lead) s.save(g, kk);
    if constexpr (CL) cg::this_cluster().sync();         // no CTA leaves while others may write to its words
    leave(m, st, cond, use_cond);
}

// FP64, several slots per thread.
__global__ void __launch_bounds__(kPersistMaxThreads, 2)
k_persist_engine(IterArgs<double> g, PersistLayout lay, PersistPtrs pp, double *U, int bar_extra, int n_iters,
                 int check_every, DevStatus *st, double rho_d, cudaGraphConditionalHandle cond, int use_cond) {
    using T = double;
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
    SlotRec *slots = reinterpret_cast<SlotRec *>(sm + lay.off_slots);
    T *rb = reinterpret_cast<T *>(sm + lay.off_r);                 // rho x of the slots
    T *rns = reinterpret_cast<T *>(sm + lay.off_rn);               // 1 / N by copy count N
    T *vb = reinterpret_cast<T *>(sm + lay.off_vb);
    T *tb = reinterpret_cast<T *>(sm + lay.off_tb);
    double *xrs = reinterpret_cast<double *>(sm + lay.off_xrs);
    double *lrs = reinterpret_cast<double *>(sm + lay.off_lrs);
    double *cobj = reinterpret_cast<double *>(sm + lay.off_cobj);
    const Misc m(sm + lay.off_misc);

    stage<int4>(srec, g.srec + s0, ns);
    stage<int>(items, g.citems + j0, nj);
    for (int i = tid; i < nv; i += nthr) vb[i] = T(0);
    for (int i = tid; i < 256; i += nthr) rns[i] = i ? 1.0 / (double)i : 0.0;
    if (tid == 0) {
        m.flags[0] = 0;
        m.flags[1] = 0;
        *m.loc = *st;
    }
    __syncthreads();
    stage_factors<T, false>(F, g, srec, nullptr, nullptr, s0, ns);
    constexpr int XW = 2;
    u64 *X0 = pp.xu, *X1 = pp.xu + (size_t)XW * L;
    for (int k = tid; k < nk; k += nthr) {
        const int kk = k0 + k, gi = g.gk[kk], mt = g.cmeta[kk], seg = g.segp[kk], own = g.pk[kk] - (seg >> 8);
        Slot<T, false> s;
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
    auto fetch = [&](Slot<T, false> &s, int k, int &seg, int &own) {
        const SlotRec q = slots[k];
        seg = q.seg;
        own = (int)((unsigned)q.mo >> 24);
        place(s, srec[(q.mo & 0xffffff) >> 8], q.mo & 255);
        unpack(s, q);
        s.rn = rns[q.seg & 255];
        s.r = rb[k];
        s.v = vb[s.pos];
    };
    if (tid < 12) xput(pp.part, (tid / 6) * P * 6 + rank * 6 + tid % 6, 0.0, 0xffffffffu);
    bool running = grid_barrier(pp.sync, (unsigned long long)(P + bar_extra), m.flags);
    unsigned nb = 0;
    auto iteration = [&](int it, auto tested) -> bool {
        constexpr bool CHK = decltype(tested)::value;
        const u64 *Xin = (it & 1) ? X1 : X0;
        u64 *Xout = (it & 1) ? X0 : X1;
        double acc[6] = {0, 0, 0, 0, 0, 0};
        Slot<T, false> s;
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
            tb[j] = dot_col(F + r.x + (itm & 255) * fstride(npad), vb + r.y, npad);
        }
        __syncthreads();
        for (int k = tid; k < nk; k += nthr) {
            fetch(s, k, seg, own);
            const T old = s.state();
            s.template local_update<false, false>(F, tb, g, 0, 1);
            pack(slots[k], s);
            if ((seg & 255) > 1) xput(Xout, (seg >> 8) + own, s.u, (unsigned)it + 1u);
            if constexpr (CHK) {
                s.test_slot(acc, g, old, xrs[k], lrs[k]);
                U[(seg >> 8) + own] = s.u;
            }
        }
        if constexpr (CHK) return test_iteration<false>(m, pp, 0u, acc, it, check_every, P, nb++, st, rho_d);
        return true;
    };
    for (int it = 0; it < n_iters && running; ++it) {
        if (((it + 1) % check_every) == 0 || it == n_iters - 1) running = iteration(it, std::true_type{});
        else running = iteration(it, std::false_type{});
    }
    for (int k = tid; k < nk; k += nthr) {
        Slot<T, false> s;
        int seg, own;
        fetch(s, k, seg, own);
        s.save(g, k0 + k);
    }
    leave(m, st, cond, use_cond);
}

// FP32, several slots per thread: the slots' fields in arrays of shared memory,
// u in two plain buffers of the exchange behind a grid barrier per iteration
// (with every copy read through L2, polling its words costs more than the
// barrier).  The arithmetic of a slot is Slot<float, false>'s.  us per iteration
// with stamped words and a record per slot, and in this form: 123 buses on 2 and
// 4 CTAs 6.5 and 4.3, 4.5 and 3.4; 1000 on 16 8.2, 4.9; 12,000 and 18,000 on two
// CTAs per SM 8.7 and 10.5, 4.5 and 6.2.
__global__ void __launch_bounds__(kPersistMaxThreads, 2)
k_persist_slots(IterArgs<float> g, PersistLayout lay, PersistPtrs pp, float *U, int bar_extra, int n_iters,
                int check_every, DevStatus *st, double rho_d, cudaGraphConditionalHandle cond, int use_cond) {
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
    float *F = reinterpret_cast<float *>(sm + lay.off_F);
    int4 *srec = reinterpret_cast<int4 *>(sm + lay.off_srec);
    int *items = reinterpret_cast<int *>(sm + lay.off_items);
    int *meta = reinterpret_cast<int *>(sm + lay.off_slots);       // subsystem << 8 | row
    int *seg = meta + nk, *pk = seg + nk;                          // copies; the slot's own place among them
    float *lam = reinterpret_cast<float *>(pk + nk), *xs = lam + nk, *bt = xs + nk, *ct = bt + nk, *lo = ct + nk,
          *hi = lo + nk;
    float *rb = reinterpret_cast<float *>(sm + lay.off_r);         // x of the slots
    float *rns = reinterpret_cast<float *>(sm + lay.off_rn);       // 1 / (rho N) by copy count N
    float *vb = reinterpret_cast<float *>(sm + lay.off_vb);        // lambda / rho, from the global update on v
    float *tb = reinterpret_cast<float *>(sm + lay.off_tb);
    double *xrs = reinterpret_cast<double *>(sm + lay.off_xrs);
    double *lrs = reinterpret_cast<double *>(sm + lay.off_lrs);
    double *cobj = reinterpret_cast<double *>(sm + lay.off_cobj);
    const Misc m(sm + lay.off_misc);
    float *Y0 = reinterpret_cast<float *>(pp.xu), *Y1 = Y0 + L;    // u read by even / odd iterations
    const float rho = g.rho, inv_rho = g.inv_rho;

    stage<int4>(srec, g.srec + s0, ns);
    stage<int>(items, g.citems + j0, nj);
    stage<int>(meta, g.cmeta + k0, nk);
    stage<int>(seg, g.segp + k0, nk);
    stage<int>(pk, g.pk + k0, nk);
    stage<float>(lam, g.mu + k0, nk);
    stage<float>(xs, g.ds + k0, nk);
    stage<float>(bt, g.bt + k0, nk);
    stage<float>(rns, g.recip, 256);
    stage<double>(lrs, g.lamr + k0, nk);
    for (int i = tid; i < nv; i += nthr) vb[i] = 0.0f;
    if (tid == 0) {
        m.flags[0] = 0;
        m.flags[1] = 0;
        *m.loc = *st;
    }
    __syncthreads();
    stage_factors<float, false>(F, g, srec, nullptr, nullptr, s0, ns);
    for (int k = tid; k < nk; k += nthr) {
        const int gi = g.gk[k0 + k];
        ct[k] = g.ct[gi];
        lo[k] = g.lbt[gi];
        hi[k] = g.ubt[gi];
        xrs[k] = g.xr[gi];
        cobj[k] = pk[k] == (seg[k] >> 8) ? g.c64[gi] : 0.0;
        vb[srec[meta[k] >> 8].y + (meta[k] & 255)] = __fmul_rn(lam[k], inv_rho);
        __stcg(Y0 + pk[k], rho * xs[k] - lam[k]);
    }
    if (tid < 12) xput(pp.part, (tid / 6) * P * 6 + rank * 6 + tid % 6, 0.0, 0xffffffffu);
    unsigned long long arrivals = (unsigned long long)(P + bar_extra);
    bool running = grid_barrier(pp.sync, arrivals, m.flags);
    unsigned nb = 0;
    auto iteration = [&](int it, auto tested) -> bool {
        constexpr bool CHK = decltype(tested)::value;
        const float *Yin = (it & 1) ? Y1 : Y0;
        float *Yout = (it & 1) ? Y0 : Y1;
        double acc[6] = {0, 0, 0, 0, 0, 0};
        for (int k = tid; k < nk; k += nthr) {
            const int sp = seg[k], us = sp >> 8, cnt = sp & 255;
            float sigma = 0.0f;
            constexpr int SEGW = 8;                    // copies' loads in flight, summed in copy order
            for (int q0 = 0; q0 < cnt; q0 += SEGW) {
                float v[SEGW];
#pragma unroll
                for (int j = 0; j < SEGW; ++j) v[j] = q0 + j < cnt ? __ldcg(Yin + us + q0 + j) : 0.0f;
#pragma unroll
                for (int j = 0; j < SEGW; ++j)
                    if (q0 + j < cnt) sigma += v[j];
            }
            float x = (sigma - ct[k]) * rns[cnt];
            if (x < lo[k]) x = lo[k];
            if (x > hi[k]) x = hi[k];
            const int pos = srec[meta[k] >> 8].y + (meta[k] & 255);
            rb[k] = x;
            vb[pos] = x + vb[pos];
            if constexpr (CHK) {
                const double xd = xrs[k] + (double)x;
                acc[2] += xd * xd;
                acc[5] += cobj[k] * xd;
                U[(size_t)L + pk[k]] = rho * xs[k] - lam[k];       // the u behind this global update, for the solution
            }
        }
        __syncthreads();
        for (int j = tid; j < nj; j += nthr) {
            const int itm = items[j];
            const int4 r = srec[itm >> 8];
            const int npad = (r.w >> 1) & 0x1ff;
            tb[j] = dot_col(F + r.x + (itm & 255) * fstride(npad), vb + r.y, npad);
        }
        __syncthreads();
        for (int k = tid; k < nk; k += nthr) {
            const int4 r = srec[meta[k] >> 8];
            const int row = meta[k] & 255, f = r.w >> 10, cs = fstride((r.w >> 1) & 0x1ff), pos = r.y + row;
            const float *Fr = F + r.x + row, *tt = tb + r.z;
            float y0 = 0.0f, y1 = 0.0f;
            int c = 0;
            for (; c + 1 < f; c += 2) {
                y0 += Fr[c * cs] * tt[c];
                y1 += Fr[(c + 1) * cs] * tt[c + 1];
            }
            if (c < f) y0 += Fr[c * cs] * tt[c];
            const float x = rb[k], old = xs[k];
            const float xm = ((r.w & 1) ? (y0 + y1) : vb[pos] - (y0 + y1)) + bt[k];
            const float res = x - xm;
            const float l = lam[k] + rho * res, u = rho * xm - l;
            xs[k] = xm;
            lam[k] = l;
            vb[pos] = __fmul_rn(l, inv_rho);
            __stcg(Yout + pk[k], u);
            if constexpr (CHK) {
                const double rd = (double)res, dd = (double)xm - (double)old;
                const double xsd = xrs[k] + (double)xm, lamd = lrs[k] + (double)l;
                acc[0] += rd * rd;
                acc[1] += dd * dd;
                acc[3] += xsd * xsd;
                acc[4] += lamd * lamd;
                U[pk[k]] = u;
            }
        }
        if constexpr (CHK) {
            if (!test_iteration<false>(m, pp, 0u, acc, it, check_every, P, nb++, st, rho_d)) return false;
        }
        if (it + 1 == n_iters) return true;
        arrivals += (unsigned long long)P;
        return grid_barrier(pp.sync, arrivals, m.flags);
    };
    for (int it = 0; it < n_iters && running; ++it) {
        if (((it + 1) % check_every) == 0 || it == n_iters - 1) running = iteration(it, std::true_type{});
        else running = iteration(it, std::false_type{});
    }
    for (int k = tid; k < nk; k += nthr) {
        g.mu[k0 + k] = lam[k];
        g.ds[k0 + k] = xs[k];
    }
    leave(m, st, cond, use_cond);
}

// The variant of a layout (kernel attributes, occupancy and launch agree on it).
template <typename T>
const void *persist_fn(const PersistLayout &lay) {
    if (!lay.local) return sizeof(T) == 4 ? (const void *)k_persist_slots : (const void *)k_persist_engine;
    return lay.own       ? (const void *)k_persist_local<T, false, true, false>
           : lay.cluster ? (const void *)k_persist_local<T, true, false, false>
           : lay.two     ? (const void *)k_persist_local<T, false, false, true>
                         : (const void *)k_persist_local<T, false, false, false>;
}

}  // namespace

static void fill_cfg(const PersistLayout &lay, cudaLaunchConfig_t *cfg, cudaLaunchAttribute *attr, cudaStream_t s) {
    memset(cfg, 0, sizeof(*cfg));
    cfg->gridDim = dim3(lay.P, 1, 1);
    cfg->blockDim = dim3(lay.threads, 1, 1);
    cfg->dynamicSmemBytes = lay.bytes;
    cfg->stream = s;
    if (lay.cluster) {
        attr[0].id = cudaLaunchAttributeClusterDimension;
        attr[0].val.clusterDim.x = lay.P;
        attr[0].val.clusterDim.y = 1;
        attr[0].val.clusterDim.z = 1;
    } else {
        attr[0].id = cudaLaunchAttributeCooperative;
        attr[0].val.cooperative = 1;
    }
    cfg->attrs = attr;
    cfg->numAttrs = 1;
}

template <typename T>
int prepare_persist_engine(const PersistLayout &lay) {
    const void *fn = persist_fn<T>(lay);
    if (allow_dynamic_smem(fn, lay.bytes)) return -1;
    if (lay.cluster && cudaFuncSetAttribute(fn, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess) return -1;
    return 0;
}

// CTAs that can be resident on n_sm SMs (a cluster: its own P when the stream's
// SMs hold one, else 0).
template <typename T>
long long persist_resident(const PersistLayout &lay, int n_sm, cudaStream_t s) {
    int n = 0;
    if (lay.cluster) {
        cudaLaunchConfig_t cfg;
        cudaLaunchAttribute attr[1];
        fill_cfg(lay, &cfg, attr, s);
        return cudaOccupancyMaxActiveClusters(&n, persist_fn<T>(lay), &cfg) == cudaSuccess && n > 0 ? lay.P : 0;
    }
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, persist_fn<T>(lay), lay.threads, lay.bytes) != cudaSuccess)
        return 0;
    return (long long)n * n_sm;
}

// Bytes of an exchange buffer: two buffers of n entries.
template <typename T>
size_t persist_exchange_bytes(long long n) { return (size_t)2 * n * (sizeof(T) == 4 ? 8 : 16); }

template <typename T>
int launch_persist_engine(const IterArgs<T> &g, const PersistLayout &lay, const PersistPtrs &pp, T *U,
                          int bar_extra, int n_iters, int check_every, DevStatus *st, double rho,
                          cudaGraphConditionalHandle cond, int use_cond, cudaStream_t s) {
    // the barrier counter starts at 0 in every launch
    if (!lay.cluster && cudaMemsetAsync(pp.sync, 0, sizeof(unsigned long long), s) != cudaSuccess) return -1;
    cudaLaunchConfig_t cfg;
    cudaLaunchAttribute attr[1];
    fill_cfg(lay, &cfg, attr, s);
    IterArgs<T> ga = g;
    PersistLayout la = lay;
    PersistPtrs pa = pp;
    void *args[] = {&ga, &la, &pa, &U, &bar_extra, &n_iters, &check_every, &st, &rho, &cond, &use_cond};
    return cudaLaunchKernelExC(&cfg, persist_fn<T>(lay), args) == cudaSuccess ? 0 : -1;
}

#define OPF_PERSIST_INST(T)                                                                                   \
    template int prepare_persist_engine<T>(const PersistLayout &);                                                        \
    template long long persist_resident<T>(const PersistLayout &, int, cudaStream_t);                       \
    template size_t persist_exchange_bytes<T>(long long);                                                   \
    template int launch_persist_engine<T>(const IterArgs<T> &, const PersistLayout &, const PersistPtrs &,  \
                                          T *, int, int, int, DevStatus *, double,                            \
                                          cudaGraphConditionalHandle, int, cudaStream_t);
OPF_PERSIST_INST(float)
OPF_PERSIST_INST(double)
#undef OPF_PERSIST_INST

}  // namespace opf
