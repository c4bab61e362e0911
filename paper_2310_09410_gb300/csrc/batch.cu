// Batched ADMM (Algorithm 1) over many instances of one model: every instance
// shares A_s, c and the bounds (so M_s = -Abar_s and its factor F) and has its
// own right-hand side b, hence its own bbar = A_s^+ b.
//
//  k_batch_engine  n_iters iterations of Algorithm 1 for the K instances of
//                  one CTA, all resident: factors, u = rho x_s - lambda and
//                  rho x in shared memory; lambda and bbar~ in tensor memory
//                  (FP32 plans) or streamed from L2 as 16-byte vectors, the
//                  test data from L2.  Per iteration:
//                    G. per (global, instance): Eq. closed_1 as a fixed-order
//                       sum over the global's copies of u, rho x stored into
//                       the copies' slots (a global with one copy and no
//                       bounds needs none: with c~ = 0 its rho x is the u of
//                       its slot);
//                    -- CTA barrier --
//                    L. per warp task: J member subsystems x K instances,
//                       in units of rho (no multiplies): V = rho x_g + lambda
//                       (= rho v), rho x_s = M V + rho bbar~ as one pass over
//                       the factor rows (w_r = <F_r, V>, y += w_r F_r),
//                       lambda <- V - rho x_s (Eq. ADMM-3 with
//                       rho x_g = V - lambda), u = rho x_s - lambda;
//                    -- CTA barrier --
//                  and every check_every iterations the Sec. III-C sums per
//                  instance in FP64 and the test; finished instances freeze.
//  k_bref_*        FP64 re-centring: x_ref = next global update of the FP64
//                  state, lambda_ref = lambda (less delta at unbounded
//                  globals, so that their shifted cost is zero), shifted data
//                  written in the engine layout (the engine iterates on
//                  x_s - x_ref[g] and lambda - lambda_ref, the change of
//                  variables of the single-instance engines).
//  k_bunshift_*    back to the unshifted FP64 state.
//  k_bbar          bbar = A_s^+ b per instance and subsystem (Sec. III-B).
#include <cuda_runtime.h>

#include <cmath>
#include <cstdint>

#include "opf_internal.h"
#include "smem_limit.h"
#include "test_rule.cuh"
#include "tmem.cuh"

namespace opf {

namespace {

template <typename T>
struct Q4 {
    T v[4];
};

__device__ __forceinline__ Q4<float> ld4(const float *p) {
    const float4 t = *reinterpret_cast<const float4 *>(p);
    return {{t.x, t.y, t.z, t.w}};
}
__device__ __forceinline__ Q4<double> ld4(const double *p) {
    const double2 a = *reinterpret_cast<const double2 *>(p);
    const double2 b = *reinterpret_cast<const double2 *>(p + 2);
    return {{a.x, a.y, b.x, b.y}};
}
__device__ __forceinline__ void st4(float *p, const Q4<float> &q) {
    *reinterpret_cast<float4 *>(p) = make_float4(q.v[0], q.v[1], q.v[2], q.v[3]);
}
__device__ __forceinline__ void st4(double *p, const Q4<double> &q) {
    *reinterpret_cast<double2 *>(p) = make_double2(q.v[0], q.v[1]);
    *reinterpret_cast<double2 *>(p + 2) = make_double2(q.v[2], q.v[3]);
}

__device__ __forceinline__ float clampT(float x, float lo, float hi) { return x < lo ? lo : (x > hi ? hi : x); }
// FP64: compared as order-preserving integers (a double's bits, the lower 63
// flipped when negative); an FP64 compare occupies a sub-partition's FP64 pipe
// for about 64 cycles, as an FMA does.  NaN stays NaN.
__device__ __forceinline__ long long ordered(double x) {
    const long long b = __double_as_longlong(x);
    return b ^ ((b >> 63) & 0x7fffffffffffffffll);
}
__device__ __forceinline__ double clampT(double x, double lo, double hi) {
    if (((unsigned long long)__double_as_longlong(x) << 1) > 0xffe0000000000000ull) return x;
    return ordered(x) < ordered(lo) ? lo : (ordered(x) > ordered(hi) ? hi : x);
}

}  // namespace

// ============================================================ engine
// K-wide register rows: K consecutive values moved with the widest aligned
// vector loads/stores (the offsets used are multiples of K elements).
template <typename T, int K>
struct RowK {
    T v[K];
};

template <typename T, int K, bool L2ONLY>
__device__ __forceinline__ void load_row(RowK<T, K> &r, const T *p) {
    if constexpr (K * sizeof(T) >= 16) {
#pragma unroll
        for (int i = 0; i < K; i += 16 / sizeof(T)) {
            if constexpr (sizeof(T) == 4) {
                const float4 t = L2ONLY ? __ldcg(reinterpret_cast<const float4 *>(p + i))
                                        : *reinterpret_cast<const float4 *>(p + i);
                r.v[i] = t.x; r.v[i + 1] = t.y; r.v[i + 2] = t.z; r.v[i + 3] = t.w;
            } else {
                const double2 t = L2ONLY ? __ldcg(reinterpret_cast<const double2 *>(p + i))
                                         : *reinterpret_cast<const double2 *>(p + i);
                r.v[i] = t.x; r.v[i + 1] = t.y;
            }
        }
    } else {
#pragma unroll
        for (int i = 0; i < K; ++i) r.v[i] = L2ONLY ? __ldcg(p + i) : p[i];
    }
}

template <typename T, int K>
__device__ __forceinline__ void store_row(T *p, const RowK<T, K> &r) {
    if constexpr (K * sizeof(T) >= 16) {
#pragma unroll
        for (int i = 0; i < K; i += 16 / sizeof(T)) {
            if constexpr (sizeof(T) == 4)
                *reinterpret_cast<float4 *>(p + i) = make_float4(r.v[i], r.v[i + 1], r.v[i + 2], r.v[i + 3]);
            else
                *reinterpret_cast<double2 *>(p + i) = make_double2(r.v[i], r.v[i + 1]);
        }
    } else {
#pragma unroll
        for (int i = 0; i < K; ++i) p[i] = r.v[i];
    }
}

__device__ __forceinline__ Q4<float> ld4cg(const float *p) {
    const float4 t = __ldcg(reinterpret_cast<const float4 *>(p));
    return {{t.x, t.y, t.z, t.w}};
}
__device__ __forceinline__ Q4<double> ld4cg(const double *p) {
    const double2 a = __ldcg(reinterpret_cast<const double2 *>(p));
    const double2 b = __ldcg(reinterpret_cast<const double2 *>(p + 2));
    return {{a.x, a.y, b.x, b.y}};
}
__device__ __forceinline__ void st4cg(float *p, const Q4<float> &q) {
    __stcg(reinterpret_cast<float4 *>(p), make_float4(q.v[0], q.v[1], q.v[2], q.v[3]));
}
__device__ __forceinline__ void st4cg(double *p, const Q4<double> &q) {
    __stcg(reinterpret_cast<double2 *>(p), make_double2(q.v[0], q.v[1]));
    __stcg(reinterpret_cast<double2 *>(p + 2), make_double2(q.v[2], q.v[3]));
}

// One warp task with exactly NQT chunks per position.  bt holds +bbar~ for
// members with M = F^T F and -bbar~ for M = I - F^T F, so that y = bt + F^T w
// gives x_s = y or v - y.
// Adds a task's test sums over its J member positions to the warp's sums of the
// column, quantities 0, 1, 3, 4, spread over the positions as they are added:
// at K = 8 FP64 adds of 4 instead of 12 (each occupies the sub-partition's FP64
// pipe for about 64 cycles, and the tasks' were a third of a tested iteration).
template <int K>
__device__ __forceinline__ void add_column_sums(double *redw, int sc, int jpos, double c0, double c1, double c3,
                                                double c4) {
    static_assert(K <= 8, "four member positions at least");
    const bool b0 = jpos & 1, b1 = jpos & 2;
    const double p0 = (b0 ? c3 : c0) + __shfl_xor_sync(0xffffffffu, b0 ? c0 : c3, K);
    const double p1 = (b0 ? c4 : c1) + __shfl_xor_sync(0xffffffffu, b0 ? c1 : c4, K);
    double r = (b1 ? p1 : p0) + __shfl_xor_sync(0xffffffffu, b1 ? p0 : p1, 2 * K);
#pragma unroll
    for (int o = 4 * K; o < 32; o <<= 1) r += __shfl_xor_sync(0xffffffffu, r, o);
    if (jpos < 4) redw[sc * 6 + 3 * (jpos & 1) + (jpos >> 1)] += r;
}

// Shared-memory slot array: chunk ch, slot e, column sc at slot_row(ch, e) * K
// + sc.  Between the two phases of an iteration it holds, at every slot, x of
// the slot's global (written there by the global update); otherwise
// u = rho x_s - lambda of the slot.  slot_row swizzles the four slots of a
// chunk so that the lanes that share a shared-memory transaction (consecutive
// chunks, one slot each) fall on distinct banks at each row width (K = 2 in
// FP32 with the swizzle of 32-byte rows: 4-way conflicts, the loads of u at the
// start of a task 840 cycles).  Padding slots hold 0.
template <typename T, int K>
__device__ __forceinline__ int upos(int ch, int e, int sc) {
    return slot_row(ch, e, K * (int)sizeof(T)) * K + sc;
}

// A lane's places in a task's chunks.  A task's first chunk and the chunks of
// its next positions are multiples of J = 32 / K apart, which the swizzle does
// not see, so they are offsets that the lane keeps for the launch.
struct LaneRows {
    int at[4];
};

// ---- tensor memory (tcgen05, tmem.cuh): lambda and bbar~ of the tasks,
// 32-bit columns.
// 8 consecutive columns of the lane: lambda (4) then bbar~ (4) of one chunk
__device__ __forceinline__ void tm_ld8(unsigned taddr, Q4<float> &m, Q4<float> &b) {
    unsigned r[8];
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
                 : "r"(taddr)
                 : "memory");
#pragma unroll
    for (int e = 0; e < 4; ++e) {
        m.v[e] = __uint_as_float(r[e]);
        b.v[e] = __uint_as_float(r[4 + e]);
    }
}
__device__ __forceinline__ void tm_st8(unsigned taddr, const Q4<float> &m, const Q4<float> &b) {
    asm volatile("tcgen05.st.sync.aligned.32x32b.x8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"r"(taddr),
                 "r"(__float_as_uint(m.v[0])), "r"(__float_as_uint(m.v[1])), "r"(__float_as_uint(m.v[2])),
                 "r"(__float_as_uint(m.v[3])), "r"(__float_as_uint(b.v[0])), "r"(__float_as_uint(b.v[1])),
                 "r"(__float_as_uint(b.v[2])), "r"(__float_as_uint(b.v[3]))
                 : "memory");
}
__device__ __forceinline__ void tm_st4(unsigned taddr, const Q4<float> &m) {
    asm volatile("tcgen05.st.sync.aligned.32x32b.x4.b32 [%0], {%1, %2, %3, %4};" ::"r"(taddr),
                 "r"(__float_as_uint(m.v[0])), "r"(__float_as_uint(m.v[1])), "r"(__float_as_uint(m.v[2])),
                 "r"(__float_as_uint(m.v[3]))
                 : "memory");
}
__device__ __forceinline__ void tm_ld4(unsigned taddr, Q4<float> &m) {
    unsigned r[4];
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0, %1, %2, %3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
                 : "r"(taddr)
                 : "memory");
#pragma unroll
    for (int e = 0; e < 4; ++e) m.v[e] = __uint_as_float(r[e]);
}

// Tensor-memory staging of one task (TMTASK): at the start of a launch
// lambda and bbar~ from the engine arrays into the task's columns; at a
// freeze or the end lambda back to the engine array for the columns flagged
// in `wcols` (bit sc), after the lanes' own loads.
template <int K, int NQT>
__device__ __forceinline__ void tm_stage_in(const BatchTask &tk, unsigned tl, const float *mu_c, const float *bt_c,
                                            int jpos, int sc, float rho) {
    constexpr int J = 32 / K;
    const unsigned col = (unsigned)(tk.tm >> 2);
#pragma unroll
    for (int q = 0; q < NQT; ++q) {
        const int off = ((tk.ch0 + jpos + q * J) * K + sc) * 4;
        Q4<float> b = ld4cg(bt_c + off);
#pragma unroll
        for (int e = 0; e < 4; ++e) b.v[e] *= rho;     // rho bbar~
        tm_st8(tl + col + 8 * q, ld4cg(mu_c + off), b);
    }
}
template <int K, int NQT>
__device__ __forceinline__ void tm_stage_out(const BatchTask &tk, unsigned tl, float *mu_c, int jpos, int sc,
                                             bool write) {
    constexpr int J = 32 / K;
    const unsigned col = (unsigned)(tk.tm >> 2);
#pragma unroll
    for (int q = 0; q < NQT; ++q) {
        Q4<float> m;
        tm_ld4(tl + col + 8 * q, m);
        tm_wait_ld();
        if (write) st4cg(mu_c + ((tk.ch0 + jpos + q * J) * K + sc) * 4, m);
    }
}

// The slot array holds rho x_g at every slot when the task starts (the global
// update wrote it; a one-copy unbounded global's slot holds its u, which is
// that value) and gets u at the end; y starts at +-rho bbar~ (the FP64 arrays
// hold it scaled, FP32 tensor-memory plans stage it scaled, the other FP32
// ones scale it on load).  FP64 form:
template <int K, int NQT, bool>
__device__ __forceinline__ void batch_task(const BatchTask &tk, const double *Fs, double *us, double *mu_c,
                                           const double *bt_c, double *ds_c, const double *lr_c, const double *xs_c,
                                           int jpos, int sc, const LaneRows &lr, double, double inv_rho, bool check, bool act, bool wds,
                                           double *redw, unsigned) {
    constexpr int J = 32 / K;
    const int mode1 = (tk.modes >> (jpos >> tk.lp)) & 1;
    double v[4 * NQT], y[4 * NQT];
    double c0 = 0.0, c1 = 0.0, c3 = 0.0, c4 = 0.0;
    const int ch0 = tk.ch0 + jpos;
    double *ut = us + tk.ch0 * 4 * K;
#pragma unroll
    for (int q = 0; q < NQT; ++q) {
        const int ch = ch0 + q * J;
        const int off = (ch * K + sc) * 4;
        const Q4<double> m4 = ld4cg(mu_c + off), b4 = ld4cg(bt_c + off);
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            y[4 * q + e] = b4.v[e];
            v[4 * q + e] = ut[lr.at[e] + q * J * 4 * K] + m4.v[e];
        }
    }
    // rho x_s = M V + rho bbar~ over the factor rows, two rows per step
    const int rstride = NQT * J * 4;
    const double *F0 = Fs + tk.foff + jpos * 4;
    const int red_top = tk.p * K;
    // (the task's row count is even: a member's missing rows are zero)
    for (int r = 0; r < tk.f; r += 2, F0 += 2 * rstride) {
        const double *F1 = F0 + rstride;
        // one accumulation chain per row (four partial sums and their adds
        // measured 4.5 % slower per launch: more instructions)
        double s0 = 0.0, s1 = 0.0;
#pragma unroll
        for (int q = 0; q < NQT; ++q) {
            const Q4<double> f0 = ld4(F0 + q * J * 4);
            const Q4<double> f1 = ld4(F1 + q * J * 4);
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                s0 += f0.v[e] * v[4 * q + e];
                s1 += f1.v[e] * v[4 * q + e];
            }
        }
        for (int o = K; o < red_top; o <<= 1) {
            s0 += __shfl_xor_sync(0xffffffffu, s0, o);
            s1 += __shfl_xor_sync(0xffffffffu, s1, o);
        }
#pragma unroll
        for (int q = 0; q < NQT; ++q) {
            const Q4<double> f0 = ld4(F0 + q * J * 4);
            const Q4<double> f1 = ld4(F1 + q * J * 4);
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                y[4 * q + e] += f0.v[e] * s0;
                y[4 * q + e] += f1.v[e] * s1;
            }
        }
    }
#pragma unroll
    for (int q = 0; q < NQT; ++q) {
        const int ch = ch0 + q * J;
        const int off = (ch * K + sc) * 4;
        Q4<double> x4, m4, u4, r4;
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            const double vv = v[4 * q + e];
            const double rx = mode1 ? y[4 * q + e] : vv - y[4 * q + e];     // rho x_s
            const double mun = vv - rx;
            r4.v[e] = rx;
            m4.v[e] = mun;
            u4.v[e] = rx - mun;
        }
        // x_s~ (written on wds iterations, test terms) only when it is used: a
        // multiply costs 64 cycles
        if (wds) {
#pragma unroll
            for (int e = 0; e < 4; ++e) x4.v[e] = r4.v[e] * inv_rho;
        }
        if (check) {
            const Q4<double> o4 = ld4cg(ds_c + off);
            const Q4<double> l4 = ld4cg(lr_c + off);
            const Q4<double> g4 = ld4cg(xs_c + off);
            double t0 = 0.0, t1 = 0.0, t3 = 0.0, t4 = 0.0;
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                const double d0 = (ut[lr.at[e] + q * J * 4 * K] - r4.v[e]) * inv_rho, d1 = x4.v[e] - o4.v[e];
                const double xa = x4.v[e] + g4.v[e];
                const double la = m4.v[e] + l4.v[e];
                t0 += d0 * d0;
                t1 += d1 * d1;
                t3 += xa * xa;
                t4 += la * la;
            }
            c0 += t0;
            c1 += t1;
            c3 += t3;
            c4 += t4;
        }
#pragma unroll
        for (int e = 0; e < 4; ++e) ut[lr.at[e] + q * J * 4 * K] = u4.v[e];
        if (act) {
            st4cg(mu_c + off, m4);
            if (wds) st4cg(ds_c + off, x4);
        }
    }
    if (check) {
        add_column_sums<K>(redw, sc, jpos, c0, c1, c3, c4);
    }
}

// ---- FP32: packed pairs (two values per 64-bit register)
// What bounds an FP32 iteration: with every SM's CTA full (K = 8) issue slots
// and shared-memory transactions, with few instances (K = 2) the latency of
// the longest task and of the global update.  Hence one instruction per two
// multiply-adds; a row's sum over a member's lanes with its levels unrolled (a
// loop over them took 90 cycles per level, twice the shuffle and the add);
// every tensor-memory load of a task before one wait; a slot array free of
// bank conflicts at each K; global-update items sorted so that a warp's lanes
// take the same branches.  us per iteration with a test every 100, against scalar
// multiply-adds: 123 buses, 40 instances (K = 2) 3.80 -> 2.52; 34 buses, 200
// instances (K = 2) 2.26 -> 1.59; 123 buses, 1024 instances (K = 8) 6.53 -> 6.14.
using u64 = unsigned long long;
__device__ __forceinline__ u64 pk(float a, float b) {
    u64 r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
    return r;
}
__device__ __forceinline__ void unpk(u64 p, float &a, float &b) { asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(p)); }
__device__ __forceinline__ u64 fma2(u64 a, u64 b, u64 c) {
    u64 r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
    return r;
}
__device__ __forceinline__ u64 mul2(u64 a, u64 b) {
    u64 r;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ u64 add2(u64 a, u64 b) {
    u64 r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}

// R factor rows of a task whose members span 2^LP lanes: w_r = <F_r, V> over
// the member's lanes, y += w_r F_r.  A row's product is two chains (the even
// and the odd slots of a lane), added at the end.
template <int K, int NQT, int R, int LP>
__device__ __forceinline__ void rows(const float *F0, int rstride, const u64 (&v)[2 * NQT], u64 (&y)[2 * NQT]) {
    constexpr int J = 32 / K;
    u64 s[R];
#pragma unroll
    for (int q = 0; q < NQT; ++q)
#pragma unroll
        for (int i = 0; i < R; ++i) {
            const ulonglong2 a = *reinterpret_cast<const ulonglong2 *>(F0 + i * rstride + q * J * 4);
            s[i] = q == 0 ? mul2(a.x, v[0]) : fma2(a.x, v[2 * q], s[i]);
            s[i] = fma2(a.y, v[2 * q + 1], s[i]);
        }
    float t[R];
#pragma unroll
    for (int i = 0; i < R; ++i) {
        float e, o;
        unpk(s[i], e, o);
        t[i] = e + o;
    }
#pragma unroll
    for (int o = K; o < (K << LP); o <<= 1)
#pragma unroll
        for (int i = 0; i < R; ++i) t[i] += __shfl_xor_sync(0xffffffffu, t[i], o);
#pragma unroll
    for (int i = 0; i < R; ++i) s[i] = pk(t[i], t[i]);
#pragma unroll
    for (int q = 0; q < NQT; ++q)
#pragma unroll
        for (int i = 0; i < R; ++i) {
            const ulonglong2 a = *reinterpret_cast<const ulonglong2 *>(F0 + i * rstride + q * J * 4);
            y[2 * q] = fma2(a.x, s[i], y[2 * q]);
            y[2 * q + 1] = fma2(a.y, s[i], y[2 * q + 1]);
        }
}

// The f rows (an even number: a member's missing rows are zero), two per step;
// with one instance per CTA, where a warp has a task or two and waits on their
// chains, six or four while they last (34 buses 1.68 -> 1.56 us per iteration).
template <int K, int NQT, int LP>
__device__ __forceinline__ void task_rows(const float *F0, int rstride, int f, const u64 (&v)[2 * NQT],
                                          u64 (&y)[2 * NQT]) {
    int r = 0;
    if constexpr (K == 1 && NQT == 1)
#pragma unroll 1
        for (; r + 6 <= f; r += 6, F0 += 6 * rstride) rows<K, NQT, 6, LP>(F0, rstride, v, y);
    if constexpr (K == 1 && NQT <= 2)
#pragma unroll 1
        for (; r + 4 <= f; r += 4, F0 += 4 * rstride) rows<K, NQT, 4, LP>(F0, rstride, v, y);
#pragma unroll 1
    for (; r < f; r += 2, F0 += 2 * rstride) rows<K, NQT, 2, LP>(F0, rstride, v, y);
}

// Keeps uses of the values after the point where it stands (a tensor-memory wait).
__device__ __forceinline__ void tie(Q4<float> &q) {
    asm volatile("" : "+f"(q.v[0]), "+f"(q.v[1]), "+f"(q.v[2]), "+f"(q.v[3]));
}

// batch_task in FP32 with packed pairs: the same arithmetic, the factor rows by rows().
template <int K, int NQT, bool TM>
__device__ __forceinline__ void batch_task(const BatchTask &tk, const float *Fs, float *us, float *mu_c,
                                           const float *bt_c, float *ds_c, const float *lr_c, const float *xs_c,
                                           int jpos, int sc, const LaneRows &lr, float rho, float inv_rho, bool check,
                                           bool act, bool wds, double *redw, unsigned tl) {
    constexpr int J = 32 / K;
    const bool mode1 = (tk.modes >> (jpos >> tk.lp)) & 1;
    u64 v[2 * NQT], y[2 * NQT];
    float f0 = 0.f, f1 = 0.f, f3 = 0.f, f4 = 0.f;     // test terms, FP32 over the task's chunks
    const int ch0 = tk.ch0 + jpos;
    float *ut = us + tk.ch0 * 4 * K;
    const unsigned tcol = tl + (unsigned)(tk.tm >> 2);
    {
        Q4<float> m4[NQT], b4[NQT];
#pragma unroll
        for (int q = 0; q < NQT; ++q) {
            if constexpr (TM) {
                tm_ld8(tcol + 8 * q, m4[q], b4[q]);
            } else {
                const int off = ((ch0 + q * J) * K + sc) * 4;
                m4[q] = ld4cg(mu_c + off);
                b4[q] = ld4cg(bt_c + off);
#pragma unroll
                for (int e = 0; e < 4; ++e) b4[q].v[e] *= rho;
            }
        }
        if constexpr (TM) {                  // every load of the task in flight, one wait
            tm_wait_ld();
#pragma unroll
            for (int q = 0; q < NQT; ++q) {
                tie(m4[q]);
                tie(b4[q]);
            }
        }
#pragma unroll
        for (int q = 0; q < NQT; ++q) {
            const int ch = ch0 + q * J;
            y[2 * q] = pk(b4[q].v[0], b4[q].v[1]);
            y[2 * q + 1] = pk(b4[q].v[2], b4[q].v[3]);
            v[2 * q] = add2(pk(ut[lr.at[0] + q * J * 4 * K], ut[lr.at[1] + q * J * 4 * K]), pk(m4[q].v[0], m4[q].v[1]));
            v[2 * q + 1] = add2(pk(ut[lr.at[2] + q * J * 4 * K], ut[lr.at[3] + q * J * 4 * K]), pk(m4[q].v[2], m4[q].v[3]));
        }
    }
    // rho x_s = M V + rho bbar~ over the factor rows, two per step
    const int rstride = NQT * J * 4;
    const float *F0 = Fs + tk.foff + jpos * 4;
    switch (tk.lp) {
        case 0: task_rows<K, NQT, 0>(F0, rstride, tk.f, v, y); break;
        case 1: task_rows<K, NQT, 1>(F0, rstride, tk.f, v, y); break;
        case 2: task_rows<K, NQT, 2>(F0, rstride, tk.f, v, y); break;
        case 3: if constexpr (J >= 8) task_rows<K, NQT, 3>(F0, rstride, tk.f, v, y); break;
        case 4: if constexpr (J >= 16) task_rows<K, NQT, 4>(F0, rstride, tk.f, v, y); break;
        default: if constexpr (J >= 32) task_rows<K, NQT, 5>(F0, rstride, tk.f, v, y); break;
    }
    // rho x_s = y or V - y, as ca V + cb y with exact coefficients
    const float ca = mode1 ? 0.0f : 1.0f, cb = mode1 ? 1.0f : -1.0f;
    const u64 ca2 = pk(ca, ca), cb2 = pk(cb, cb), neg = pk(-1.0f, -1.0f), ir2 = pk(inv_rho, inv_rho);
#pragma unroll
    for (int q = 0; q < NQT; ++q) {
        const int ch = ch0 + q * J;
        const int off = (ch * K + sc) * 4;
        Q4<float> m4, u4;
        u64 rx[2];
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            rx[h] = fma2(y[2 * q + h], cb2, mul2(v[2 * q + h], ca2));
            const u64 mun = fma2(rx[h], neg, v[2 * q + h]);
            const u64 un = fma2(mun, neg, rx[h]);
            unpk(mun, m4.v[2 * h], m4.v[2 * h + 1]);
            unpk(un, u4.v[2 * h], u4.v[2 * h + 1]);
        }
        if (check) {
            // x_s~ before, lambda_ref, x_ref (padding slots hold 0)
            const Q4<float> o4 = ld4cg(ds_c + off), l4 = ld4cg(lr_c + off), g4 = ld4cg(xs_c + off);
            float t0 = 0.f, t1 = 0.f, t3 = 0.f, t4 = 0.f;
            Q4<float> r4, x4;
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                unpk(rx[h], r4.v[2 * h], r4.v[2 * h + 1]);
                unpk(mul2(rx[h], ir2), x4.v[2 * h], x4.v[2 * h + 1]);
            }
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                const float d0 = (ut[lr.at[e] + q * J * 4 * K] - r4.v[e]) * inv_rho, d1 = x4.v[e] - o4.v[e];
                const float xa = x4.v[e] + g4.v[e];
                const float la = m4.v[e] + l4.v[e];
                t0 += d0 * d0;
                t1 += d1 * d1;
                t3 += xa * xa;
                t4 += la * la;
            }
            f0 += t0;
            f1 += t1;
            f3 += t3;
            f4 += t4;
        }
#pragma unroll
        for (int e = 0; e < 4; ++e) ut[lr.at[e] + q * J * 4 * K] = u4.v[e];
        // (tensor memory: every lane; a frozen column keeps iterating there,
        // its lambda went to the engine array when it froze)
        if constexpr (TM) tm_st4(tcol + 8 * q, m4);
        else if (act) st4cg(mu_c + off, m4);
        if (act && wds) {
            Q4<float> x4;
#pragma unroll
            for (int h = 0; h < 2; ++h) unpk(mul2(rx[h], ir2), x4.v[2 * h], x4.v[2 * h + 1]);
            st4cg(ds_c + off, x4);
        }
    }
    if (check) {
        double c0 = (double)f0, c1 = (double)f1, c3 = (double)f3, c4 = (double)f4;
        add_column_sums<K>(redw, sc, jpos, c0, c1, c3, c4);
    }
}

// K: instance columns per CTA (compile time), J = 32 / K member positions.
// NQ: chunks of 4 slots a lane can hold (registers v and y: 2 * 4 * NQ).
// FG: factors read from global memory (L1/L2) instead of shared memory.
// TM (FP32 only): lambda and bbar~ of the tasks in tensor memory for the
// launch instead of streamed from L2; the tasks of lane quadrant q run on the
// warps w with w % 4 == q (a dynamic schedule per quadrant).
template <typename T, int K, int NQ, bool FG, bool TM>
__global__ void __launch_bounds__(512, 1)
    k_batch_engine(BatchArgs<T> a, int n_iters, int check_every) {
    constexpr int J = 32 / K;
    constexpr int KS = K == 1 ? 0 : K == 2 ? 1 : K == 4 ? 2 : K == 8 ? 3 : K == 16 ? 4 : 5;
    constexpr int KQ = K < 4 ? K : 4;          // columns per global-update item
    constexpr int NQD = K / KQ;                  // items per global
    constexpr int QS = NQD == 1 ? 0 : NQD == 2 ? 1 : NQD == 4 ? 2 : 3;
    // later copies' rows of a global-update item in flight together: 4, 2 for FP64
    // rows of four, whose registers (with four items per thread and four rows
    // 224 bytes of a thread spilled) the rest of the iteration needs.  us per
    // FP64 iteration, four items and four rows / one item and one row / one and
    // two: 5, 13, 34 and 123 buses, 400 instances 11.2, 16.1, 21.4 and 90.4 / 10.0,
    // 15.3, 21.2 and 86.5 / 9.9, 16.0, 21.0 and 86.3; 1024 instances of 34 and 123
    // 35.5 and 180 / 35.8 and 173 / 35.6 and 173.  One item per thread at a time
    // in FP32 too (2 to 4 were no faster).
    constexpr int CB = (sizeof(T) == 8 && KQ == 4) ? 2 : 4;
    extern __shared__ __align__(16) unsigned char smraw[];
    T *Fsm = reinterpret_cast<T *>(smraw);
    const T *Fs = FG ? a.Fpk : Fsm;
    T *us = reinterpret_cast<T *>(smraw + a.off_u);
    int4 *gts = reinterpret_cast<int4 *>(smraw + a.off_gt);      // [Gs] (row0, row1, copies | first extra << 8, bounded index)
    T *rcs = reinterpret_cast<T *>(smraw + a.off_rc);            // 1 / N by copy count N
    BatchTask *tks = reinterpret_cast<BatchTask *>(smraw + a.off_task);   // the warp tasks
    int *usg = reinterpret_cast<int *>(smraw + a.off_useg);      // slot-array rows of the third and later copies
    T *bnd = reinterpret_cast<T *>(smraw + a.off_bnd);           // [NB][3][K]: rho (bounds - x_ref), c~
    double *red = reinterpret_cast<double *>(smraw + a.off_red);
    int *flags = reinterpret_cast<int *>(smraw + a.off_flag);    // [0,K) running, [K,2K) just finished
    int *tnext = flags + 2 * K;                                    // next task of the dynamic schedule (per quadrant)
    __shared__ unsigned tm_base;                                   // tensor-memory address of the allocation
    const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
    const int nthr = blockDim.x;
    const int c = blockIdx.x;
    if (tid < K) {
        const int in = a.inst[c * K + tid];
        flags[tid] = (in >= 0 && !a.st[in].done) ? 1 : 0;
        flags[K + tid] = 0;
    }
    __syncthreads();
    {
        int any = 0;
        for (int q = 0; q < K; ++q) any |= flags[q];
        if (!any) return;
    }
    // factors and the global-update tables into shared memory (nF is a multiple of 4)
    if (!FG)
        for (int i = tid * 4; i < a.nF; i += nthr * 4) st4(Fsm + i, ld4(a.Fpk + i));
    for (int j = tid; j < a.Gs; j += nthr) gts[j] = __ldg(a.gtab + j);
    // 1 / N by copy count N: the global update stores rho x = (sum u - c~) / N
    for (int i = tid; i < kBatchRecip; i += nthr) rcs[i] = i ? (T)(1.0 / (double)i) : T(0);
    for (int i = tid; i < a.n_tasks; i += nthr) tks[i] = a.tasks[i];
    for (int k = tid; k < a.n_uxt; k += nthr) usg[k] = __ldg(a.uxt + k);
    const size_t sb = (size_t)c * a.NCH * K * 4;     // this CTA's slot arrays
    const size_t gb = (size_t)c * a.G * K;           // global arrays
    const size_t bb = (size_t)c * a.NB * K;          // bounded-global arrays
    for (int idx = tid; idx < a.NB * K; idx += nthr) {
        const int b = idx >> KS, col = idx & (K - 1);
        bnd[(b * 3) * K + col] = a.rho * __ldcg(a.lbt + bb + idx);         // rho (bounds - x_ref)
        bnd[(b * 3 + 1) * K + col] = a.rho * __ldcg(a.ubt + bb + idx);
        bnd[(b * 3 + 2) * K + col] = __ldcg(a.cbt + bb + idx);              // c~
    }
    T *mu_c = a.mu + sb, *ds_c = a.ds + sb;
    const T *bt_c = a.bt + sb, *lr_c = a.lref + sb, *xs_c = a.xsr + sb;
    // u = rho d - mu into the swizzled slot array
    for (int idx = tid; idx < a.NCH * K; idx += nthr) {
        const int ch = idx >> KS, col = idx & (K - 1);
        const Q4<T> d = ld4cg(ds_c + (size_t)idx * 4), m = ld4cg(mu_c + (size_t)idx * 4);
#pragma unroll
        for (int e = 0; e < 4; ++e) us[upos<T, K>(ch, e, col)] = a.rho * d.v[e] - m.v[e];
    }
    const int sc = tid & (K - 1);
    const int jpos = lane >> KS;
    LaneRows lr;
#pragma unroll
    for (int e = 0; e < 4; ++e) lr.at[e] = upos<T, K>(jpos, e, sc);
    const int n_warps = nthr >> 5;
    const int qd = w & 3, wq = w >> 2, nwq = n_warps >> 2;     // quadrant, warp in it, warps per quadrant
    unsigned tl = 0;                                             // this warp's tensor-memory lane base
    if constexpr (TM) {
        if (w == 0) tm_alloc(&tm_base, a.tm_cols);
        tm_fence_before();
        __syncthreads();
        tm_fence_after();
        tl = tm_base + ((unsigned)(32 * qd) << 16);
        for (int t = a.qstart[qd] + wq; t < a.qstart[qd + 1]; t += nwq) {
            const BatchTask tk = a.tasks[t];
            switch (tk.nq) {
                case 1: tm_stage_in<K, 1>(tk, tl, mu_c, bt_c, jpos, sc, a.rho); break;
                case 2: tm_stage_in<K, 2>(tk, tl, mu_c, bt_c, jpos, sc, a.rho); break;
                case 3: tm_stage_in<K, 3>(tk, tl, mu_c, bt_c, jpos, sc, a.rho); break;
                default: tm_stage_in<K, 4>(tk, tl, mu_c, bt_c, jpos, sc, a.rho); break;
            }
        }
        tm_wait_st();
        tm_fence_before();
    }
    __syncthreads();
    if constexpr (TM) tm_fence_after();
    const T rho = a.rho, inv_rho = a.inv_rho;
    double *redw = red + (size_t)w * K * 6;      // this warp's test sums per column
    int last_check = 0;
    bool all_done = false;
    const int GK = a.G * K;
    const int GQ = a.Gs * NQD;       // the globals the global update computes (the table's first Gs)
    for (int it = 0; it < n_iters; ++it) {
        const bool check = check_every > 0 && ((it + 1) % check_every == 0);
        const bool last = it == n_iters - 1;
        const bool wds = check || last || (check_every > 0 && ((it + 2) % check_every == 0));
        const bool act = flags[sc] != 0;
        if (check && lane < K)
#pragma unroll
            for (int q = 0; q < 6; ++q) redw[lane * 6 + q] = 0.0;
        if constexpr (TM) {
            if (tid < 4) tnext[tid] = a.qstart[tid] + nwq;
        } else if (tid == 0) {
            *tnext = n_warps;
        }
        // ---- G: global update (Eq. closed_1).  An item is one global and KQ of
        // its columns: sum of u over the copies, shift by c~ (bounded globals,
        // whose table entry names their bounded index; elsewhere c~ = 0),
        // 1 / N, clip to rho (bounds - x_ref), and rho x stored into every
        // copy's slot
        // (items of many copies come first; the last round, when it is not
        // full, goes to the last threads, which had none of those)
        for (int b0 = 0; b0 < GQ; b0 += nthr) {
            const int item = b0 + (b0 + nthr > GQ ? nthr - 1 - tid : tid);
            if (item >= GQ) continue;
            const int h = item & (NQD - 1);
            const int4 gt = gts[item >> QS];
            const int cnt = gt.z & 0xff;                      // (every global has a copy)
            const int row0 = gt.x + h * KQ, row1 = gt.y + h * KQ;
            const int st0 = (gt.z >> 8) - 2;                  // usg[st0 + q]: copy q >= 2
            RowK<T, KQ> sum;
            load_row<T, KQ, false>(sum, us + row0);
            if (cnt > 1) {
                RowK<T, KQ> u1;
                load_row<T, KQ, false>(u1, us + row1);
#pragma unroll
                for (int k = 0; k < KQ; ++k) sum.v[k] += u1.v[k];
            }
            for (int q = 2; q < cnt; q += CB) {               // CB copies' loads in flight
                int rr[CB];
#pragma unroll
                for (int c = 0; c < CB; ++c) rr[c] = q + c < cnt ? usg[st0 + q + c] : 0;
                RowK<T, KQ> uq[CB];
#pragma unroll
                for (int c = 0; c < CB; ++c)
                    if (q + c < cnt) load_row<T, KQ, false>(uq[c], us + rr[c] + h * KQ);
#pragma unroll
                for (int c = 0; c < CB; ++c)
                    if (q + c < cnt)
#pragma unroll
                        for (int k = 0; k < KQ; ++k) sum.v[k] += uq[c].v[k];
            }
            const T rcp = rcs[cnt];
            if (gt.w >= 0) {
                RowK<T, KQ> lo, hi, cr;
                load_row<T, KQ, false>(cr, bnd + (gt.w * 3 + 2) * K + h * KQ);
                load_row<T, KQ, false>(lo, bnd + (gt.w * 3) * K + h * KQ);
                load_row<T, KQ, false>(hi, bnd + (gt.w * 3 + 1) * K + h * KQ);
#pragma unroll
                for (int k = 0; k < KQ; ++k) sum.v[k] = (sum.v[k] - cr.v[k]) * rcp;
#pragma unroll
                for (int k = 0; k < KQ; ++k) sum.v[k] = clampT(sum.v[k], lo.v[k], hi.v[k]);
            } else {
#pragma unroll
                for (int k = 0; k < KQ; ++k) sum.v[k] *= rcp;
            }
            store_row<T, KQ>(us + row0, sum);
            if (cnt > 1) store_row<T, KQ>(us + row1, sum);
            for (int q = 2; q < cnt; q += CB) {
                int rr[CB];
#pragma unroll
                for (int c = 0; c < CB; ++c) rr[c] = q + c < cnt ? usg[st0 + q + c] : 0;
#pragma unroll
                for (int c = 0; c < CB; ++c)
                    if (q + c < cnt) store_row<T, KQ>(us + rr[c] + h * KQ, sum);
            }
        }
        __syncthreads();
        if (check || last) {
            // x of each global (rho x at its first copy): objective and
            // ||B x||^2 per column on test iterations, and x~ of the running
            // instances for their results (thread column sc = tid % K)
            // (FP32 plans: x_ref + x~ and the thread's partial sums in FP32,
            // FP64 from the warp sums on; FP64 plans: FP64 throughout)
            double c2 = 0.0, c5 = 0.0;
            T p2 = T(0), p5 = T(0);
            constexpr int XB = 4;        // items whose loads are in flight together
            for (int i0 = tid; i0 < GK; i0 += XB * nthr) {
                int gx[XB], gi[XB];
                T xr[XB], cost[XB];
#pragma unroll
                for (int q = 0; q < XB; ++q) {
                    const int item = i0 + q * nthr;
                    gx[q] = item < GK ? __ldg(a.gx + (item >> KS)) : 0;      // first copy's row | copies << 24
                    gi[q] = item < GK ? __ldg(a.gperm + (item >> KS)) : -1;
                }
                if (check)
#pragma unroll
                    for (int q = 0; q < XB; ++q) {
                        xr[q] = gi[q] >= 0 ? __ldcg(a.xrf + gb + (size_t)gi[q] * K + sc) : T(0);
                        cost[q] = gi[q] >= 0 ? __ldg(a.cost + gi[q]) : T(0);
                    }
#pragma unroll
                for (int q = 0; q < XB; ++q) {
                    if (gi[q] < 0) continue;
                    const T xv = us[(gx[q] & 0xffffff) + sc] * a.inv_rho;
                    if (flags[sc]) a.xo[gb + (size_t)gi[q] * K + sc] = xv;
                    if (check) {
                        const unsigned n = (unsigned)gx[q] >> 24;
                        if constexpr (sizeof(T) == 4) {
                            const T xa = xv + xr[q];
                            p2 += (T)n * xa * xa;
                            p5 += cost[q] * xa;
                        } else {
                            const double xa = (double)xv + (double)xr[q];
                            c2 += (double)n * xa * xa;
                            c5 += (double)cost[q] * xa;
                        }
                    }
                }
            }
            if constexpr (sizeof(T) == 4) {
                c2 = (double)p2;
                c5 = (double)p5;
            }
            if (check) {
                const bool b0 = jpos & 1;
                double r = (b0 ? c5 : c2) + __shfl_xor_sync(0xffffffffu, b0 ? c2 : c5, K);
                for (int o = 2 * K; o < 32; o <<= 1) r += __shfl_xor_sync(0xffffffffu, r, o);
                if (jpos < 2) redw[sc * 6 + (b0 ? 5 : 2)] += r;
            }
            __syncthreads();      // the slots still hold x: read before phase L overwrites them
        }
        // ---- L: local update (Eq. closed_2) and dual update (Eq. ADMM-3)
        // tasks in decreasing cost; warps take the next one as they finish
        // (test iterations: task t on warp t % n_warps, a fixed summation order)
        {
            // each warp's first task is its own (the counter starts at
            // n_warps); the next task's index is claimed at the start of a
            // task and read at its end, so the atomic's latency is hidden
            // (tensor-memory plans: the same within the warp's quadrant)
            int t = TM ? a.qstart[qd] + wq : w;
            const int t_end = TM ? a.qstart[qd + 1] : a.n_tasks;
            const int t_step = TM ? nwq : n_warps;
            int *cnt = TM ? tnext + qd : tnext;
            while (t < t_end) {
                int claim = 0;
                if (!check && lane == 0) claim = atomicAdd(cnt, 1);
                const BatchTask tk = tks[t];
                switch (tk.nq) {
                    case 1: batch_task<K, 1, TM>(tk, Fs, us, mu_c, bt_c, ds_c, lr_c, xs_c, jpos, sc, lr, rho,
                                                    inv_rho, check, act, wds, redw, tl); break;
                    case 2: if constexpr (NQ >= 2) batch_task<K, 2, TM>(tk, Fs, us, mu_c, bt_c, ds_c, lr_c, xs_c,
                                                                           jpos, sc, lr, rho, inv_rho, check, act,
                                                                           wds, redw, tl); break;
                    case 3: if constexpr (NQ >= 3) batch_task<K, 3, TM>(tk, Fs, us, mu_c, bt_c, ds_c, lr_c, xs_c,
                                                                           jpos, sc, lr, rho, inv_rho, check, act,
                                                                           wds, redw, tl); break;
                    default: if constexpr (NQ >= 4) batch_task<K, 4, TM>(tk, Fs, us, mu_c, bt_c, ds_c, lr_c, xs_c,
                                                                            jpos, sc, lr, rho, inv_rho, check, act,
                                                                            wds, redw, tl); break;
                }
                t = check ? t + t_step : __shfl_sync(0xffffffffu, claim, 0);
            }
            if constexpr (TM) {
                tm_wait_st();
                tm_fence_before();
            }
        }
        if (check) {
            __syncthreads();
            if constexpr (TM) tm_fence_after();
            // eight lanes per column: lane q sums quantity q of the warps' parts
            // in warp order and takes its square root (5 in turn by one thread
            // took some 7000 cycles), the first decides
            for (int c0 = 4 * w; c0 < K; c0 += 4 * n_warps) {
                const int col = c0 + (lane >> 3), q = lane & 7;
                double sum = 0.0, root[5], s6[6];
                if (col < K && q < 6)
                    for (int ww = 0; ww < n_warps; ++ww) sum += red[((size_t)ww * K + col) * 6 + q];
                const double mine = q < 5 ? sqrt(sum) : 0.0;
#pragma unroll
                for (int i = 0; i < 6; ++i) {
                    s6[i] = __shfl_sync(0xffffffffu, sum, i, 8);
                    if (i < 5) root[i] = __shfl_sync(0xffffffffu, mine, i, 8);
                }
                if (col < K && q == 0) {
                    flags[K + col] = 0;
                    if (flags[col]) {
                        const int in = a.inst[c * K + col];
                        apply_roots(&a.st[in], s6, root, a.rho_d, check_every);
                        if (a.st[in].done) {
                            flags[col] = 0;
                            flags[K + col] = 1;
                        }
                    }
                }
            }
            __syncthreads();
            last_check = it + 1;
            if constexpr (TM) {
                // lambda of the columns that just finished, to the engine array
                int fin = 0;
                for (int q = 0; q < K; ++q) fin |= flags[K + q];
                if (fin)
                    for (int t = a.qstart[qd] + wq; t < a.qstart[qd + 1]; t += nwq) {
                        const BatchTask tk = tks[t];
                        const bool wr = flags[K + sc] != 0;
                        switch (tk.nq) {
                            case 1: tm_stage_out<K, 1>(tk, tl, (float *)mu_c, jpos, sc, wr); break;
                            case 2: tm_stage_out<K, 2>(tk, tl, (float *)mu_c, jpos, sc, wr); break;
                            case 3: tm_stage_out<K, 3>(tk, tl, (float *)mu_c, jpos, sc, wr); break;
                            default: tm_stage_out<K, 4>(tk, tl, (float *)mu_c, jpos, sc, wr); break;
                        }
                    }
            }
            int any = 0;
            for (int q = 0; q < K; ++q) any |= flags[q];
            if (!any) {
                all_done = true;
                break;
            }
        } else {
            __syncthreads();
            if constexpr (TM) tm_fence_after();
        }
    }
    if (!all_done && tid < K && flags[tid]) a.st[a.inst[c * K + tid]].iter += n_iters - last_check;
    if constexpr (TM) {
        // lambda of the columns still running, then the allocation is freed
        if (!all_done)
            for (int t = a.qstart[qd] + wq; t < a.qstart[qd + 1]; t += nwq) {
                const BatchTask tk = tks[t];
                const bool wr = flags[sc] != 0;
                switch (tk.nq) {
                    case 1: tm_stage_out<K, 1>(tk, tl, (float *)mu_c, jpos, sc, wr); break;
                    case 2: tm_stage_out<K, 2>(tk, tl, (float *)mu_c, jpos, sc, wr); break;
                    case 3: tm_stage_out<K, 3>(tk, tl, (float *)mu_c, jpos, sc, wr); break;
                    default: tm_stage_out<K, 4>(tk, tl, (float *)mu_c, jpos, sc, wr); break;
                }
            }
        tm_fence_before();
        __syncthreads();
        tm_fence_after();
        if (w == 0) tm_dealloc(tm_base, a.tm_cols);
    }
}

// ============================================================ per-instance data
// Engine column of an instance: ipos[inst] = c * K + sc (-1: not placed).

// Start point of Sec. V-A for instances [i0, i0 + cnt): x_s = x0[g], lambda = 0.
__global__ void k_binit(int i0, int cnt, int L, const int *gk, const double *x0, double *xs, double *lam,
                        DevStatus *st, long long max_iter, double eps_rel, double eps_abs) {
    const long long n = (long long)cnt * L;
    for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < n; t += (long long)gridDim.x * blockDim.x) {
        const int in = i0 + (int)(t / L), k = (int)(t % L);
        xs[(size_t)in * L + k] = x0[gk[k]];
        lam[(size_t)in * L + k] = 0.0;
        if (k == 0) {
            DevStatus z;
            memset(&z, 0, sizeof(z));
            z.max_iter = max_iter;
            z.eps_rel = eps_rel;
            z.eps_abs_pres = eps_abs;
            st[in] = z;
        }
    }
}

// Warm start of instances [i0, i0 + cnt): x_s and lambda copied from one
// start state (device slot order), e.g. a converged base-load solution.
__global__ void k_bwarm(int i0, int cnt, int L, const double *xs0, const double *lam0, double *xs, double *lam) {
    const long long n = (long long)cnt * L;
    for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < n; t += (long long)gridDim.x * blockDim.x) {
        const int in = i0 + (int)(t / L), k = (int)(t % L);
        xs[(size_t)in * L + k] = xs0[k];
        lam[(size_t)in * L + k] = lam0[k];
    }
}

__global__ void k_bfill(int cnt, int nrows, const double *b0, double *rhs) {
    const long long n = (long long)cnt * nrows;
    for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < n; t += (long long)gridDim.x * blockDim.x)
        rhs[t] = b0[t % nrows];
}

// rhs in device row order from canonical rows, or from load values.
__global__ void k_brhs_perm(int i0, int cnt, int nrows, const int *c2d, const double *src, double *rhs) {
    const long long n = (long long)cnt * nrows;
    for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < n; t += (long long)gridDim.x * blockDim.x) {
        const int j = (int)(t / nrows), r = (int)(t % nrows);
        rhs[(size_t)(i0 + j) * nrows + c2d[r]] = src[t];
    }
}

__global__ void k_brhs_loads(int i0, int cnt, int nrows, int nload, const int *rsrc, const double *rcoef,
                             const double *b0, const double *lp, const double *lq, double *rhs) {
    const long long n = (long long)cnt * nrows;
    for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < n; t += (long long)gridDim.x * blockDim.x) {
        const int j = (int)(t / nrows), r = (int)(t % nrows);
        const int s = rsrc[r];
        double v = b0[r];
        if (s >= 0) {
            const double *src = (s & 1) ? lq : lp;
            v = rcoef[r] * src[(size_t)j * nload * 3 + (s >> 1)];
        }
        rhs[(size_t)(i0 + j) * nrows + r] = v;
    }
}

// bbar = A_s^+ b per (instance, slot): slot k of device subsystem d = meta >> 8
// at position meta & 255.
__global__ void k_bbar(int i0, int cnt, int L, const int *meta, const int *sm, const int *boff,
                       const long long *pioff, const double *pinv, int nrows, const double *rhs,
                       double *bbar) {
    const long long n = (long long)cnt * L;
    for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < n; t += (long long)gridDim.x * blockDim.x) {
        const int in = i0 + (int)(t / L), k = (int)(t % L);
        const int d = meta[k] >> 8, cpos = meta[k] & 255, m = sm[d];
        const double *P = pinv + pioff[d] + (long long)cpos * m;
        const double *b = rhs + (size_t)in * nrows + boff[d];
        double acc = 0.0;
        for (int i = 0; i < m; ++i) acc += P[i] * b[i];
        bbar[(size_t)in * L + k] = acc;
    }
}

// Consistency of A_s x = b_s per instance: every rejected-row combination
// must annihilate b_s (relative to the largest |b| of the subsystem).
__global__ void k_bconsistent(int i0, int cnt, int S, const int *sm, const int *boff, const long long *toff,
                              const int *nrej, const double *Tw, int nrows, const double *rhs, int *bad) {
    const long long n = (long long)cnt * S;
    for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < n; t += (long long)gridDim.x * blockDim.x) {
        const int in = i0 + (int)(t / S), d = (int)(t % S);
        const int m = sm[d], nr = nrej[d];
        if (nr == 0) continue;
        const double *b = rhs + (size_t)in * nrows + boff[d];
        double bmax = 0.0;
        for (int i = 0; i < m; ++i) bmax = fmax(bmax, fabs(b[i]));
        const double *Tr = Tw + toff[d] + (long long)m * m;
        for (int q = 0; q < nr; ++q) {
            double acc = 0.0;
            for (int i = 0; i < m; ++i) acc += Tr[(long long)q * m + i] * b[i];
            if (!(fabs(acc) <= 1e-9 * (1.0 + bmax))) bad[in] = 1;
        }
    }
}

// ============================================================ re-centring
// Per (instance, global), instances still running: x_ref = clip((sum over the
// copies of rho x_s - lambda) - c) / (rho N)) in FP64 (the next global
// update), c~ = c + sum lambda_ref, bounds - x_ref, all in the engine layout.
// The change of variables is exact for any reference dual; at an unbounded
// global i it is lambda_ref_k = lambda_k - delta_i with delta_i = (c_i + sum
// over the copies of lambda) / N_i (FP64, kept in dref), which makes c~_i
// zero (up to rounding), and delta_i is itself small near a solution (the
// stationarity of Eq. closed_1 makes c_i + sum lambda = rho sum (x_k - x_i)).
// At a bounded global lambda_ref = lambda (delta = 0): there c~ is the bound's
// multiplier, which the clip of the global update removes, and a copy of it in
// every lambda~ would cost the FP32 iterations their small values.  c~ of the
// bounded globals also goes to cbt, in the layout of the bounds.
template <typename T>
__global__ void k_bref_globals(int n_inst, int G, int L, int K, int kshift, int NB, const int *ipos,
                               const int2 *gseg, const int *uslot, const int *bidx, const double *c64,
                               const double *lb, const double *ub, double rho, const double *xsv,
                               const double *lam, DevStatus *st, double *xref, double *dref, T *ct, T *xrf,
                               T *lbt, T *ubt, T *cbt) {
    const long long n = (long long)n_inst * G;
    for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < n; t += (long long)gridDim.x * blockDim.x) {
        const int in = (int)(t / G), i = (int)(t % G);
        if (st[in].done || ipos[in] < 0) continue;
        const int2 sg = gseg[i];
        const double *xi = xsv + (size_t)in * L, *li = lam + (size_t)in * L;
        double s = 0.0, ls = 0.0;
        for (int q = 0; q < sg.y; ++q) {
            const int k = uslot[sg.x + q];
            s += rho * xi[k] - li[k];
            ls += li[k];
        }
        double x = (s - c64[i]) / (rho * sg.y);
        x = fmin(fmax(x, lb[i]), ub[i]);
        xref[(size_t)in * G + i] = x;
        const int b = bidx[i];
        const double delta = b >= 0 ? 0.0 : (c64[i] + ls) / sg.y;
        dref[(size_t)in * G + i] = delta;
        const int pos = ipos[in], cc = pos >> kshift, sc = pos & (K - 1);
        const size_t e = ((size_t)cc * G + i) * K + sc;
        const double cs = c64[i] + (ls - sg.y * delta);
        ct[e] = (T)cs;
        xrf[e] = (T)x;
        if (b >= 0) {
            const size_t eb = ((size_t)cc * NB + b) * K + sc;
            lbt[eb] = (T)(lb[i] - x);
            ubt[eb] = (T)(ub[i] - x);
            cbt[eb] = (T)cs;
        }
        if (i == 0) st[in].pad = 1;     // shifted: unshift after the engine
    }
}

// Per (subsystem, instance), one warp: bbar~ = M (x_ref[g] + lambda_ref / rho)
// + bbar - x_ref[g], d = x_s - x_ref[g], mu = lambda - lambda_ref, lambda_ref,
// in the engine layout (lambda_ref = lambda - delta[g]).
// One subsystem of one instance by `nl` lanes starting at lane `l0` of the
// warp (v and t staged in v[], tt[]): the two FP64 products of the shifted
// bbar, written in the engine layout.
template <typename T>
__device__ __forceinline__ void bref_one(int in, bool valid, int d, int l0, int nl, int lane, const int4 h,
                                         const int4 q2, const double *F64, const int *ipos, const int *gk,
                                         const int *sch, double rho, const double *xref, const double *dref,
                                         const double *xsv, const double *lam, const double *bbar, int G, int L,
                                         int K, int kshift, int NCH, double *v, double *tt, T *bt, T *ds, T *mu,
                                         T *lref, T *xsr) {
    const int so = h.x, n = h.y, f = h.z, mode = h.w, npad = q2.y;
    const double *Fs = F64 + q2.x;
    const int ll = lane - l0;
    const double *xr = xref + (size_t)in * G, *dr = dref + (size_t)in * G;
    const double *xi = xsv + (size_t)in * L, *li = lam + (size_t)in * L, *bi = bbar + (size_t)in * L;
    if (valid)
        for (int r = ll; r < n; r += nl) v[r] = xr[gk[so + r]] + (li[so + r] - dr[gk[so + r]]) / rho;
    __syncwarp();
    if (valid)
        for (int cc = ll; cc < f; cc += nl) {
            double acc = 0.0;
            for (int r = 0; r < n; ++r) acc += Fs[(long long)cc * npad + r] * v[r];
            tt[cc] = acc;
        }
    __syncwarp();
    if (!valid) return;
    const int pos = ipos[in], cta = pos >> kshift, sc = pos & (K - 1);
    for (int r = ll; r < n; r += nl) {
        double yv = 0.0;
        for (int cc = 0; cc < f; ++cc) yv += Fs[(long long)cc * npad + r] * tt[cc];
        const double mv = mode ? yv : v[r] - yv;
        const int k = so + r;
        const double xg = xr[gk[k]];
        const int p = sch[k];
        const size_t e = (((size_t)cta * NCH + (p >> 2)) * K + sc) * 4 + (p & 3);
        const double btv = mv + bi[k] - xg;
        const double dg = dr[gk[k]];
        // the engine starts y at rho times this; the FP64 arrays hold the product
        const double yv0 = mode ? btv : -btv;
        bt[e] = sizeof(T) == 8 ? (T)(rho * yv0) : (T)yv0;
        ds[e] = (T)(xi[k] - xg);
        mu[e] = (T)dg;
        lref[e] = (T)(li[k] - dg);
        if (xsr) xsr[e] = (T)xg;
    }
}

// Per (subsystem, pair of instances), running instances only: bbar~ =
// M (x_ref[g] + lambda_ref / rho) + bbar - x_ref[g], d = x_s - x_ref[g],
// mu = 0, lambda_ref, in the engine layout.  A subsystem with at most 16
// slots and 16 factor columns takes a half-warp per instance (the FP64 pipe
// issues a warp instruction at the same cost however many lanes are active),
// a larger one the whole warp for each instance in turn.
template <typename T>
__global__ void __launch_bounds__(128) k_bref_slots(int S, int n_inst, int G, int L, int K, int kshift, int NCH,
                                                    const int *ipos, const int4 *sub, const int4 *sub2,
                                                    const double *F64, const int *gk, const int *sch,
                                                    double rho, const double *xref, const double *dref,
                                                    const double *xsv, const double *lam, const double *bbar,
                                                    const DevStatus *st, T *bt, T *ds, T *mu, T *lref,
                                                    T *xsr) {
    __shared__ double buf[4][2][OPF_MAX_NS];
    const int wl = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const long long task = (long long)blockIdx.x * 4 + wl;
    const int npair = (n_inst + 1) / 2;
    if (task >= (long long)S * npair) return;
    const int pair = (int)(task / S), d = (int)(task % S);
    const int4 h = sub[d], q2 = sub2[d];
    if (h.y <= 16 && h.z <= 16) {
        const int half = lane >> 4, in = 2 * pair + half;
        const bool valid = in < n_inst && !st[in].done && ipos[in] >= 0;
        bref_one<T>(in, valid, d, half * 16, 16, lane, h, q2, F64, ipos, gk, sch, rho, xref, dref, xsv, lam, bbar,
                    G, L, K, kshift, NCH, buf[wl][0] + half * 128, buf[wl][1] + half * 128, bt, ds, mu, lref,
                    xsr);
    } else {
        for (int q = 0; q < 2; ++q) {
            const int in = 2 * pair + q;
            if (in >= n_inst) break;
            const bool valid = !st[in].done && ipos[in] >= 0;
            bref_one<T>(in, valid, d, 0, 32, lane, h, q2, F64, ipos, gk, sch, rho, xref, dref, xsv, lam, bbar, G,
                        L, K, kshift, NCH, buf[wl][0], buf[wl][1], bt, ds, mu, lref, xsr);
            __syncwarp();
        }
    }
}

// Back to the unshifted FP64 state for instances that ran (status pad = 1):
// x_s = x_ref[g] + d, lambda = lambda_ref + mu = lambda - delta[g] + mu.
template <typename T>
__global__ void k_bunshift_slots(int n_inst, int G, int L, int K, int kshift, int NCH, const int *ipos,
                                 const int *gk, const int *sch, const double *xref, const double *dref,
                                 const T *ds, const T *mu, const DevStatus *st, double *xsv, double *lam) {
    const long long n = (long long)n_inst * L;
    for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < n; t += (long long)gridDim.x * blockDim.x) {
        const int in = (int)(t / L), k = (int)(t % L);
        if (!st[in].pad || ipos[in] < 0) continue;
        const int pos = ipos[in], cta = pos >> kshift, sc = pos & (K - 1);
        const int p = sch[k];
        const size_t e = (((size_t)cta * NCH + (p >> 2)) * K + sc) * 4 + (p & 3);
        const size_t gi = (size_t)in * G + gk[k];
        xsv[(size_t)in * L + k] = xref[gi] + (double)ds[e];
        lam[(size_t)in * L + k] = (lam[(size_t)in * L + k] - dref[gi]) + (double)mu[e];
    }
}

template <typename T>
__global__ void k_bunshift_globals(int n_inst, int G, int K, int kshift, const int *ipos, const double *xref,
                                   const T *xo, const DevStatus *st, double *x) {
    const long long n = (long long)n_inst * G;
    for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < n; t += (long long)gridDim.x * blockDim.x) {
        const int in = (int)(t / G), i = (int)(t % G);
        if (!st[in].pad || ipos[in] < 0) continue;
        const int pos = ipos[in], cta = pos >> kshift, sc = pos & (K - 1);
        x[(size_t)in * G + i] = xref[(size_t)in * G + i] + (double)xo[((size_t)cta * G + i) * K + sc];
    }
}

// Clears the shifted marks of the plan's instances (ipos >= 0); flag = 1
// while one of them still runs (and the graph condition, when a conditional
// node drives the loop).
__global__ void k_bany(int n_inst, const int *ipos, DevStatus *st, int *flag, cudaGraphConditionalHandle cond,
                       int use_cond) {
    __shared__ int any;
    if (threadIdx.x == 0) any = 0;
    __syncthreads();
    int mine = 0;
    for (int i = threadIdx.x; i < n_inst; i += blockDim.x) {
        if (ipos[i] < 0) continue;
        st[i].pad = 0;
        mine |= st[i].done ? 0 : 1;
    }
    if (mine) atomicOr(&any, 1);
    __syncthreads();
    if (threadIdx.x == 0) {
        *flag = any;
        if (use_cond) cudaGraphSetConditional(cond, any ? 1u : 0u);
    }
}

// Objective c^T x per instance (one warp each, fixed order).
__global__ void k_bobjective(int n_inst, int G, const double *c64, const double *x, double *obj) {
    const int wg = (int)((blockIdx.x * (long long)blockDim.x + threadIdx.x) >> 5), lane = threadIdx.x & 31;
    if (wg >= n_inst) return;
    double s = 0.0;
    for (int i = lane; i < G; i += 32) s += c64[i] * x[(size_t)wg * G + i];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if (lane == 0) obj[wg] = s;
}

// Prepares the polish: instances that stopped without a numeric failure run again.
__global__ void k_brestart(int n_inst, DevStatus *st, long long add_max) {
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n_inst; i += gridDim.x * blockDim.x) {
        if (st[i].numeric) continue;
        st[i].done = 0;
        st[i].converged = 0;
        if (st[i].max_iter < st[i].iter + add_max) st[i].max_iter = st[i].iter + add_max;
    }
}

// Factors packed per task: element (r, q, jpos, e) of task t from the FP64
// factor of member mb = jpos >> lp (memb[t * J + mb], -1: none), slot
// c = ((jpos & (p-1)) * nq + q) * 4 + e.
template <typename T>
__global__ void k_bpack(int n_tasks, int J, const BatchTask *tasks, const int *memb, const int4 *sub,
                        const int4 *sub2, const double *F64, T *dst) {
    const int t = blockIdx.x;
    if (t >= n_tasks) return;
    const BatchTask tk = tasks[t];
    const int n = tk.f * tk.nq * J * 4;
    for (int x = threadIdx.x; x < n; x += blockDim.x) {
        const int e = x & 3, jpos = (x >> 2) % J, q = (x / (4 * J)) % tk.nq, r = x / (4 * J * tk.nq);
        const int mb = jpos >> tk.lp, part = jpos & (tk.p - 1);
        const int d = memb[t * J + mb];
        double v = 0.0;
        if (d >= 0) {
            const int4 h = sub[d], q2 = sub2[d];
            const int cpos = (part * tk.nq + q) * 4 + e;
            if (r < h.z && cpos < h.y) v = F64[q2.x + (long long)r * q2.y + cpos];
        }
        dst[tk.foff + x] = (T)v;
    }
}

// ============================================================ launchers
static inline int bl(long long n, int t) {
    long long b = (n + t - 1) / t;
    if (b < 1) b = 1;
    if (b > 8192) b = 8192;
    return (int)b;
}

// Instantiated shapes: FP32 with factors in shared memory (K = 1, 2, 4, 8; NQ = 4),
// lambda and bbar~ in tensor memory or streamed from L2; FP64 (NQ = 2,
// K = 1, 2, 4) with factors in shared or global memory.
template <typename T>
static const void *engine_fn(int K, int nq, bool fg, bool tm) {
    if constexpr (sizeof(T) == 4) {
        if (fg || nq != 4) return nullptr;
        if (K == 1) return tm ? (const void *)k_batch_engine<float, 1, 4, false, true>
                              : (const void *)k_batch_engine<float, 1, 4, false, false>;
        if (K == 2) return tm ? (const void *)k_batch_engine<float, 2, 4, false, true>
                              : (const void *)k_batch_engine<float, 2, 4, false, false>;
        if (K == 4) return tm ? (const void *)k_batch_engine<float, 4, 4, false, true>
                              : (const void *)k_batch_engine<float, 4, 4, false, false>;
        if (K == 8) return tm ? (const void *)k_batch_engine<float, 8, 4, false, true>
                              : (const void *)k_batch_engine<float, 8, 4, false, false>;
    } else {
        if (nq != 2 || tm) return nullptr;
        if (K == 1) return fg ? (const void *)k_batch_engine<double, 1, 2, true, false> : (const void *)k_batch_engine<double, 1, 2, false, false>;
        if (K == 2) return fg ? (const void *)k_batch_engine<double, 2, 2, true, false> : (const void *)k_batch_engine<double, 2, 2, false, false>;
        if (K == 4) return fg ? (const void *)k_batch_engine<double, 4, 2, true, false> : (const void *)k_batch_engine<double, 4, 2, false, false>;
    }
    return nullptr;
}

template <typename T>
int batch_engine_prepare(int K, int nq, bool fg, bool tm, unsigned bytes) {
    const void *fn = engine_fn<T>(K, nq, fg, tm);
    if (!fn) return -1;
    return allow_dynamic_smem(fn, bytes);
}

template <typename T>
int batch_engine_launch(const BatchArgs<T> &a, int nq, bool fg, int ctas, int threads, unsigned bytes, int n_iters,
                        int check_every, cudaStream_t s) {
    const void *fn = engine_fn<T>(a.K, nq, fg, a.tm != 0);
    if (!fn) return -1;
    BatchArgs<T> aa = a;
    void *args[] = {(void *)&aa, (void *)&n_iters, (void *)&check_every};
    return cudaLaunchKernel(fn, dim3(ctas), dim3(threads), args, bytes, s) == cudaSuccess ? 0 : -1;
}

template <typename T>
int batch_engine_max_ctas_per_sm(int K, int nq, bool fg, bool tm, int threads, unsigned bytes) {
    const void *fn = engine_fn<T>(K, nq, fg, tm);
    if (!fn) return -1;
    int n = 0;
    return cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, fn, threads, bytes) == cudaSuccess ? n : -1;
}

template int batch_engine_prepare<float>(int, int, bool, bool, unsigned);
template int batch_engine_prepare<double>(int, int, bool, bool, unsigned);
template int batch_engine_launch<float>(const BatchArgs<float> &, int, bool, int, int, unsigned, int, int,
                                        cudaStream_t);
template int batch_engine_launch<double>(const BatchArgs<double> &, int, bool, int, int, unsigned, int, int,
                                         cudaStream_t);
template int batch_engine_max_ctas_per_sm<float>(int, int, bool, bool, int, unsigned);
template int batch_engine_max_ctas_per_sm<double>(int, int, bool, bool, int, unsigned);

void launch_binit(int i0, int cnt, int L, const int *gk, const double *x0, double *xs, double *lam,
                  DevStatus *st, long long max_iter, double eps_rel, double eps_abs, cudaStream_t s) {
    k_binit<<<bl((long long)cnt * L, 256), 256, 0, s>>>(i0, cnt, L, gk, x0, xs, lam, st, max_iter, eps_rel, eps_abs);
}

void launch_bwarm(int i0, int cnt, int L, const double *xs0, const double *lam0, double *xs, double *lam,
                  cudaStream_t s) {
    k_bwarm<<<bl((long long)cnt * L, 256), 256, 0, s>>>(i0, cnt, L, xs0, lam0, xs, lam);
}

void launch_bfill(int cnt, int nrows, const double *b0, double *rhs, cudaStream_t s) {
    k_bfill<<<bl((long long)cnt * nrows, 256), 256, 0, s>>>(cnt, nrows, b0, rhs);
}

void launch_brhs_perm(int i0, int cnt, int nrows, const int *c2d, const double *src, double *rhs, cudaStream_t s) {
    k_brhs_perm<<<bl((long long)cnt * nrows, 256), 256, 0, s>>>(i0, cnt, nrows, c2d, src, rhs);
}

void launch_brhs_loads(int i0, int cnt, int nrows, int nload, const int *rsrc, const double *rcoef,
                       const double *b0, const double *lp, const double *lq, double *rhs, cudaStream_t s) {
    k_brhs_loads<<<bl((long long)cnt * nrows, 256), 256, 0, s>>>(i0, cnt, nrows, nload, rsrc, rcoef, b0, lp, lq, rhs);
}

void launch_bbar(int i0, int cnt, int L, const int *meta, const int *sm, const int *boff, const long long *pioff,
                 const double *pinv, int nrows, const double *rhs, double *bbar, cudaStream_t s) {
    k_bbar<<<bl((long long)cnt * L, 256), 256, 0, s>>>(i0, cnt, L, meta, sm, boff, pioff, pinv, nrows, rhs, bbar);
}

void launch_bconsistent(int i0, int cnt, int S, const int *sm, const int *boff, const long long *toff,
                        const int *nrej, const double *Tw, int nrows, const double *rhs, int *bad, cudaStream_t s) {
    k_bconsistent<<<bl((long long)cnt * S, 128), 128, 0, s>>>(i0, cnt, S, sm, boff, toff, nrej, Tw, nrows, rhs, bad);
}

template <typename T>
void launch_bref(int n_inst, int S, int G, int L, int K, int kshift, int NCH, int NB, const int *ipos,
                 const int2 *gseg, const int *uslot, const int *bidx, const double *c64, const double *lb,
                 const double *ub, double rho, const double *xsv, const double *lam, DevStatus *st,
                 double *xref, double *dref, T *ct, T *xrf, T *lbt, T *ubt, T *cbt, const int4 *sub,
                 const int4 *sub2, const double *F64, const int *gk, const int *sch, const double *bbar, T *bt,
                 T *ds, T *mu, T *lref, T *xsr, cudaStream_t s) {
    k_bref_globals<T><<<bl((long long)n_inst * G, 256), 256, 0, s>>>(n_inst, G, L, K, kshift, NB, ipos, gseg, uslot,
                                                                    bidx, c64, lb, ub, rho, xsv, lam, st, xref,
                                                                    dref, ct, xrf, lbt, ubt, cbt);
    const long long warps = (long long)S * ((n_inst + 1) / 2);
    k_bref_slots<T><<<(int)((warps + 3) / 4), 128, 0, s>>>(S, n_inst, G, L, K, kshift, NCH, ipos, sub, sub2, F64,
                                                           gk, sch, rho, xref, dref, xsv, lam, bbar, st, bt, ds, mu,
                                                           lref, xsr);
}

template <typename T>
void launch_bunshift(int n_inst, int G, int L, int K, int kshift, int NCH, const int *ipos, const int *gk,
                     const int *sch, const double *xref, const double *dref, const T *ds, const T *mu, const T *xo,
                     const DevStatus *st, double *xsv, double *lam, double *x, cudaStream_t s) {
    k_bunshift_slots<T><<<bl((long long)n_inst * L, 256), 256, 0, s>>>(n_inst, G, L, K, kshift, NCH, ipos, gk, sch,
                                                                      xref, dref, ds, mu, st, xsv, lam);
    k_bunshift_globals<T><<<bl((long long)n_inst * G, 256), 256, 0, s>>>(n_inst, G, K, kshift, ipos, xref, xo, st, x);
}

template void launch_bref<float>(int, int, int, int, int, int, int, int, const int *, const int2 *, const int *,
                                 const int *, const double *, const double *, const double *, double,
                                 const double *, const double *, DevStatus *, double *, double *, float *,
                                 float *, float *, float *, float *, const int4 *, const int4 *, const double *,
                                 const int *, const int *, const double *, float *, float *, float *, float *,
                                 float *, cudaStream_t);
template void launch_bref<double>(int, int, int, int, int, int, int, int, const int *, const int2 *, const int *,
                                  const int *, const double *, const double *, const double *, double,
                                  const double *, const double *, DevStatus *, double *, double *, double *,
                                  double *, double *, double *, double *, const int4 *, const int4 *, const double *,
                                  const int *, const int *, const double *, double *, double *, double *,
                                  double *, double *, cudaStream_t);
template void launch_bunshift<float>(int, int, int, int, int, int, const int *, const int *, const int *,
                                     const double *, const double *, const float *, const float *, const float *,
                                     const DevStatus *, double *, double *, double *, cudaStream_t);
template void launch_bunshift<double>(int, int, int, int, int, int, const int *, const int *, const int *,
                                      const double *, const double *, const double *, const double *,
                                      const double *, const DevStatus *, double *, double *, double *,
                                      cudaStream_t);

void launch_bany(int n_inst, const int *ipos, DevStatus *st, int *flag, cudaGraphConditionalHandle cond,
                 int use_cond, cudaStream_t s) {
    k_bany<<<1, 1024, 0, s>>>(n_inst, ipos, st, flag, cond, use_cond);
}

void launch_bobjective(int n_inst, int G, const double *c64, const double *x, double *obj, cudaStream_t s) {
    k_bobjective<<<bl((long long)n_inst * 32, 256), 256, 0, s>>>(n_inst, G, c64, x, obj);
}

void launch_brestart(int n_inst, DevStatus *st, long long add_max, cudaStream_t s) {
    k_brestart<<<bl(n_inst, 256), 256, 0, s>>>(n_inst, st, add_max);
}

template <typename T>
void launch_bpack(int n_tasks, int J, const BatchTask *tasks, const int *memb, const int4 *sub, const int4 *sub2,
                  const double *F64, T *dst, cudaStream_t s) {
    if (n_tasks > 0) k_bpack<T><<<n_tasks, 256, 0, s>>>(n_tasks, J, tasks, memb, sub, sub2, F64, dst);
}
template void launch_bpack<float>(int, int, const BatchTask *, const int *, const int4 *, const int4 *,
                                  const double *, float *, cudaStream_t);
template void launch_bpack<double>(int, int, const BatchTask *, const int *, const int4 *, const int4 *,
                                   const double *, double *, cudaStream_t);

}  // namespace opf
