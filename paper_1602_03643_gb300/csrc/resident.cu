// Resident solves: one cooperative launch runs a whole linear solve.
//
// A Krylov iteration on a few thousand to a few hundred thousand rows moves so
// little data that a kernel per operation costs far more in launch gaps, block
// reductions and last-block tickets (4-7 us each, measured) than in memory traffic.
// Here every block keeps a contiguous chunk of rows for the whole solve: its part of
// the matrix and of every vector sits in shared memory, only what neighbours gather
// goes through L2.  The blocks meet at a counter in L2 (1.25 us at 152 blocks,
// measured; a flag per block that every block polls took 3.2 us, its 23,000 polls
// contending for a few lines).  A grid-wide sum is one such meeting: the blocks'
// partial sums are written before it and added by every block in block order after
// it, so all blocks hold the same bits and take the same decisions without a
// broadcast.  Matrix entries that come from L2 (the coarser multigrid levels) are
// fetched before a meeting, the gathers that need the other blocks' data after it.
// The launch is cooperative: all blocks are resident, so every wait ends; each is
// bounded all the same (OASIS_EWAIT).
//
// Bound by latency: a Jacobi CG iteration on 68,921 rows takes 5.3 us, of which the
// meeting 1.0, the block's and the blocks' partial sums 0.5 + 1.0, the scalars 0.7 and
// the product with its vector updates 2.1 (separate kernel: 15 us).  Whole steps, us,
// separate kernels against resident: 1,089 dofs float64 multigrid 1500 / 660; 2,184
// dofs float64 Jacobi, eager, host arrays 4020 / 1230; 68,921 mixed Jacobi 5830 / 1900;
// 117,600 with two scalars and the consistent-mass update (multigrid pressure separate)
// 3040 / 1940; 160,680 (triangles) mixed multigrid 2120 / 1430.  One thread per row (where there are
// rows enough for the threads) took 2.1 us in the product above where 4 lanes per row
// took 3.5: fewer shuffles and a full warp in the row's vector updates.  Tried and
// not kept: one 16-block cluster with its hardware barrier (0.3 us) for small systems
// (1,089 rows 611 -> 639, 6,859 rows 523 -> 622 us per step: 16 SMs take longer over
// the rows than the cheaper meetings save).
#include <algorithm>
#include <type_traits>

#include "kern.cuh"
#include "resident.cuh"

namespace oasis {

namespace {

// sweeps of one solve at most, as in the separate kernels (step.cu)
constexpr int kResMaxSweeps = 1000;

template <class P>
constexpr int res_threads() {
    return 512;
}

// ------------------------------------------------------------------ values
__device__ __forceinline__ void zero(float& a) { a = 0.f; }
__device__ __forceinline__ void zero(double& a) { a = 0.0; }
__device__ __forceinline__ void zero(ff& a) { a = {0.f, 0.f}; }
__device__ __forceinline__ void add_to(float& a, float b) { a += b; }
__device__ __forceinline__ void add_to(double& a, double b) { a += b; }
// lazily normalised: the high parts by an error-free two-sum, errors and low parts in
// float (a chain of additions then waits for one float addition each, not for twenty)
__device__ __forceinline__ void add_to(ff& a, ff b) {
    const ff t = two_sum(a.hi, b.hi);
    a.hi = t.hi;
    a.lo += t.lo + b.lo;
}
__device__ __forceinline__ float shfl(float a, int o) { return __shfl_xor_sync(0xffffffffu, a, o); }
__device__ __forceinline__ double shfl(double a, int o) { return __shfl_xor_sync(0xffffffffu, a, o); }
__device__ __forceinline__ ff shfl(ff a, int o) { return acc_shfl(a, o); }
__device__ __forceinline__ float normal(float a) { return a; }
__device__ __forceinline__ double normal(double a) { return a; }
__device__ __forceinline__ ff normal(ff a) { return lazy_norm(a); }
template <class A>
__device__ __forceinline__ A wider(float a) { return {a, 0.f}; }
template <class A>
__device__ __forceinline__ A wider(ff a) { return a; }

template <class T>
using LiteA = typename LiteAcc<T>::type;

// The Krylov scalars.  Float64 path: float64.  Mixed path: what one iteration hands to
// the next is exact (a grid-wide sum, float-float as it comes) or derived in float64 by
// the block's last warp while the others go on; the coefficients that the vectors wait
// for are float32 and come from quotients in float-float (a float64 operation occupies
// the pipe for 64 cycles: a CG iteration with all of its scalars in float64 took 6.0 us
// where it takes 5.3).  The sums may be as small as float32 holds: they are brought to
// the order of one by a power of two first, and 1 / rho, which may be beyond float32, is
// formed of the scaled rho only.
__device__ __forceinline__ double x_hi(double a) { return a; }
__device__ __forceinline__ float x_hi(ff a) { return a.hi; }
__device__ __forceinline__ double x_mul(double a, double b) { return a * b; }
__device__ __forceinline__ ff x_mul(ff a, ff b) {
    ff p = two_prod(a.hi, b.hi);
    p.lo = __fmaf_rn(a.hi, b.lo, __fmaf_rn(a.lo, b.hi, p.lo));
    return fast_two_sum(p.hi, p.lo);
}
__device__ __forceinline__ double x_div(double a, double b) { return a / b; }
// to ~float-float accuracy: one correction by the exact remainder of the float
// quotient (Dekker 1971)
__device__ __forceinline__ ff x_div(ff a, ff b) {
    const float q = a.hi / b.hi;
    const ff p = two_prod(q, b.hi);
    const float rem = ((a.hi - p.hi) - p.lo) + __fmaf_rn(-q, b.lo, a.lo);
    return fast_two_sum(q, rem / b.hi);
}
// a power of two that brings a to the order of one (zero, infinity and NaN stay)
__device__ __forceinline__ double unit_of(double) { return 1.0; }
__device__ __forceinline__ float unit_of(ff a) {
    return __uint_as_float((254u << 23) - min(__float_as_uint(a.hi) & 0x7f800000u, 253u << 23));
}
__device__ __forceinline__ double x_scaled(double a, double) { return a; }
__device__ __forceinline__ ff x_scaled(ff a, float s) { return {a.hi * s, a.lo * s}; }
// a / b as a value
template <class X>
__device__ __forceinline__ auto quotient(X a, X b) {
    const auto s = unit_of(b);
    return x_hi(x_div(x_scaled(a, s), x_scaled(b, s)));
}
// the float64 limit of a sum's stopping test in the sum's leading type: not above it
__device__ __forceinline__ double limit_of(double, double d) { return d; }
__device__ __forceinline__ float limit_of(float, double d) { return __double2float_rd(d); }

// What a CG iteration hands to the next: rho = <r, u> and 1 / alpha.
template <class X>
struct CgCarry;
template <>
struct CgCarry<double> {
    double rho, alpha, irho, ialpha;
    // sweep's first product: alpha = rho / <w, u>
    __device__ __forceinline__ double start(double g, double wu) {
        rho = g;
        return alpha = g / wu;
    }
    // beta = g / rho, alpha = g / (<w, u> - beta g / alpha_old); false: a breakdown
    __device__ __forceinline__ bool next(double g, double wu, double& al, double& be) {
        be = rho == 0.0 ? 0.0 : g * irho;
        const double den = alpha == 0.0 ? 0.0 : wu - be * g * ialpha;
        const bool ok = den > 0.0 && isfinite(den) && isfinite(g) && rho != 0.0;
        al = alpha = ok ? g / den : 0.0;
        rho = g;
        return ok;
    }
    // between two iterations, off the critical path, by one warp: its lanes take a
    // quotient each; g, wu: the sums that start or next had
    __device__ __forceinline__ void carry(int lane, bool, double, double) {
        const double q = 1.0 / (lane == 0 ? rho : alpha);
        if (lane == 0 && rho != 0.0) irho = q;
        if (lane == 1 && alpha != 0.0) ialpha = q;
    }
};
template <>
struct CgCarry<ff> {
    ff rho, irho, ialpha;                // irho: of rho times unit; ialpha: of ia
    float unit;
    double ia;                           // 1 / alpha
    __device__ __forceinline__ float start(ff g, ff wu) { return quotient(g, wu); }
    __device__ __forceinline__ bool next(ff g, ff wu, float& al, float& be) {
        const ff gs = x_scaled(g, unit), b = x_mul(gs, irho);
        const ff den = ff_sub(x_scaled(wu, unit), x_mul(x_mul(b, gs), ialpha));
        const bool ok = den.hi > 0.f && isfinite(den.hi) && isfinite(g.hi) && rho.hi != 0.f;
        al = ok ? x_div(gs, den).hi : 0.f;
        be = rho.hi != 0.f ? b.hi : 0.f;
        return ok;
    }
    // 1 / alpha = <w, u> / g - (g / rho) / alpha_old
    __device__ __forceinline__ void carry(int lane, bool first, ff g, ff wu) {
        const float s = unit_of(g);
        const ff num = lane == 0 ? wu : lane == 1 ? g : ff{1.f, 0.f};
        const ff den = lane == 0 ? g : lane == 1 ? rho : x_scaled(g, s);
        const double q = first && lane == 1 ? 0.0 : acc_double(num) / acc_double(den);
        const double q1 = __shfl_sync(0xffffffffu, q, 1);
        const double next_ia = first ? q : q - q1 * ia;
        const ff f = ff_from_double(lane == 0 ? next_ia : q);
        if (lane == 0) {
            ia = next_ia;
            ialpha = f;
            rho = g;
            unit = s;
        }
        if (lane == 2) irho = f;
    }
};
// alpha / omega of a BiCGStab iteration, off the critical path: alpha = rho / <rhat, v>,
// omega = <t, s> / <t, t>
__device__ __forceinline__ double alpha_over_omega(double rho, double rv, double ts, double tt) {
    return (rho / rv) / (ts / tt);
}
__device__ __forceinline__ ff alpha_over_omega(ff rho, ff rv, ff ts, ff tt) {
    // float32's range: the products stay within float64's
    return ff_from_double((acc_double(rho) * acc_double(tt)) / (acc_double(rv) * acc_double(ts)));
}

// ------------------------------------------------------------------ meetings
__device__ __forceinline__ void add_release(uint32_t* p) {
    asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(p) : "memory");
}
__device__ __forceinline__ uint32_t ld_acquire(const uint32_t* p) {
    uint32_t v;
    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}

// Every block's writes so far become visible to every block; false in all threads
// of a block whose wait ran out.  goal: arrivals that the meeting waits for.  The limit
// of a wait, if not the usual one, stands behind the counter (resident_set_wait).
__device__ __forceinline__ bool grid_barrier(uint32_t* count, uint32_t goal) {
    __syncthreads();
    bool ok = true;
    if (threadIdx.x == 0) {
        add_release(count);
        if ((int32_t)(ld_acquire(count) - goal) < 0) {
            const long long t0 = clock64(), set = *reinterpret_cast<const volatile long long*>(count + 2),
                            limit = set > 0 ? set : kBarrierLimitCycles;
            while ((int32_t)(ld_acquire(count) - goal) < 0)
                if (clock64() - t0 > limit) {
                    ok = false;
                    break;
                }
        }
    }
    return __syncthreads_and(ok) != 0;
}

// K values per lane summed over the warp; value k ends up in the lanes whose
// leading log2(K) bits are k.  Each step halves the values a lane carries by
// swapping half of them with its partner, so K values take K - 1 + log2(32 / K)
// additions instead of 5 K.
template <int K, class A>
__device__ __forceinline__ A warp_sums(A (&v)[K]) {
    const int lane = threadIdx.x & 31;
    int o = 16;
#pragma unroll
    for (int m = K; m > 1; m /= 2, o /= 2) {
        const bool up = (lane & o) != 0;
#pragma unroll
        for (int i = 0; i < m / 2; ++i) {
            const A give = up ? v[i] : v[i + m / 2];
            A keep = up ? v[i + m / 2] : v[i];
            add_to(keep, shfl(give, o));
            v[i] = keep;
        }
    }
#pragma unroll
    for (; o > 0; o /= 2) add_to(v[0], shfl(v[0], o));
    return v[0];
}

struct GridMeet {
    ResidentSync m;
    uint32_t goal = 0, parity = 0;
    __device__ explicit GridMeet(const ResidentSync& s) : m(s) {}

    // arrivals that the next meeting waits for
    __device__ __forceinline__ uint32_t next() {
        parity ^= 1u;
        return goal += gridDim.x;
    }
    __device__ __forceinline__ bool barrier() { return grid_barrier(m.count, next()); }

    // Values k of NV, `count` parts each, summed by the block's first warps (K values
    // per warp): out(k, sum) in one lane of the warp.
    template <int NV, class A, class Part, class Out>
    static __device__ __forceinline__ void add_parts(int count, Part&& part, Out&& out) {
        constexpr int K = NV <= 4 ? 1 : NV <= 8 ? 2 : 4;
        const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = (int)(blockDim.x >> 5);
        for (int g = wid; g * K < NV; g += nw) {
            A acc[K];
#pragma unroll
            for (int k = 0; k < K; ++k) acc_zero(acc[k]);
            for (int b = lane; b < count; b += 32) {
#pragma unroll
                for (int k = 0; k < K; ++k)
                    if (g * K + k < NV) add_to(acc[k], part(g * K + k, b));
            }
            const A sum = normal(warp_sums<K, A>(acc));
            constexpr int per = 32 / K;
            if (lane % per == 0 && g * K + lane / per < NV) out(g * K + lane / per, sum);
        }
    }

    // tot[k] = sum over the grid of v[k] (the same bits in every block), valid for
    // all threads on return, in a fixed order: over the block, then over the blocks,
    // in A (float-float or float64; float values first over a warp in float).  Only
    // the lanes lg = (k % NR) % G of each group of G lanes hold values k that are not
    // zero, and only the first `groups` groups hold any.
    template <int NV, int NR, int G, class T, class A>
    __device__ __forceinline__ bool sum(T (&v)[NV], A* tot, int groups) {
        static_assert(NV <= kResValues, "too many values");
        const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = (int)(blockDim.x >> 5);
        A* part = reinterpret_cast<A*>(m.partial) + (size_t)(parity ^ 1u) * kResValues * gridDim.x;
        auto store = [&](int k, A x) { part[(size_t)k * gridDim.x + blockIdx.x] = x; };
        if constexpr (sizeof(T) == 8 && std::is_same<T, double>::value) {
            // float64: an addition costs a warp 64 cycles however many lanes take part,
            // so the values go through shared memory to few warps
            constexpr int kSlots = G == 1 ? res_threads<Fp64>() : res_threads<Fp64>() / G;
            __shared__ double sh[NV][kSlots];
            const int slot = threadIdx.x / G, lg = threadIdx.x % G;
            if (slot < groups)
#pragma unroll
                for (int k = 0; k < NV; ++k)
                    if ((k % NR) % G == lg) sh[k][slot] = v[k];
            __syncthreads();
            add_parts<NV, A>(min(groups, (int)blockDim.x / G), [&](int k, int b) { return sh[k][b]; }, store);
        } else {
            __shared__ T sh[NV][32];
            if constexpr (NV > 4) {
                constexpr int K = NV <= 8 ? 8 : 16, per = 32 / K;
                T w[K];
#pragma unroll
                for (int k = 0; k < K; ++k) {
                    if (k < NV) w[k] = v[k];
                    else zero(w[k]);
                }
                const T x = warp_sums<K, T>(w);
                if (lane % per == 0 && lane / per < NV) sh[lane / per][wid] = x;
            } else {
#pragma unroll
                for (int k = 0; k < NV; ++k) {
                    T w[1] = {v[k]};
                    const T x = warp_sums<1, T>(w);
                    if (lane == 0) sh[k][wid] = x;
                }
            }
            __syncthreads();
            add_parts<NV, A>(nw, [&](int k, int b) { return wider<A>(sh[k][b]); }, store);
        }
        if (!barrier()) return false;
        add_parts<NV, A>((int)gridDim.x, [&](int k, int b) { return lite_load(&part[(size_t)k * gridDim.x + b]); },
                         [&](int k, A x) { tot[k] = x; });
        __syncthreads();
        return true;
    }

    // The last block to leave clears the counter for the next launch (every block
    // has passed its last wait by then).
    __device__ __forceinline__ void leave() {
        __syncthreads();
        if (threadIdx.x == 0 && take_last_ticket(m.ticket)) {
            *m.count = 0u;
            *m.ticket = 0u;
        }
    }
};

// Rows of this block.
struct Chunk {
    int lo = 0, hi = 0;
    Chunk() = default;
    __device__ explicit Chunk(int n) {
        const int c = (n + (int)gridDim.x - 1) / (int)gridDim.x;
        lo = min(n, c * (int)blockIdx.x);
        hi = min(n, lo + c);
    }
};

__device__ __forceinline__ float wide(uint16_t b) { return __uint_as_float((uint32_t)b << 16); }
__device__ __forceinline__ double wide(double v) { return v; }

// ------------------------------------------------------------------ products
// sum_j a_ij x(j) for the rows [0, count) of a block, N values per column: G lanes
// per row and M entries per lane in flight.  ptr(i) is row i's first entry, entry(q,
// j, a) reads an entry's column and value, gather(j) the column's operand, add(acc,
// value, operand) adds their product; epi(i, lane in group, sums) has the sums in
// every lane of the row's group.  meet() runs once, after the first entries have been
// fetched and before the first gather.  VA: type of the values.
template <int G, int M, int N, class A, class VA, class Ptr, class Entry, class Meet, class Gather, class Add,
          class Epi>
__device__ __forceinline__ bool res_rows(int count, Ptr&& ptr, Entry&& entry, Meet&& meet, Gather&& gather, Add&& add,
                                         Epi&& epi) {
    const int lg = threadIdx.x & (G - 1), step = (int)blockDim.x / G;
    // a warp's lanes walk on together: i is the group's row, w the warp's first one
    int i = (int)threadIdx.x / G, w = (int)(threadIdx.x & ~31u) / G;
    int32_t q = 0, e = 0, j[M];
    VA av[M];
    auto row = [&] {
        q = i < count ? ptr(i) + lg : 0;
        e = i < count ? ptr(i + 1) : 0;
    };
    auto fetch = [&] {
#pragma unroll
        for (int k = 0; k < M; ++k) {
            j[k] = -1;
            if (q + k * G < e) entry(q + k * G, j[k], av[k]);
        }
    };
    row();
    fetch();
    if (!meet()) return false;
    while (w < count) {
        A acc[N];
#pragma unroll
        for (int c = 0; c < N; ++c) zero(acc[c]);
        for (;;) {
            decltype(gather(0)) g[M];
#pragma unroll
            for (int k = 0; k < M; ++k)
                if (j[k] >= 0) g[k] = gather(j[k]);
#pragma unroll
            for (int k = 0; k < M; ++k)
                if (j[k] >= 0) add(acc, av[k], g[k]);
            q += M * G;
            if (q >= e) break;
            fetch();
        }
#pragma unroll
        for (int c = 0; c < N; ++c) {
            acc[c] = normal(acc[c]);
#pragma unroll
            for (int o = G / 2; o > 0; o >>= 1) add_to(acc[c], shfl(acc[c], o));
        }
        if (i < count) epi(i, lg, acc);
        i += step;
        w += step;
        if (w < count) {
            row();
            fetch();
        }
    }
    return true;
}

// lane groups of a block that res_rows gives rows to
template <int G>
__device__ __forceinline__ int used_groups(int rows) {
    return min((int)blockDim.x / G, rows);
}

// The block's rows of a CSR matrix: copied to shared memory (float: column and value
// side by side, one 8-byte load), or, where they do not fit there (STAGED = false),
// read from global memory.
template <class V, bool STAGED>
struct ResMatrix {
    const int32_t *rp, *ci;
    const V* av;
    int32_t e0 = 0;                      // first entry of the block's rows
    // carved from `at`; every thread of the block copies
    __device__ __forceinline__ void fill(unsigned char*& at, const ResidentPlan& pl, const Chunk& ch,
                                         const int32_t* __restrict__ g_rp, const int32_t* __restrict__ g_ci,
                                         const V* __restrict__ g_av) {
        const int count = ch.hi - ch.lo;
        e0 = count > 0 ? __ldg(g_rp + ch.lo) : 0;
        if constexpr (!STAGED) {
            rp = g_rp + ch.lo;
            ci = g_ci + e0;
            av = g_av + e0;
            return;
        }
        V* s_av = reinterpret_cast<V*>(at);
        int32_t* s_ci = reinterpret_cast<int32_t*>(at + (sizeof(V) == 4 ? 0 : (size_t)pl.entries * sizeof(V)));
        at += (size_t)pl.entries * (sizeof(V) + 4);
        int32_t* s_rp = reinterpret_cast<int32_t*>(at);
        at += (size_t)(pl.rows + 1) * 4;
        at = reinterpret_cast<unsigned char*>(((size_t)at + 15) & ~(size_t)15);
        const int32_t e1 = count > 0 ? __ldg(g_rp + ch.hi) : 0;
        for (int k = threadIdx.x; k <= count; k += blockDim.x) s_rp[k] = count > 0 ? __ldg(g_rp + ch.lo + k) - e0 : 0;
        for (int32_t k = threadIdx.x; k < e1 - e0; k += blockDim.x) {
            const int32_t j = __ldg(g_ci + e0 + k);
            const V v = __ldg(g_av + e0 + k);
            if constexpr (sizeof(V) == 4) {
                reinterpret_cast<int2*>(s_ci)[k] = make_int2(j, __float_as_int(v));
            } else {
                s_ci[k] = j;
                s_av[k] = v;
            }
        }
        rp = s_rp;
        ci = s_ci;
        av = s_av;
    }
    __device__ __forceinline__ int32_t ptr(int i) const { return STAGED ? rp[i] : __ldg(rp + i) - e0; }
    __device__ __forceinline__ void entry(int q, int32_t& j, V& v) const {
        if constexpr (!STAGED) {
            j = __ldg(ci + q);
            v = __ldg(av + q);
        } else if constexpr (sizeof(V) == 4) {
            const int2 p = reinterpret_cast<const int2*>(ci)[q];
            j = p.x;
            v = __int_as_float(p.y);
        } else {
            j = ci[q];
            v = av[q];
        }
    }
    __device__ __forceinline__ int32_t column(int q) const {
        return STAGED ? ci[sizeof(V) == 4 ? 2 * q : q] : __ldg(ci + q);
    }
};
template <class V>
__device__ __forceinline__ V* res_carve(unsigned char*& at, int count) {
    V* p = reinterpret_cast<V*>(at);
    at += ((size_t)count * sizeof(V) + 15) & ~(size_t)15;
    return p;
}
// the same on the host: bytes of a matrix and of one vector
template <class V>
size_t res_matrix_bytes(int rows, int entries) {
    return ((size_t)entries * (sizeof(V) + 4) + (size_t)(rows + 1) * 4 + 15) / 16 * 16 + 16;
}
template <class V>
size_t res_vector_bytes(int count) {
    return ((size_t)count * sizeof(V) + 15) / 16 * 16;
}

// ------------------------------------------------------------------ BiCGStab
// Scalars of the columns, the same in every block (all from grid-wide sums).
template <class V, int NR>
struct BicgScalars {
    using X = LiteA<V>;
    X tot[kResValues];
    double bb[NR], rr[NR];
    X rho[NR], rv[NR], ao[NR], rr_in[NR];   // <rhat, r>, <rhat, v>, alpha / omega, <r, r>
    V al[NR], om[NR], be[NR], stop[NR];     // stop: the inner solve ends at or below it
    int it_total[NR], col_done[NR], in_done[NR], act[NR], status;
};

// Right-preconditioned BiCGStab with Jacobi inside refinement sweeps: the method,
// the stopping tests and the counters of the separate kernels (k_bicg_*, step.cu).
// Per iteration the blocks meet four times (mixed) or five (float64): after p and
// ph; for <rhat, v>; [float64: after sh;] for <t, s> and <t, t>; and for <rhat, r> and
// <r, r> of the new residual, summed from r itself (as differences of sums that come
// with t, without a meeting of their own, they would lose the digits by which r is
// smaller than s).  The mixed path spares the meeting after sh: each neighbour's
// sh_j = d_j r_j - alpha d_j v_j is formed again from what is gathered; in float64
// the extra arithmetic would cost more than the meeting.  Published, in pub: ph,
// then (mixed) D^-1 r and D^-1 v, or (float64) sh.
template <class P, int D, int NR, int G, int M, bool STAGED>
__global__ void __launch_bounds__(res_threads<P>(), 1) k_resident_bicg(StepData<P> a, int k0, Ctl ctl,
                                                                       ResidentPlan pl, ResidentSync sy,
                                                                       Pub<typename P::V, NR>* pub) {
    using V = typename P::V;
    using S = typename P::S;
    using Acc = typename P::Acc;
    using X = LiteA<V>;
    using Pb = Pub<V, NR>;
    extern __shared__ __align__(16) unsigned char dsm[];
    __shared__ BicgScalars<V, NR> sc;
    GridMeet gm(sy);
    const Chunk ch((int)a.n);
    const int rows = ch.hi - ch.lo, count = rows * NR, tid = threadIdx.x;
    const int groups = used_groups<G>(rows);
    unsigned char* at = dsm;
    ResMatrix<V, STAGED> mat;
    mat.fill(at, pl, ch, a.rp, a.col, a.A);
    V* const r = res_carve<V>(at, pl.rows * NR);
    V* const rh = res_carve<V>(at, pl.rows * NR);
    V* const p = res_carve<V>(at, pl.rows * NR);
    V* const v = res_carve<V>(at, pl.rows * NR);
    V* const t = res_carve<V>(at, pl.rows * NR);
    V* const dl = res_carve<V>(at, pl.rows * NR);
    V* const di = res_carve<V>(at, pl.rows);
    for (int i = tid; i < rows; i += blockDim.x) di[i] = a.dinvA[ch.lo + i];
    Pb* const ph = pub;
    Pb* const q1 = pub + a.n;            // D^-1 r (mixed), sh (float64)
    Pb* const q2 = pub + 2 * a.n;        // D^-1 v (mixed)
    KrylovState* st = a.stu;
    if (tid < NR) {
        sc.bb[tid] = st->bb[k0 + tid];
        sc.rr[tid] = st->rr[k0 + tid];
        acc_zero(sc.rr_in[tid]);
        sc.col_done[tid] = st->col_done[k0 + tid];
        sc.in_done[tid] = 1;
        sc.it_total[tid] = st->it_total[k0 + tid];
        acc_zero(sc.rho[tid]);
        sc.al[tid] = sc.om[tid] = sc.be[tid] = V(0);
    }
    if (tid == 0) sc.status = st->status;
    int sweeps = st->sweeps;
    __syncthreads();
    auto any_active = [&] {
        bool any = false;
#pragma unroll
        for (int c = 0; c < NR; ++c) any |= !sc.col_done[c] && !sc.in_done[c];
        return any;
    };
    auto ptr = [&](int i) { return mat.ptr(i); };
    auto entry = [&](int q, int32_t& j, V& v) { mat.entry(q, j, v); };
    auto now = [] { return true; };
    auto add = [](V(&acc)[NR], V av, const Pb& g) {
#pragma unroll
        for (int c = 0; c < NR; ++c) acc[c] += av * g.v[c];
    };
    const int spare = (int)blockDim.x - 32;
    // position of local element e = row * NR + c in an [n][D] array
    auto pos = [&](int e) { return (size_t)(ch.lo + e / NR) * D + k0 + e % NR; };
    bool ok = true;
    for (;;) {
        // r = r0 - A Delta with float64-quality products
        {
            Acc part[NR];
#pragma unroll
            for (int c = 0; c < NR; ++c) acc_zero(part[c]);
            res_rows<G, M, NR, Acc, V>(
                rows, ptr, entry, now,
                [&](int j) {
                    Vec<S, NR> g;
#pragma unroll
                    for (int c = 0; c < NR; ++c) g.v[c] = a.du[(size_t)j * D + k0 + c];
                    return g;
                },
                [](Acc(&acc)[NR], V av, const Vec<S, NR>& g) {
#pragma unroll
                    for (int c = 0; c < NR; ++c) lazy_add_prod(acc[c], g.v[c], av);
                },
                [&](int i, int lg, const Acc(&acc)[NR]) {
#pragma unroll
                    for (int c = 0; c < NR; ++c) {
                        if (c % G != lg || sc.col_done[c]) continue;
                        const int e = i * NR + c;
                        const V rv = s_v(s_sub(a.r0[pos(e)], s_of_acc(acc[c])));
                        r[e] = rh[e] = rv;
                        dl[e] = 0;
                        acc_prod(part[c], rv, rv);
                    }
                });
            ok = gm.template sum<NR, NR, G, Acc, Acc>(part, sc.tot, used_groups<G>(rows));
        }
        if (!ok) break;
        if (tid < NR && !sc.col_done[tid]) {
            const double rr = acc_double(sc.tot[tid]);
            sc.rr[tid] = rr;
            if (!isfinite(rr)) {
                sc.status = OASIS_ENAN;
                sc.col_done[tid] = 1;
            } else if (rr <= ctl.rtol2 * sc.bb[tid]) {
                sc.col_done[tid] = 1;
            } else if (sc.it_total[tid] >= ctl.max_it || sweeps >= kResMaxSweeps) {
                sc.status = OASIS_ENOTCONV;
                sc.col_done[tid] = 1;
            } else {
                sc.in_done[tid] = 0;
                sc.rho[tid] = sc.rr_in[tid] = sc.tot[tid];
                sc.stop[tid] = limit_of(V(0), fmax(ctl.inner2 * rr, ctl.abs2 * sc.bb[tid]));
            }
        }
        ++sweeps;
        __syncthreads();
        if (!any_active()) break;
        // p = r, ph = D^-1 p
        for (int e = tid; e < count; e += blockDim.x) {
            const int gi = ch.lo + e / NR, c = e % NR;
            const V rv = r[e], dr = di[e / NR] * rv;
            p[e] = rv;
            ph[gi].v[c] = dr;
            if constexpr (P::mixed) q1[gi].v[c] = dr;
        }
        for (int it_in = 0;;) {
            if (!(ok = gm.barrier())) break;
            // v = A ph, alpha = rho / <rhat, v>
            {
                V part[NR] = {};
                res_rows<G, M, NR, V, V>(
                    rows, ptr, entry, now, [&](int j) { return ph[j]; }, add,
                    [&](int i, int lg, const V(&acc)[NR]) {
#pragma unroll
                        for (int c = 0; c < NR; ++c) {
                            if (c % G != lg) continue;
                            const int e = i * NR + c;
                            v[e] = acc[c];
                            if constexpr (P::mixed) q2[ch.lo + i].v[c] = di[i] * acc[c];
                            part[c] += rh[e] * acc[c];
                        }
                    });
                if (!(ok = gm.template sum<NR, NR, G, V, X>(part, sc.tot, groups))) break;
            }
            if (tid < NR) {
                int act = !sc.col_done[tid] && !sc.in_done[tid];
                if (act) {
                    const X rv = sc.tot[tid];
                    if (x_hi(rv) == V(0) || !isfinite(x_hi(rv))) {
                        sc.in_done[tid] = 1;      // breakdown: restart from the float64-quality residual
                        sc.it_total[tid] += 1;
                        sc.al[tid] = V(0);
                        act = 0;
                    } else {
                        sc.rv[tid] = rv;
                        sc.al[tid] = quotient(sc.rho[tid], rv);
                    }
                }
                sc.act[tid] = act;
            }
            __syncthreads();
            if (!any_active()) break;
            if constexpr (!P::mixed) {
                for (int e = tid; e < count; e += blockDim.x)
                    q1[ch.lo + e / NR].v[e % NR] = di[e / NR] * (r[e] - sc.al[e % NR] * v[e]);
                if (!(ok = gm.barrier())) break;
            }
            // t = A sh, omega = <t, s> / <t, t>
            {
                V part[2 * NR] = {};
                V al[NR];
#pragma unroll
                for (int c = 0; c < NR; ++c) al[c] = sc.al[c];
                res_rows<G, (P::mixed && NR > 1 ? (M + 1) / 2 : M), NR, V, V>(
                    rows, ptr, entry, now,
                    [&](int j) {
                        Pb g = q1[j];
                        if constexpr (P::mixed) {
                            const Pb h = q2[j];
#pragma unroll
                            for (int c = 0; c < NR; ++c) g.v[c] -= al[c] * h.v[c];
                        }
                        return g;
                    },
                    add,
                    [&](int i, int lg, const V(&acc)[NR]) {
#pragma unroll
                        for (int c = 0; c < NR; ++c) {
                            if (c % G != lg) continue;
                            const int e = i * NR + c;
                            const V tv = acc[c], sv = r[e] - al[c] * v[e];
                            t[e] = tv;
                            part[c] += tv * sv;
                            part[NR + c] += tv * tv;
                        }
                    });
                if (!(ok = gm.template sum<2 * NR, NR, G, V, X>(part, sc.tot, groups))) break;
            }
            if (tid < NR && sc.act[tid]) {
                const X ts = sc.tot[tid], tt = sc.tot[NR + tid];
                sc.om[tid] = x_hi(tt) > V(0) && isfinite(x_hi(tt)) ? quotient(ts, tt) : V(0);
            }
            __syncthreads();
            // off the critical path, by threads of the last warp
            if (tid >= spare && tid < spare + NR) {
                const int c = tid - spare;
                if (sc.act[c]) sc.ao[c] = alpha_over_omega(sc.rho[c], sc.rv[c], sc.tot[c], sc.tot[NR + c]);
            }
            // delta += alpha ph + omega sh, r = s - omega t, <rhat, r>, <r, r>
            {
                V part[2 * NR] = {};
                for (int i = tid / G; i < rows; i += (int)blockDim.x / G) {
                    const int lg = tid % G;
                    const V d = di[i];
#pragma unroll
                    for (int c = 0; c < NR; ++c) {
                        if (c % G != lg || !sc.act[c]) continue;
                        const int e = i * NR + c;
                        const V al = sc.al[c], om = sc.om[c], sv = r[e] - al * v[e];
                        dl[e] += al * (d * p[e]) + om * (d * sv);
                        const V rv = sv - om * t[e];
                        r[e] = rv;
                        part[c] += rh[e] * rv;
                        part[NR + c] += rv * rv;
                    }
                }
                if (!(ok = gm.template sum<2 * NR, NR, G, V, X>(part, sc.tot, groups))) break;
            }
            if (tid < NR && sc.act[tid]) {
                const X rho = sc.tot[tid], rr = sc.tot[NR + tid], old = sc.rho[tid];
                sc.it_total[tid] += 1;
                if (x_hi(old) != V(0) && sc.om[tid] != V(0)) {
                    const auto s = unit_of(old);
                    sc.be[tid] = x_hi(x_div(x_mul(x_scaled(rho, s), sc.ao[tid]), x_scaled(old, s)));
                } else {
                    sc.be[tid] = V(0);
                }
                sc.rho[tid] = rho;
                sc.rr_in[tid] = rr;
                if (!isfinite(x_hi(rr)) || x_hi(rr) <= sc.stop[tid] || sc.om[tid] == V(0) || x_hi(rho) == V(0) ||
                    sc.it_total[tid] >= ctl.max_it || it_in + 1 >= ctl.sweep_cap)
                    sc.in_done[tid] = 1;
            }
            ++it_in;
            __syncthreads();
            if (!any_active()) break;
            // p = r + beta (p - omega v), ph = D^-1 p
            for (int e = tid; e < count; e += blockDim.x) {
                const int row = e / NR, c = e % NR;
                if (!sc.act[c]) continue;
                const V d = di[row], rv = r[e], pv = rv + sc.be[c] * (p[e] - sc.om[c] * v[e]);
                p[e] = pv;
                ph[ch.lo + row].v[c] = d * pv;
                if constexpr (P::mixed) q1[ch.lo + row].v[c] = d * rv;
            }
        }
        if (!ok) break;
        // Delta += delta
        __syncthreads();
        for (int e = tid; e < count; e += blockDim.x)
            if (!sc.col_done[e % NR]) {
                const size_t o = pos(e);
                a.du[o] = s_addv(a.du[o], dl[e]);
            }
        if (!(ok = gm.barrier())) break;
    }
    if (blockIdx.x == 0) {
        __syncthreads();
        if (tid < NR) {
            const int k = k0 + tid;
            st->rr[k] = sc.rr[tid];
            st->rr_in[k] = acc_double(sc.rr_in[tid]);
            st->col_done[k] = 1;
            st->in_done[k] = 1;
            st->it_total[k] = sc.it_total[tid];
        }
        if (tid == 0) {
            st->sweeps = sweeps;
            st->status = ok ? sc.status : OASIS_EWAIT;
        }
    }
    gm.leave();
}

// ------------------------------------------------------------------ pressure CG
template <class V>
struct CgScalars {
    using X = LiteA<V>;
    X tot[kResValues], rr_in;
    CgCarry<X> carry;
    double bb, rr;
    V al, be, stop;                      // stop: the inner solve ends at or below it
    int it_total, col_done, in_done, status;
};

// One operator of the multigrid cycle on this block's rows, its entries read from
// global memory: out = T x (restriction), out = w d (2 r - A w d x) (smoothing; x is
// r), out = y + S x (prolongation).  The blocks meet at `goal` arrivals (0: no
// meeting) after the first entries have been fetched.  Not inlined: nine shapes of
// it in one kernel would spill.
enum LevelOp { kLevelRestrict, kLevelSmooth, kLevelProlong };
template <class V>
struct LevelArgs {
    using AV = typename ResidentLevel<V>::AV;
    int n;
    const int32_t *rp, *ci;
    const AV* a;
    const V *x, *y, *d;
    V w;
    V* out;
};
template <class V, int OP, int G, int M>
__device__ __noinline__ bool level_rows_g(LevelArgs<V> L, uint32_t* count, uint32_t goal) {
    const Chunk ch(L.n);
    const int32_t* __restrict__ rp = L.rp;
    const int32_t* __restrict__ ci = L.ci;
    const typename LevelArgs<V>::AV* __restrict__ a = L.a;
    const V* __restrict__ d = L.d;
    return res_rows<G, M, 1, V, V>(
        ch.hi - ch.lo, [&](int i) { return __ldg(rp + ch.lo + i); },
        [&](int q, int32_t& j, V& v) {
            j = __ldg(ci + q);
            v = (V)wide(__ldg(a + q));
        },
        [&] { return goal == 0 || grid_barrier(count, goal); },
        [&](int j) {
            if constexpr (OP == kLevelSmooth) return L.w * __ldg(d + j) * L.x[j];
            else return L.x[j];
        },
        [](V(&acc)[1], V m, V x) { acc[0] += m * x; },
        [&](int i, int lg, const V(&acc)[1]) {
            if (lg != 0) return;
            const int gi = ch.lo + i;
            if constexpr (OP == kLevelRestrict) L.out[gi] = acc[0];
            else if constexpr (OP == kLevelSmooth) L.out[gi] = L.w * __ldg(d + gi) * (V(2) * L.x[gi] - acc[0]);
            else L.out[gi] = L.y[gi] + acc[0];
        });
}
template <class V, int OP>
__device__ __forceinline__ bool level_rows(int g, const LevelArgs<V>& L, uint32_t* count, uint32_t goal) {
    if (g <= 1) return level_rows_g<V, OP, 1, 8>(L, count, goal);
    if (g <= 4) return level_rows_g<V, OP, 4, 4>(L, count, goal);
    if (g <= 8) return level_rows_g<V, OP, 8, 8>(L, count, goal);
    return level_rows_g<V, OP, 32, 4>(L, count, goal);
}

// One V(1,1) cycle u = M r, two meetings per level: with the level's operator A,
// Jacobi weight w, D = diag(A) and S = P - w D^-1 A P, the cycle that smooths once
// before and once after the coarse correction is
//   M = 2 w D^-1 - w D^-1 A w D^-1 + S M_c S^T
// (the pre-smoothed residual is (I - A w D^-1) r, its restriction S^T r; the
// post-smoother acts on the correction as I - w D^-1 A).  So one phase brings
// y = (2 w D^-1 - w D^-1 A w D^-1) r and the next level's input S^T r, the other
// x = y + S x_c, where smoothing, restriction, prolongation and smoothing one after
// the other take four.  S^T is the transpose of S to the bit, so M is symmetric.
// met: r is visible already.  The result is not yet visible to other blocks.
template <class V, class Fine>
__device__ __forceinline__ bool res_vcycle(GridMeet& gm, const ResidentAmg<V>& m, bool met, Fine&& fine) {
    for (int l = 0; l < m.levels; ++l) {
        const ResidentLevel<V>& L = m.lv[l];
        const bool last = l + 1 == m.levels;
        const LevelArgs<V> down{last ? m.nc : m.lv[l + 1].n, L.t_rp, L.t_ci, L.t, L.r, nullptr, nullptr, L.w,
                                last ? m.rc : m.lv[l + 1].r};
        if (!level_rows<V, kLevelRestrict>(L.gt, down, gm.m.count, l == 0 && met ? 0u : gm.next())) return false;
        if (l == 0) {
            fine(L.w, L.y);
        } else {
            const LevelArgs<V> smooth{L.n, L.a_rp, L.a_ci, L.a, L.r, nullptr, L.d, L.w, L.y};
            level_rows<V, kLevelSmooth>(L.ga, smooth, gm.m.count, 0u);
        }
    }
    if (!gm.barrier()) return false;
    {
        // dense coarsest level, one warp per row
        using V2 = typename std::conditional<sizeof(V) == 4, float4, double2>::type;
        constexpr int E = (int)(sizeof(V2) / sizeof(V));
        const int lane = threadIdx.x & 31, nv = m.ld / E;
        const V2* rv = reinterpret_cast<const V2*>(m.rc);
        const int nw = (int)(blockDim.x >> 5);
        for (int i = (int)(threadIdx.x >> 5) * gridDim.x + blockIdx.x; i < m.nc; i += nw * gridDim.x) {
            const V2* row = reinterpret_cast<const V2*>(m.inv + (size_t)i * m.ld);
            V acc = 0;
#pragma unroll 4
            for (int c = lane; c < nv; c += 32) {
                const V2 p = __ldg(row + c), q = rv[c];
                if constexpr (E == 4) acc += p.x * q.x + p.y * q.y + p.z * q.z + p.w * q.w;
                else acc += p.x * q.x + p.y * q.y;
            }
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
            if (lane == 0) m.xc[i] = acc;
        }
    }
    for (int l = m.levels - 1; l >= 0; --l) {
        const ResidentLevel<V>& L = m.lv[l];
        const LevelArgs<V> up{L.n, L.s_rp, L.s_ci, L.s, l + 1 < m.levels ? m.lv[l + 1].x : m.xc, L.y, nullptr, L.w, L.x};
        if (!level_rows<V, kLevelProlong>(L.gs, up, gm.m.count, gm.next())) return false;
    }
    return true;
}

// The tail of a V-cycle of separate kernels: the small levels' kernels took 3.5-5 us
// each whatever their size; one launch with two meetings per level takes ~2.5 us per
// meeting.
template <class V>
__global__ void __launch_bounds__(512, 1) k_resident_tail(ResidentAmg<V> m, KrylovState* st, ResidentSync sy) {
    if (st->col_done[0] || st->in_done[0]) return;
    GridMeet gm(sy);
    const bool ok = res_vcycle<V>(gm, m, true, [&](V w, V* y) {
        const ResidentLevel<V>& L = m.lv[0];
        const LevelArgs<V> smooth{L.n, L.a_rp, L.a_ci, L.a, L.r, nullptr, L.d, w, y};
        level_rows<V, kLevelSmooth>(L.ga, smooth, nullptr, 0u);
    });
    if (!ok && threadIdx.x == 0) st->status = OASIS_EWAIT;
    gm.leave();
}

// How the pressure CG is preconditioned and how its iteration is arranged.
enum ResCg {
    kCgJacobi = 0,   // Jacobi, u published: two meetings per iteration (u; the dots)
    kCgQuads = 1,    // Jacobi, one meeting: every neighbour's new u is formed again from
                     // its gathered r, w and s, as in k_pcg_iter_sell
    kCgAmg = 2       // multigrid
};

template <class P>
constexpr int kJacobiForm = P::mixed ? kCgQuads : kCgJacobi;

// Chronopoulos-Gear CG inside refinement sweeps: the method, stopping tests and
// counters of the separate kernels (k_pcg_outer_sell, k_amg_cg_*, k_pcg_iter_sell;
// step.cu).
template <class P, int G, int M, int MODE, bool STAGED>
__global__ void __launch_bounds__(res_threads<P>(), 1) k_resident_cg(StepData<P> a, Ctl ctl,
                                                                     ResidentAmg<typename P::V> m, ResidentPlan pl,
                                                                     ResidentSync sy) {
    using V = typename P::V;
    using S = typename P::S;
    using Acc = typename P::Acc;
    using X = LiteA<V>;
    using Q = CgQuad<V>;
    extern __shared__ __align__(16) unsigned char dsm[];
    __shared__ CgScalars<V> sc;
    GridMeet gm(sy);
    const Chunk ch((int)a.n);
    const int rows = ch.hi - ch.lo, tid = threadIdx.x;
    const int groups = used_groups<G>(rows);
    unsigned char* at = dsm;
    ResMatrix<V, STAGED> mat;
    mat.fill(at, pl, ch, a.rp, a.col, a.K);
    V* const r = res_carve<V>(at, pl.rows);
    V* const w = res_carve<V>(at, pl.rows);
    V* const s = res_carve<V>(at, pl.rows);
    V* const p = res_carve<V>(at, pl.rows);
    V* const dl = res_carve<V>(at, pl.rows);
    V* const di = res_carve<V>(at, pl.rows);
    for (int i = tid; i < rows; i += blockDim.x) di[i] = a.dinvK[ch.lo + i];
    KrylovState* st = a.stp;
    if (tid == 0) {
        sc.col_done = st->col_done[0];
        sc.it_total = st->it_total[0];
        sc.status = st->status;
        sc.rr = sc.bb = 0.0;
        acc_zero(sc.rr_in);
    }
    int sweeps = st->sweeps, first = st->first, it_in = 0;
    double meanp = 0.0;
    S mean;
    if constexpr (P::mixed) mean = make_float2(st->mean_hi, st->mean_lo);
    else mean = st->mean;
    const S* __restrict__ Kout = a.Kout;
    const V* __restrict__ dinv = a.dinvK;
    __syncthreads();
    auto ptr = [&](int i) { return mat.ptr(i); };
    auto entry = [&](int q, int32_t& j, V& v) { mat.entry(q, j, v); };
    auto now = [] { return true; };
    auto add = [](V(&acc)[1], V kv, V x) { acc[0] += kv * x; };
    bool ok = true;
    // u = M r (multigrid), then w = K u with <r, u>, <w, u>, <r, r>; the meeting that
    // makes r (Jacobi: u) visible comes first, unless the caller's sum was one
    constexpr int kDots = 3;
    auto product = [&](bool met) {
        auto meet = [&] { return met || gm.barrier(); };
        if constexpr (MODE == kCgAmg) {
            if (!res_vcycle<V>(gm, m, met, [&](V om, V* y) {
                    res_rows<G, M, 1, V, V>(
                        rows, ptr, entry, now, [&](int j) { return om * __ldg(dinv + j) * a.ar[j]; }, add,
                        [&](int i, int lg, const V(&acc)[1]) {
                            if (lg == 0) y[ch.lo + i] = om * di[i] * (V(2) * r[i] - acc[0]);
                        });
                }))
                return false;
        }
        V part[kDots] = {};
        if (!res_rows<G, M, 1, V, V>(
                rows, ptr, entry, [&] { return MODE == kCgAmg ? gm.barrier() : meet(); },
                [&](int j) { return a.au[j]; }, add,
                [&](int i, int lg, const V(&acc)[1]) {
                    if (lg != 0) return;
                    const V wv = acc[0], rv = r[i];
                    const V u = MODE == kCgAmg ? a.au[ch.lo + i] : di[i] * rv;
                    w[i] = wv;
                    part[0] += rv * u;
                    part[1] += wv * u;
                    part[2] += rv * rv;
                }))
            return false;
        return gm.template sum<kDots, 1, G, V, X>(part, sc.tot, groups);
    };
    // off the critical path (by the last warp while the others start on the product); the sums stay where they are until the blocks have met again
    auto carry = [&] {
        const int lane = tid - ((int)blockDim.x - 32);
        if (lane >= 0) sc.carry.carry(lane, it_in == 0, sc.tot[0], sc.tot[1]);
    };
    // the coefficients of the next update, and the inner stopping test
    auto finish = [&] {
        ++it_in;
        if (tid == 0) {
            const X rr = sc.tot[2];
            sc.it_total += 1;
            const bool sound = sc.carry.next(sc.tot[0], sc.tot[1], sc.al, sc.be);
            sc.rr_in = rr;
            if (!sound || !isfinite(x_hi(rr)) || x_hi(rr) <= sc.stop || sc.it_total >= ctl.max_it || it_in >= ctl.sweep_cap)
                sc.in_done = 1;
        }
        __syncthreads();
    };
    for (;;) {
        // r = (b - mean b) - K x with float64-quality products
        {
            Acc part[3];
#pragma unroll
            for (int k = 0; k < 3; ++k) acc_zero(part[k]);
            res_rows<G, M, 1, Acc, S>(
                rows, ptr,
                [&](int q, int32_t& j, S& v) {
                    j = mat.column(q);
                    v = __ldg(Kout + mat.e0 + q);
                },
                now,
                [&](int j) { return a.x[j]; },
                [](Acc(&acc)[1], S kv, S x) { lazy_add_prod_s(acc[0], kv, x); },
                [&](int i, int lg, const Acc(&acc)[1]) {
                    if (lg != 0) return;
                    const int gi = ch.lo + i;
                    const S bi = s_sub(a.b[gi], mean);
                    const V rv = s_v(s_sub(bi, s_of_acc(acc[0]))), xv = s_v(a.x[gi]), bv = s_v(bi);
                    if (!sc.col_done) {
                        r[i] = rv;
                        p[i] = 0;
                        s[i] = 0;
                        dl[i] = 0;
                        if constexpr (MODE == kCgAmg) a.ar[gi] = rv;
                        else a.au[gi] = di[i] * rv;
                    }
                    a.xv[gi] = xv;
                    acc_prod(part[0], rv, rv);
                    acc_prod(part[1], bv, bv);
                    acc_addv(part[2], s_v(a.pstar[gi]));
                    acc_addv(part[2], xv);
                });
            if (!(ok = gm.template sum<3, 1, G, Acc, Acc>(part, sc.tot, used_groups<G>(rows)))) break;
        }
        if (tid == 0) {
            if (first) sc.bb = acc_double(sc.tot[1]);
            if (sc.status != OASIS_OK) sc.col_done = 1;
            if (!sc.col_done) {
                const double rr = acc_double(sc.tot[0]);
                sc.rr = rr;
                if (!isfinite(rr)) {
                    sc.status = OASIS_ENAN;
                    sc.col_done = 1;
                } else if (rr <= ctl.rtol2 * sc.bb) {
                    sc.col_done = 1;
                } else if (sc.it_total >= ctl.max_it || sweeps >= kResMaxSweeps) {
                    sc.status = OASIS_ENOTCONV;
                    sc.col_done = 1;
                } else {
                    sc.in_done = 0;
                    sc.stop = limit_of(V(0), fmax(ctl.inner2 * rr, ctl.abs2 * sc.bb));
                }
            }
        }
        __syncthreads();
        if (blockIdx.x == 0 && tid == 0) meanp = acc_double(sc.tot[2]) / (double)a.n;
        first = 0;
        ++sweeps;
        it_in = 0;
        if (sc.col_done) break;
        // first product of the sweep: alpha = gamma / delta, beta = 0
        if (!(ok = product(true))) break;
        if (tid == 0) {
            const X g0 = sc.tot[0], d0 = sc.tot[1];
            if (!(x_hi(d0) > V(0)) || !isfinite(x_hi(d0)) || !isfinite(x_hi(g0))) {
                sc.in_done = 1;
                sc.it_total += 1;
            } else {
                sc.al = sc.carry.start(g0, d0);
            }
            sc.be = V(0);
        }
        __syncthreads();
        if constexpr (MODE == kCgQuads) {
            for (int i = tid; i < rows; i += blockDim.x) a.pq1[ch.lo + i] = Q{r[i], w[i], V(0), di[i]};
            if (!(ok = gm.barrier())) break;
        }
        while (!sc.in_done) {
            const V al = sc.al, be = sc.be;
            carry();
            if constexpr (MODE == kCgQuads) {
                const Q* qo = (it_in & 1) ? a.pq0 : a.pq1;
                Q* qn = (it_in & 1) ? a.pq1 : a.pq0;
                V part[3] = {};
                res_rows<G, M, 1, V, V>(
                    rows, ptr, entry, now, [&](int j) {
                        const Q g = qo[j];
                        return g.d * (g.r - al * (g.w + be * g.s));
                    }, add,
                    [&](int i, int lg, const V(&acc)[1]) {
                        if (lg != 0) return;
                        const V wo = w[i], ro = r[i], d = di[i];
                        const V pv = d * ro + be * p[i], sv = wo + be * s[i];
                        p[i] = pv;
                        s[i] = sv;
                        dl[i] += al * pv;
                        const V rv = ro - al * sv, wv = acc[0];
                        r[i] = rv;
                        w[i] = wv;
                        qn[ch.lo + i] = Q{rv, wv, sv, d};
                        const V un = d * rv;
                        part[0] += rv * un;
                        part[1] += wv * un;
                        part[2] += rv * rv;
                    });
                if (!(ok = gm.template sum<3, 1, G, V, X>(part, sc.tot, groups))) break;
                finish();
                continue;
            }
            // p = u + beta p, s = w + beta s, delta += alpha p, r -= alpha s
            V part[1] = {};
            for (int i = tid; i < rows; i += blockDim.x) {
                const V u = MODE == kCgAmg ? a.au[ch.lo + i] : di[i] * r[i];
                const V pv = be == V(0) ? u : u + be * p[i];
                const V sv = be == V(0) ? w[i] : w[i] + be * s[i];
                p[i] = pv;
                s[i] = sv;
                dl[i] += al * pv;
                const V rv = r[i] - al * sv;
                r[i] = rv;
                if constexpr (MODE == kCgAmg) {
                    a.ar[ch.lo + i] = rv;
                    part[0] += rv * rv;
                } else {
                    a.au[ch.lo + i] = di[i] * rv;
                }
            }
            if constexpr (MODE == kCgAmg) {
                // a residual that meets the inner test ends the solve before another cycle;
                // the sum is the meeting that makes r visible
                if (!(ok = gm.template sum<1, 1, 1, V, X>(part, sc.tot, min(rows, (int)blockDim.x)))) break;
                if (tid == 0) {
                    const X rr = sc.tot[0];
                    if (!isfinite(x_hi(rr)) || x_hi(rr) <= sc.stop || sc.it_total + 1 >= ctl.max_it || it_in + 1 >= ctl.sweep_cap) {
                        sc.rr_in = rr;
                        sc.it_total += 1;
                        sc.in_done = 1;
                    }
                }
                __syncthreads();
                if (sc.in_done) {
                    ++it_in;
                    break;
                }
            }
            if (!(ok = product(MODE == kCgAmg))) break;
            finish();
        }
        if (!ok) break;
        // x += delta
        __syncthreads();
        for (int i = tid; i < rows; i += blockDim.x) a.x[ch.lo + i] = s_addv(a.x[ch.lo + i], dl[i]);
        if (!(ok = gm.barrier())) break;
    }
    if (blockIdx.x == 0) {
        __syncthreads();
        if (tid == 0) {
            st->bb[0] = sc.bb;
            st->rr[0] = sc.rr;
            st->rr_in[0] = acc_double(sc.rr_in);
            st->psum = meanp;
            st->meanp_hi = (float)meanp;
            st->meanp_lo = (float)(meanp - (double)(float)meanp);
            st->col_done[0] = 1;
            st->in_done[0] = 1;
            st->it_total[0] = sc.it_total;
            st->it_in = it_in;
            st->sweeps = sweeps;
            st->first = 0;
            st->status = ok ? sc.status : OASIS_EWAIT;
        }
    }
    gm.leave();
}

// ------------------------------------------------------------------ consistent mass
// The consistent-mass update's CG on the interior block of M (k_mass_*, step.cu): the
// same start, right-hand side, stopping test and counters; Dirichlet rows stay out of
// the Krylov space.  Two meetings per iteration: <p, q>; <r, z> and <r, r>, which also
// makes z visible.
template <class V, int D>
struct MassScalars {
    using X = LiteA<V>;
    X tot[kResValues];
    X rho[D], rr[D], bb[D];
    V al[D], be[D], stop[D];
    int done[D], it, status;
};
template <class P, int D, int G, int M, bool STAGED>
__global__ void __launch_bounds__(res_threads<P>(), 1) k_resident_mass(StepData<P> a, typename P::V dt, Ctl ctl,
                                                                       ResidentPlan pl, ResidentSync sy,
                                                                       Pub<typename P::V, D>* pub) {
    using V = typename P::V;
    using X = LiteA<V>;
    using Pb = Pub<V, D>;
    extern __shared__ __align__(16) unsigned char dsm[];
    __shared__ MassScalars<V, D> sc;
    GridMeet gm(sy);
    const Chunk ch((int)a.n);
    const int rows = ch.hi - ch.lo, count = rows * D, tid = threadIdx.x;
    const int groups = used_groups<G>(rows);
    unsigned char* at = dsm;
    ResMatrix<V, STAGED> mat;
    mat.fill(at, pl, ch, a.rp, a.col, a.M);
    V* const r = res_carve<V>(at, pl.rows * D);
    V* const z = res_carve<V>(at, pl.rows * D);
    V* const p = res_carve<V>(at, pl.rows * D);
    V* const q = res_carve<V>(at, pl.rows * D);
    V* const dl = res_carve<V>(at, pl.rows * D);
    V* const im = res_carve<V>(at, pl.rows);   // 1 / ML
    V* const in = res_carve<V>(at, pl.rows);   // 0 for Dirichlet rows, else 1
    Pb* const zp = pub;
    Pb* const dp = pub + a.n;                  // the start
    const int32_t* __restrict__ dir = a.dir_index;
    const V* __restrict__ Gk = a.G;
    for (int i = tid; i < rows; i += blockDim.x) {
        im[i] = a.invML[ch.lo + i];
        in[i] = dir[ch.lo + i] >= 0 ? V(0) : V(1);
    }
    KrylovState* st = a.stm;
    if (tid == 0) {
        sc.it = 0;
        sc.status = OASIS_OK;
    }
    __syncthreads();
    auto ptr = [&](int i) { return mat.ptr(i); };
    auto entry = [&](int e, int32_t& j, V& v) { mat.entry(e, j, v); };
    auto now = [] { return true; };
    // delta_0: -dt dP^k phi / ML, or g - u^I on Dirichlet rows; q holds -dt dP^k phi
    res_rows<G, M, D, V, int32_t>(
        rows, ptr,
        [&](int e, int32_t& j, int32_t& v) {
            j = mat.column(e);
            v = e;
        },
        now,
        [&](int j) { return a.xv[j]; },
        [&](V(&acc)[D], int32_t e, V ph) {
#pragma unroll
            for (int k = 0; k < D; ++k) acc[k] += __ldg(Gk + (size_t)k * a.nnz + mat.e0 + e) * ph;
        },
        [&](int i, int lg, const V(&acc)[D]) {
            const int gi = ch.lo + i, di = dir[gi];
#pragma unroll
            for (int k = 0; k < D; ++k) {
                if (k % G != lg) continue;
                const size_t o = (size_t)gi * D + k;
                const V b = di >= 0 ? V(0) : -dt * acc[k];
                const V d0 = di >= 0 ? s_v(s_sub(a.g[(size_t)di * D + k], s_add(a.u1[o], a.du[o]))) : b * im[i];
                q[i * D + k] = b;
                dl[i * D + k] = d0;
                dp[gi].v[k] = d0;
            }
        });
    bool ok = gm.barrier();
    // r = b - M delta_0 over the interior columns, b the interior system's right-hand
    // side (Dirichlet columns moved to it)
    if (ok) {
        V part[3 * D] = {};
        res_rows<G, M, 2 * D, V, V>(
            rows, ptr, entry, now,
            [&](int j) {
                Vec<V, D + 1> g;
#pragma unroll
                for (int k = 0; k < D; ++k) g.v[k] = dp[j].v[k];
                g.v[D] = dir[j] >= 0 ? V(1) : V(0);
                return g;
            },
            [](V(&acc)[2 * D], V mv, const Vec<V, D + 1>& g) {
#pragma unroll
                for (int k = 0; k < D; ++k) {
                    if (g.v[D] != V(0)) acc[D + k] -= mv * g.v[k];
                    else acc[k] += mv * g.v[k];
                }
            },
            [&](int i, int lg, const V(&acc)[2 * D]) {
#pragma unroll
                for (int k = 0; k < D; ++k) {
                    if (k % G != lg) continue;
                    const int e = i * D + k;
                    const V b = q[e] + acc[D + k];
                    const V rv = in[i] != V(0) ? b - acc[k] : V(0);
                    const V zv = rv * im[i];
                    r[e] = rv;
                    z[e] = zv;
                    p[e] = V(0);
                    q[e] = V(0);
                    zp[ch.lo + i].v[k] = zv;
                    part[k] += rv * zv;
                    part[D + k] += rv * rv;
                    if (in[i] != V(0)) part[2 * D + k] += b * b;
                }
            });
        ok = gm.template sum<3 * D, D, G, V, X>(part, sc.tot, groups);
    }
    bool live = false;
    auto alive = [&] {
        bool any = false;
#pragma unroll
        for (int k = 0; k < D; ++k) any |= !sc.done[k];
        return any && sc.status == OASIS_OK;
    };
    if (ok) {
        if (tid < D) {
            const X rz = sc.tot[tid], rr = sc.tot[D + tid], bb = sc.tot[2 * D + tid];
            sc.rho[tid] = rz;
            sc.rr[tid] = rr;
            sc.bb[tid] = bb;
            sc.be[tid] = V(0);
            sc.stop[tid] = limit_of(V(0), ctl.rtol2 * acc_double(bb));
            if (!isfinite(x_hi(rz)) || !isfinite(x_hi(rr)) || !isfinite(x_hi(bb))) sc.status = OASIS_ENAN;
            sc.done[tid] = !(x_hi(rr) > sc.stop[tid]);
        }
        __syncthreads();
        live = alive();
    }
    while (ok && live) {
        V part[D] = {};
        res_rows<G, M, D, V, V>(
            rows, ptr, entry, now, [&](int j) { return zp[j]; },
            [](V(&acc)[D], V mv, const Pb& g) {
#pragma unroll
                for (int k = 0; k < D; ++k) acc[k] += mv * g.v[k];
            },
            [&](int i, int lg, const V(&acc)[D]) {
#pragma unroll
                for (int k = 0; k < D; ++k) {
                    if (k % G != lg || in[i] == V(0) || sc.done[k]) continue;
                    const int e = i * D + k;
                    const V be = sc.be[k];
                    const V pv = be == V(0) ? z[e] : z[e] + be * p[e];
                    const V qv = be == V(0) ? acc[k] : acc[k] + be * q[e];
                    p[e] = pv;
                    q[e] = qv;
                    part[k] += pv * qv;
                }
            });
        if (!(ok = gm.template sum<D, D, G, V, X>(part, sc.tot, groups))) break;
        if (tid < D && !sc.done[tid]) {
            const X pq = sc.tot[tid];
            V al = V(0);
            if (x_hi(pq) > V(0) && isfinite(x_hi(pq))) {
                al = quotient(sc.rho[tid], pq);
            } else {
                // <p, q> = 0 with r != 0 cannot happen for SPD M: a breakdown
                sc.done[tid] = 2;
                sc.status = isfinite(x_hi(pq)) ? OASIS_EBREAKDOWN : OASIS_ENAN;
            }
            sc.al[tid] = al;
        }
        __syncthreads();
        // delta += alpha p, r -= alpha q, z = r / ML
        V sums[2 * D] = {};
        for (int i = tid; i < rows; i += blockDim.x) {
#pragma unroll
            for (int k = 0; k < D; ++k) {
                if (sc.done[k] || in[i] == V(0)) continue;
                const int e = i * D + k;
                const V al = sc.al[k];
                dl[e] += al * p[e];
                const V rv = r[e] - al * q[e], zv = rv * im[i];
                r[e] = rv;
                z[e] = zv;
                zp[ch.lo + i].v[k] = zv;
                sums[k] += rv * zv;
                sums[D + k] += rv * rv;
            }
        }
        if (!(ok = gm.template sum<2 * D, 1, 1, V, X>(sums, sc.tot, min(rows, (int)blockDim.x)))) break;
        if (tid < D && !sc.done[tid]) {
            const X rz = sc.tot[tid], rr = sc.tot[D + tid];
            sc.rr[tid] = rr;
            if (!isfinite(x_hi(rz)) || !isfinite(x_hi(rr))) {
                sc.status = OASIS_ENAN;
                sc.done[tid] = 1;
            } else if (!(x_hi(rr) > sc.stop[tid])) {
                sc.done[tid] = 1;
            } else {
                sc.be[tid] = x_hi(sc.rho[tid]) > V(0) ? quotient(rz, sc.rho[tid]) : V(0);
                sc.rho[tid] = rz;
            }
        }
        __syncthreads();
        live = alive();
        if (tid == 0) {
            sc.it += 1;
            if (live && sc.it >= ctl.max_it) sc.status = OASIS_ENOTCONV;
        }
        __syncthreads();
        live = alive();
    }
    __syncthreads();
    for (int e = tid; e < count; e += blockDim.x) a.mx[(size_t)ch.lo * D + e] = dl[e];
    if (blockIdx.x == 0 && tid == 0) {
        for (int k = 0; k < 3; ++k) {
            st->bb[k] = ok && k < D ? acc_double(sc.bb[k]) : 0.0;
            st->rr[k] = ok && k < D ? acc_double(sc.rr[k]) : 0.0;
            st->col_done[k] = 1;
            st->it_total[k] = k == 0 ? sc.it : 0;
        }
        st->in_done[0] = 1;
        st->status = ok ? sc.status : OASIS_EWAIT;
    }
    gm.leave();
}

// shared memory that the kernels hold statically (float64: the sums' slots)
template <class P>
constexpr int res_static(bool mass) {
    return (P::mixed ? 8 : mass ? 40 : 20) * 1024;
}

int device_attribute(cudaDeviceAttr what) {
    int dev = 0, v = 0;
    OASIS_CUDA(cudaGetDevice(&dev));
    OASIS_CUDA(cudaDeviceGetAttribute(&v, what, dev));
    return v;
}
// Whether the current device takes a cooperative launch of fn in this shape; sets the
// kernel's shared-memory limit for the launches to come.
template <class F>
bool fits(F fn, const ResidentPlan& pl) {
    if (!device_attribute(cudaDevAttrCooperativeLaunch)) return false;
    cudaFuncAttributes fa{};
    OASIS_CUDA(cudaFuncGetAttributes(&fa, fn));
    const int most = device_attribute(cudaDevAttrMaxSharedMemoryPerBlockOptin) - (int)fa.sharedSizeBytes;
    if (pl.smem > most) return false;
    if (pl.smem > 0) OASIS_CUDA(cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, most));
    int per_sm = 0;
    OASIS_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, fn, pl.threads, (size_t)pl.smem));
    return (int64_t)per_sm * num_sms() >= pl.blocks;
}

template <class... KArgs, class... Args>
void launch(void (*fn)(KArgs...), const ResidentPlan& pl, cudaStream_t s, Args&&... args) {
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3((unsigned)pl.blocks);
    cfg.blockDim = dim3((unsigned)pl.threads);
    cfg.dynamicSmemBytes = (size_t)pl.smem;
    cfg.stream = s;
    cudaLaunchAttribute at{};
    at.id = cudaLaunchAttributeCooperative;
    at.val.cooperative = 1;
    cfg.attrs = &at;
    cfg.numAttrs = 1;
    OASIS_CUDA(cudaLaunchKernelEx(&cfg, fn, std::forward<Args>(args)...));
}

// The shape for n rows with `vectors` values per row beside the matrix.
template <class P>
ResidentPlan plan(const std::vector<int32_t>& row_ptr, int64_t n, int vectors, bool mass = false) {
    using V = typename P::V;
    ResidentPlan p;
    if (n < 1 || n > kResidentRows) return p;
    auto shape = [&](int blocks) {
        p.rows = (int)((n + blocks - 1) / blocks);
        p.entries = 0;
        for (int64_t lo = 0; lo < n; lo += p.rows)
            p.entries = std::max(p.entries, row_ptr[std::min<int64_t>(n, lo + p.rows)] - row_ptr[lo]);
        const size_t vec = (size_t)vectors * res_vector_bytes<V>(p.rows), room = (size_t)(device_attribute(cudaDevAttrMaxSharedMemoryPerBlockOptin) - res_static<P>(mass));
        const size_t mat = res_matrix_bytes<V>(p.rows, p.entries);
        if (vec > room) return false;
        p.staged = vec + mat <= room;
        p.smem = (int)(vec + (p.staged ? mat : 0));
        p.blocks = blocks;
        return true;
    };
    // all SMs, with at least 16 rows per block.  us per step with 8 / 16 / 32 / 64: 289
    // rows float64 multigrid 565 / 540 / 578 / 643, 1,089: 508 / 482 / 508 / 565 (mixed 350
    // / 327 / 325 / 323), 512 float64 Jacobi 746 / 746 / 796 / 924, 2,197: 1099 / 1085 /
    // 1122 / 1303 (mixed 502 / 490 / 505 / 527), 4,913 mixed multigrid 481 / 480 / 472 / 451
    // (float64 948 / 951 / 949 / 1022).
    if (!shape((int)std::min<int64_t>(std::min(num_sms(), kResBlocks), (n + 15) / 16))) return p;
    // As many lanes per row as there are threads for.  Where 256 threads have a group for
    // every row the launch takes no more, half the registers of an SM, so that solves of
    // solvers on other streams run beside it; larger systems take all of every SM.  15,625
    // rows mixed multigrid, us per step and solver with 1 / 2 / 4 solvers stepped at once:
    // 642 / 369 / 350 (512 threads 549 / 532 / 548, separate kernels 1111 / 611 / 353); one
    // solver, 256 against 512 threads: 29,791 rows Jacobi 840 / 896, multigrid 751 / 732,
    // 22,801 (triangles) 484 / 505, 8,000 float64 Jacobi 1504 / 1600, 4,913 float64
    // multigrid 956 / 936.  68,921 rows with 256 threads: 1061 against 886 alone.
    const int most = p.rows * (P::mixed ? 1 : 4) <= 256 ? 256 : res_threads<P>();
    p.lanes = 8;
    while (p.lanes > (P::mixed ? 1 : 4) && p.rows * p.lanes > most) p.lanes /= 2;
    p.threads = std::min(most, std::max(256, (p.rows * p.lanes + 31) / 32 * 32));
    return p;
}

}  // namespace

constexpr size_t kSyncBytes = 512 + (size_t)2 * kResValues * kResBlocks * 8;

size_t resident_sync_bytes(int64_t n, size_t value_bytes) { return kSyncBytes + 3 * 4 * value_bytes * (size_t)n; }

ResidentSync resident_sync(void* mem) {
    auto* p = static_cast<unsigned char*>(mem);
    return {reinterpret_cast<uint32_t*>(p), reinterpret_cast<uint32_t*>(p + 256), p + 512, p + kSyncBytes};
}

// LAUNCH(lanes, entries in flight, staged) of a plan; a matrix that does not fit in
// shared memory belongs to a plan with the fewest lanes
#define OASIS_RES_SHAPE(LAUNCH)                                                              \
    constexpr int kFew = P::mixed ? 1 : 4, kTwo = P::mixed ? 2 : 4, kM = P::mixed ? 8 : 4;   \
    if (!pl.staged) LAUNCH(kFew, kM, false);                                                 \
    else if (pl.lanes >= 8) LAUNCH(8, 2, true);                                              \
    else if (pl.lanes >= 4) LAUNCH(4, 4, true);                                              \
    else if (pl.lanes >= 2) LAUNCH(kTwo, kM, true);                                          \
    else LAUNCH(kFew, kM, true)

void resident_set_wait(void* mem, int64_t cycles, cudaStream_t s) {
    OASIS_CUDA(cudaMemcpyAsync(static_cast<unsigned char*>(mem) + 8, &cycles, sizeof(cycles), cudaMemcpyHostToDevice, s));
    OASIS_CUDA(cudaStreamSynchronize(s));
}

template <class P, int D, int NR>
ResidentPlan resident_plan_bicg(const std::vector<int32_t>& row_ptr, int64_t n) {
    if (!P::mixed && NR > 1 && n > kResidentRows64) return {};
    const ResidentPlan pl = plan<P>(row_ptr, n, 6 * NR + 1);
    bool ok = pl.blocks > 0;
#define OASIS_RES_FITS(G, M, ST) ok = ok && fits(k_resident_bicg<P, D, NR, G, M, ST>, pl)
    OASIS_RES_SHAPE(OASIS_RES_FITS);
#undef OASIS_RES_FITS
    return ok ? pl : ResidentPlan{};
}
template <class P, int D>
ResidentPlan resident_plan_mass(const std::vector<int32_t>& row_ptr, int64_t n) {
    const ResidentPlan pl = plan<P>(row_ptr, n, 5 * D + 2, true);
    bool ok = pl.blocks > 0;
#define OASIS_RES_FITS(G, M, ST) ok = ok && fits(k_resident_mass<P, D, G, M, ST>, pl)
    OASIS_RES_SHAPE(OASIS_RES_FITS);
#undef OASIS_RES_FITS
    return ok ? pl : ResidentPlan{};
}
template <class P>
ResidentPlan resident_plan_cg(const std::vector<int32_t>& row_ptr, int64_t n, bool amg) {
    if (amg && row_ptr[n] > (P::mixed ? kResidentAmgEntries : kResidentAmgEntries64)) return {};
    const ResidentPlan pl = plan<P>(row_ptr, n, 6);
    bool ok = pl.blocks > 0;
    if (amg) {
#define OASIS_RES_FITS(G, M, ST) ok = ok && fits(k_resident_cg<P, G, M, kCgAmg, ST>, pl)
        OASIS_RES_SHAPE(OASIS_RES_FITS);
#undef OASIS_RES_FITS
    } else {
#define OASIS_RES_FITS(G, M, ST) ok = ok && fits(k_resident_cg<P, G, M, kJacobiForm<P>, ST>, pl)
        OASIS_RES_SHAPE(OASIS_RES_FITS);
#undef OASIS_RES_FITS
    }
    return ok ? pl : ResidentPlan{};
}
template <class V>
ResidentPlan resident_plan_tail(int64_t n) {
    ResidentPlan pl;
    pl.threads = 512;
    // at least 16 rows of the tail's finest level per block
    pl.blocks = (int)std::max<int64_t>(1, std::min<int64_t>(std::min(num_sms(), kResBlocks), (n + 15) / 16));
    return !device_attribute(cudaDevAttrMpsEnabled) && fits(k_resident_tail<V>, pl) ? pl : ResidentPlan{};
}
template ResidentPlan resident_plan_tail<float>(int64_t);
template ResidentPlan resident_plan_tail<double>(int64_t);

template <class P, int D, int NR>
void resident_bicg(const StepData<P>& q, int k0, const Ctl& c, const ResidentPlan& pl, const ResidentSync& sy,
                   cudaStream_t s) {
    auto* pub = static_cast<Pub<typename P::V, NR>*>(sy.pub);
#define OASIS_RES_LAUNCH(G, M, ST) launch(k_resident_bicg<P, D, NR, G, M, ST>, pl, s, q, k0, c, pl, sy, pub)
    OASIS_RES_SHAPE(OASIS_RES_LAUNCH);
#undef OASIS_RES_LAUNCH
}

template <class P>
void resident_cg(const StepData<P>& q, const Ctl& c, const ResidentAmg<typename P::V>& m, const ResidentPlan& pl,
                 const ResidentSync& sy, cudaStream_t s) {
    if (m.levels > 0) {
#define OASIS_RES_LAUNCH(G, M, ST) launch(k_resident_cg<P, G, M, kCgAmg, ST>, pl, s, q, c, m, pl, sy)
        OASIS_RES_SHAPE(OASIS_RES_LAUNCH);
#undef OASIS_RES_LAUNCH
    } else {
#define OASIS_RES_LAUNCH(G, M, ST) launch(k_resident_cg<P, G, M, kJacobiForm<P>, ST>, pl, s, q, c, m, pl, sy)
        OASIS_RES_SHAPE(OASIS_RES_LAUNCH);
#undef OASIS_RES_LAUNCH
    }
}

template <class P, int D>
void resident_mass(const StepData<P>& q, double dt, const Ctl& c, const ResidentPlan& pl, const ResidentSync& sy,
                   cudaStream_t s) {
    auto* pub = static_cast<Pub<typename P::V, D>*>(sy.pub);
#define OASIS_RES_LAUNCH(G, M, ST) launch(k_resident_mass<P, D, G, M, ST>, pl, s, q, (typename P::V)dt, c, pl, sy, pub)
    OASIS_RES_SHAPE(OASIS_RES_LAUNCH);
#undef OASIS_RES_LAUNCH
}
#undef OASIS_RES_SHAPE

template <class V>
ResidentAmg<V> resident_amg(const AmgHierarchy& h, AmgWork& w, int first, int blocks, int threads) {
    ResidentAmg<V> r;
    const int L = (int)h.lv.size();
    r.levels = L - first;
    r.nc = (int32_t)h.nc;
    r.ld = (int32_t)h.ld;
    if constexpr (sizeof(V) == 4) r.inv = h.inv32.p;
    else r.inv = h.inv64.p;
    auto vec = [](const DBuf<double>& b) { return reinterpret_cast<V*>(b.p); };
    r.rc = vec(w.rin[L]);
    r.xc = vec(w.xo[L]);
    auto lanes = [&](int64_t rows, size_t nnz) {
        // as many lanes per row as there are threads and entries for
        const double mean = (double)nnz / (double)std::max<int64_t>(1, rows);
        const int64_t per_block = (rows + blocks - 1) / blocks;
        int g = 32;
        while (g > 1 && (per_block * g > threads || g > mean)) g /= 2;
        return g;
    };
    for (int l = first; l < L; ++l) {
        const AmgLevelDev& v = *h.lv[l];
        ResidentLevel<V>& o = r.lv[l - first];
        o.n = (int32_t)v.n;
        o.w = (V)v.omega;
        o.a_rp = v.rp;
        o.a_ci = v.ci;
        o.s_rp = v.s_rp.p;
        o.s_ci = v.s_ci.p;
        o.t_rp = v.t_rp.p;
        o.t_ci = v.t_ci.p;
        if constexpr (sizeof(V) == 4) {
            o.d = v.d32.p;
            o.a = v.a16;
            o.s = v.s16.p;
            o.t = v.t16.p;
        } else {
            o.d = v.d64.p;
            o.a = v.a64;
            o.s = v.s64.p;
            o.t = v.t64.p;
        }
        o.r = vec(w.rin[l]);
        o.x = vec(w.xo[l]);
        o.y = vec(w.x[l]);
        o.ga = lanes(v.n, (size_t)v.nnz);
        o.gs = lanes(v.n, v.s16.n);
        o.gt = lanes(l + 1 < L ? h.lv[l + 1]->n : h.nc, v.s16.n);
    }
    return r;
}

template <class V>
void resident_tail(const AmgHierarchy& h, AmgWork& w, int first, KrylovState* st, cudaStream_t s) {
    const ResidentPlan& pl = w.tail_plan;
    launch(k_resident_tail<V>, pl, s, resident_amg<V>(h, w, first, pl.blocks, pl.threads), st, resident_sync(w.meet.p));
}
template void resident_tail<float>(const AmgHierarchy&, AmgWork&, int, KrylovState*, cudaStream_t);
template void resident_tail<double>(const AmgHierarchy&, AmgWork&, int, KrylovState*, cudaStream_t);
template ResidentAmg<float> resident_amg<float>(const AmgHierarchy&, AmgWork&, int, int, int);
template ResidentAmg<double> resident_amg<double>(const AmgHierarchy&, AmgWork&, int, int, int);

#define OASIS_RES(P)                                                                                             \
    template void resident_bicg<P, 3, 3>(const StepData<P>&, int, const Ctl&, const ResidentPlan&,               \
                                         const ResidentSync&, cudaStream_t);                                     \
    template void resident_bicg<P, 3, 1>(const StepData<P>&, int, const Ctl&, const ResidentPlan&,               \
                                         const ResidentSync&, cudaStream_t);                                     \
    template void resident_bicg<P, 2, 2>(const StepData<P>&, int, const Ctl&, const ResidentPlan&,               \
                                         const ResidentSync&, cudaStream_t);                                     \
    template void resident_bicg<P, 2, 1>(const StepData<P>&, int, const Ctl&, const ResidentPlan&,               \
                                         const ResidentSync&, cudaStream_t);                                     \
    template void resident_bicg<P, 1, 1>(const StepData<P>&, int, const Ctl&, const ResidentPlan&,               \
                                         const ResidentSync&, cudaStream_t);                                     \
    template void resident_mass<P, 3>(const StepData<P>&, double, const Ctl&, const ResidentPlan&,               \
                                      const ResidentSync&, cudaStream_t);                                        \
    template void resident_mass<P, 2>(const StepData<P>&, double, const Ctl&, const ResidentPlan&,               \
                                      const ResidentSync&, cudaStream_t);                                        \
    template void resident_cg<P>(const StepData<P>&, const Ctl&, const ResidentAmg<typename P::V>&,              \
                                 const ResidentPlan&, const ResidentSync&, cudaStream_t);                        \
    template ResidentPlan resident_plan_bicg<P, 3, 3>(const std::vector<int32_t>&, int64_t);                     \
    template ResidentPlan resident_plan_bicg<P, 3, 1>(const std::vector<int32_t>&, int64_t);                     \
    template ResidentPlan resident_plan_bicg<P, 2, 2>(const std::vector<int32_t>&, int64_t);                     \
    template ResidentPlan resident_plan_bicg<P, 2, 1>(const std::vector<int32_t>&, int64_t);                     \
    template ResidentPlan resident_plan_bicg<P, 1, 1>(const std::vector<int32_t>&, int64_t);                     \
    template ResidentPlan resident_plan_mass<P, 3>(const std::vector<int32_t>&, int64_t);                        \
    template ResidentPlan resident_plan_mass<P, 2>(const std::vector<int32_t>&, int64_t);                        \
    template ResidentPlan resident_plan_cg<P>(const std::vector<int32_t>&, int64_t, bool);
OASIS_RES(Mixed)
OASIS_RES(Fp64)
#undef OASIS_RES

}  // namespace oasis
