// persist.cu -- BiCGStab, TFQMR and the mixed-precision refinement of one
// system (or of several, each on CTAs of its own) as ONE persistent
// cooperative kernel, for systems whose vectors fit on chip.
//
// What bounds it.  A graph node of the loop in bicgstab.cu or tfqmr.cu costs
// 6 to 7 us from launch to launch on small systems whatever the kernel does
// (42 us per BiCGStab iteration for any n up to 32k unknowns), and each of
// its kernels reads and writes the Krylov vectors through L2.  Here a CTA
// owns a run of slices (32 rows each, the row-per-lane layout of spmv.cuh)
// for the whole solve: thread t handles the same rows in every pass, their
// entries of all Krylov vectors stay in its shared memory, and only the two
// vectors that the products gather are also written to global memory.  What
// remains of a pass is its arithmetic on the binary64 pipe and a barrier
// among the CTAs of the system.
//
// The barrier carries the reduction.  A CTA publishes its partial sums as
// 16-byte units (value, epoch) in a 128-byte line of its own, and warp q of
// every CTA polls unit q of all lines, so that a barrier with dot products
// costs one L2 write and one L2 read latency; every CTA folds the same
// partials in the same order and computes the same scalars, so the run is
// deterministic.  Two sets of lines alternate: a CTA writes epoch e + 2 only
// after it has passed e + 1, which every CTA reaches only after it has read
// e.  Measured, 152 CTAs, with the fold of two sums: an atomic counter and a
// broadcast 5.6 us, packed units 3.4 us, units in lines of their own 2.8 us
// (two levels over clusters of 2 to 16 CTAs: 3.6 to 3.8 us).  Waits are
// bounded in time; an expired one ends the solve with HZ_ERR_TIMEOUT.
//
// A dependent binary64 addition takes 68 cycles here, one behind a shuffle
// 209, a division 557, so sums are folded as trees of values read from
// shared memory, and the scalars of an iteration are written so that one
// division, spread over the lanes of a warp, is all that a barrier waits
// for: squared norms are compared with squared thresholds, and the exact
// test runs only where they nearly meet.  (First version, with packed units,
// shuffle sums and the scalars on one thread: 12 000 cycles per barrier, 35
// us per BiCGStab iteration on 4096 unknowns.)
//
// Measured against the graphs, whole solves: BiCGStab on 16^3 unknowns 3.1 ->
// 1.66 ms (1.31 ms on one cluster, below), on 64^3 25.4 -> 15.9 ms; mixed on
// 48^3 12.5 -> 5.3 ms; forward and adjoint TFQMR on 32^3 26.7 -> 14.5 ms.
#include <algorithm>
#include <atomic>
#include <cstring>
#include <mutex>
#include <vector>

#include "persist.cuh"

namespace hz {

constexpr int kPsMaxCta = 160;       // CTAs of one system: five per polling lane
constexpr int kPsMaxWarps = 16;      // warps per CTA, a multiple of 4
constexpr int kPsMinWarps = 4;
constexpr int kPsMaxCluster = 16;    // CTAs of one cluster
constexpr uint64_t kPsStartNs = 10000000000ull;   // the first barrier waits for the launch of all CTAs
constexpr uint64_t kPsWaitNs = 4000000000ull;

struct alignas(16) PsUnit {
    unsigned long long v, tag;
};
struct alignas(128) PsLine {   // one CTA's sums of one barrier
    PsUnit u[3];
};

// one system of a launch
struct PsSys {
    MatView<double2> A;
    MatView<float2> A32;
    double2 *x;        // the iterate, gathered at the start and the end
    double2 *xbest;    // mixed: the kept iterate
    void *g0, *g1;     // the vectors the products gather (p, s; u1, u2)
    Ctl ctl;
    Info *info;
    PsLine *lines;     // [2][ncta]
    int *err;          // set when a wait expired
    int cta0, ncta;    // CTAs [cta0, cta0 + ncta) of the grid
    int batched;       // x is the caller's; b = 0 leaves it
};

// 16-byte accesses that are single and coherent at GPU scope
__device__ __forceinline__ void st_unit(PsUnit *p, unsigned long long v, unsigned long long tag) {
    asm volatile("{\n .reg .b128 t;\n mov.b128 t, {%1, %2};\n st.relaxed.gpu.global.b128 [%0], t;\n}" ::"l"(p), "l"(v),
                 "l"(tag)
                 : "memory");
}
__device__ __forceinline__ PsUnit ld_unit(const PsUnit *p) {
    PsUnit u;
    asm volatile("{\n .reg .b128 t;\n ld.relaxed.gpu.global.b128 t, [%2];\n mov.b128 {%0, %1}, t;\n}"
                 : "=l"(u.v), "=l"(u.tag)
                 : "l"(p)
                 : "memory");
    return u;
}

// (one direction each: a two-way fence on the reading side would wait for the
// CTA's own unit to be acknowledged)
__device__ __forceinline__ void fence_release() { asm volatile("fence.release.gpu;" ::: "memory"); }
__device__ __forceinline__ void fence_acquire() { asm volatile("fence.acquire.gpu;" ::: "memory"); }

template <class R> __device__ __forceinline__ unsigned long long unit_bits(R v) {
    if constexpr (std::is_same<R, double>::value) return (unsigned long long)__double_as_longlong(v);
    else return (unsigned long long)__float_as_uint(v);
}
template <class R> __device__ __forceinline__ R unit_value(unsigned long long b) {
    if constexpr (std::is_same<R, double>::value) return __longlong_as_double((long long)b);
    else return __uint_as_float((unsigned)b);
}

// the CTAs of a system as this CTA sees them
struct Grp {
    PsLine *lines;
    int *err;
    int rank, size;
    unsigned long long epoch;   // barriers passed
};

struct PsShared {
    double val[3][kPsMaxWarps * 32];   // per-thread sums (binary32 ones in the first half)
    double scr[3][40];                 // fold scratch of one warp each
    double tot[3];
    double cl[2][3][kPsMaxCluster];    // sums of the CTAs of a cluster
    int err;
};

// the sum of a over the warp, in every lane: radix-8 and radix-4 trees over
// values in shared memory (buf: 36 entries)
template <class R>
__device__ __forceinline__ R warp_fold(R a, R *buf) {
    const int lane = threadIdx.x & 31;
    buf[lane] = a;
    __syncwarp();
    if (lane < 4) {
        const R *q = buf + 8 * lane;
        buf[32 + lane] = ((q[0] + q[1]) + (q[2] + q[3])) + ((q[4] + q[5]) + (q[6] + q[7]));
    }
    __syncwarp();
    const R r = (buf[32] + buf[33]) + (buf[34] + buf[35]);
    __syncwarp();
    return r;
}

// Barrier of the system's CTAs with NV (0..3) sums: fin(tot, lane) runs on
// the lanes of one warp of every CTA before the CTA goes on.  kFence: the
// global writes made before it are visible after it (the barriers after the
// products and F5 publish nothing but sums; a gathered vector is overwritten
// only after a later barrier with the fence).  False when a wait expired.
// kLive 3: the CTAs are one cluster.  The sums go straight into every CTA's
// shared memory and the hardware's cluster barrier stands for the lines.
template <int kLive, class R, int NV, bool kFence, class F>
__device__ __forceinline__ bool grp_reduce(Grp &g, PsShared &sh, const R (&v)[NV > 0 ? NV : 1], F fin) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarps = blockDim.x >> 5;
    if constexpr (NV > 0) {
#pragma unroll
        for (int q = 0; q < NV; ++q) reinterpret_cast<R *>(sh.val[q])[threadIdx.x] = v[q];
    }
    const unsigned long long e = ++g.epoch;
    if constexpr (kLive == 3) {
        if constexpr (NV > 0) {
            R *scr = reinterpret_cast<R *>(sh.scr[warp < NV ? warp : 0]);
            R a = R(0);
            __syncthreads();
            if (warp < NV) {
                const R *p = reinterpret_cast<const R *>(sh.val[warp]) + lane;
                for (int w = 0; w < nwarps; w += 4) a += (p[32 * w] + p[32 * w + 32]) + (p[32 * w + 64] + p[32 * w + 96]);
                a = warp_fold(a, scr);
                if (lane < g.size) st_cluster(cluster_map(smem_addr(&sh.cl[e & 1][warp][g.rank]), lane), unit_bits(a));
                __syncwarp();
            }
            cluster_barrier();
            if (warp < NV) {
                a = lane < g.size ? unit_value<R>((unsigned long long)__double_as_longlong(sh.cl[e & 1][warp][lane])) : R(0);
                a = warp_fold(a, scr);
                if (NV > 1) {
                    if (lane == 0) reinterpret_cast<R *>(sh.tot)[warp] = a;
                    asm volatile("bar.sync 1, %0;" ::"r"(32 * NV) : "memory");
                }
                if (warp == 0) {
                    R tot[NV];
                    tot[0] = a;
#pragma unroll
                    for (int q = 1; q < NV; ++q) tot[q] = reinterpret_cast<R *>(sh.tot)[q];
                    fin(tot, lane);
                }
            }
            __syncthreads();
        } else {
            cluster_barrier();
        }
        return true;
    }
    __syncthreads();
    if (warp < (NV > 0 ? NV : 1)) {
        R a = R(0);
        R *scr = reinterpret_cast<R *>(sh.scr[warp]);
        if constexpr (NV > 0) {
            const R *p = reinterpret_cast<const R *>(sh.val[warp]) + lane;
            for (int w = 0; w < nwarps; w += 4) a += (p[32 * w] + p[32 * w + 32]) + (p[32 * w + 64] + p[32 * w + 96]);
            a = warp_fold(a, scr);
        }
        PsLine *set = g.lines + (size_t)(e & 1) * g.size;
        if (kFence && warp == 0) fence_release();   // this CTA's writes (ordered by the block barrier) before its units
        if (lane == 0) st_unit(&set[g.rank].u[warp], unit_bits(a), e);
        constexpr int K = kPsMaxCta / 32;
        uint64_t t0 = 0;
        for (int spin = 0;; ++spin) {
            bool ok = true;
            PsUnit u[K];
#pragma unroll
            for (int k = 0; k < K; ++k) {
                const int c = lane + 32 * k;
                u[k].v = 0ull;
                u[k].tag = e;
                if (c < g.size) u[k] = ld_unit(&set[c].u[warp]);
            }
#pragma unroll
            for (int k = 0; k < K; ++k) ok = ok && u[k].tag == e;
            if (__all_sync(0xffffffffu, ok)) {   // (CTAs past the last one are zero bits)
                static_assert(K == 5, "the tree below");
                a = ((unit_value<R>(u[0].v) + unit_value<R>(u[1].v)) + (unit_value<R>(u[2].v) + unit_value<R>(u[3].v))) +
                    unit_value<R>(u[4].v);
                break;
            }
            if ((spin & 255) == 255) {
                if (t0 == 0) t0 = global_ns();
                const bool give_up =
                    global_ns() - t0 > (e == 1 ? kPsStartNs : kPsWaitNs) || *(volatile int *)g.err != 0;
                if (__any_sync(0xffffffffu, give_up)) {
                    if (lane == 0) {
                        atomicExch(g.err, 1);
                        *(volatile int *)&sh.err = 1;
                    }
                    a = R(0);
                    break;
                }
            }
        }
        if (kFence && warp == 0) fence_acquire();   // the other CTAs' writes before this CTA's reads
        if constexpr (NV > 0) {
            a = warp_fold(a, scr);
            if (NV > 1) {
                if (lane == 0) reinterpret_cast<R *>(sh.tot)[warp] = a;
                asm volatile("bar.sync 1, %0;" ::"r"(32 * NV) : "memory");
            }
            if (warp == 0) {
                R tot[NV];
                tot[0] = a;
#pragma unroll
                for (int q = 1; q < NV; ++q) tot[q] = reinterpret_cast<R *>(sh.tot)[q];
                if (*(volatile int *)&sh.err == 0) fin(tot, lane);
            }
        }
    }
    __syncthreads();
    return sh.err == 0;
}
template <int kLive, class R>
__device__ __forceinline__ bool grp_sync(Grp &g, PsShared &sh) {
    const R v[1] = {R(0)};
    return grp_reduce<kLive, R, 0, true>(g, sh, v, [](R *, int) {});
}

// component `part` (0 real, 1 imaginary) of a / b, as cdiv: the lanes of a
// warp share one division.  b is brought to unit size first (a power of two),
// so that its square stays in range.
__device__ __forceinline__ double cdiv_part(double2 a, double2 b, int part) {
    const int e = max(__double2hiint(b.x) & 0x7ff00000, __double2hiint(b.y) & 0x7ff00000) >> 20;   // biased exponent
    const double s = __hiloint2double((2046 - min(2045, max(1, e))) << 20, 0);
    b.x *= s;
    b.y *= s;
    const double d = b.x * b.x + b.y * b.y;
    const double y0 = part ? b.x : b.y, y1 = part ? -b.y : b.x;
    return (a.y * y0 + a.x * y1) / d * s;
}
__device__ __forceinline__ float cdiv_part(float2 a, float2 b, int part) {
    const float2 q = cdiv(a, b);
    return part ? q.y : q.x;
}
// a / b in every lane of a warp
template <class T> __device__ __forceinline__ T cdiv_pair(T a, T b, int lane) {
    const auto q = cdiv_part(a, b, lane & 1);
    T r;
    r.x = __shfl_sync(0xffffffffu, q, 0);
    r.y = __shfl_sync(0xffffffffu, q, 1);
    return r;
}
// component `part` of a b, as cmul
template <class T, class C = decltype(T::x)>
__device__ __forceinline__ C cmul_part(T a, T b, int part) {
    return part ? fma(a.x, b.y, a.y * b.x) : fma(a.x, b.x, -a.y * b.y);
}

// the slices of this CTA and its threads' walk over their rows
struct Own {
    int lo, hi, n;
    template <class F>
    __device__ __forceinline__ void rows(F f) const {
        for (int s = lo + (int)(threadIdx.x >> 5); s < hi; s += blockDim.x >> 5) {
            const int i = 32 * s + (threadIdx.x & 31);
            if (i < n) f(i);
        }
    }
};

// y = A x on the own slices, f(i, y, acc) per row
template <class V, int NV, class F>
struct PsEpi {
    using R = typename Ar<V>::R;
    using Acc = typename Ar<V>::Acc;
    F f;
    template <int N> __device__ void row(int i, V y, Acc (&acc)[N]) const { f(i, y, acc); }
};
// how a product gathers a vector: from global memory, or from its part `own`
// of each CTA's shared memory, `base` being the vector that staged columns address
template <int kLive, class V>
__device__ __forceinline__ auto ps_gather(const void *global, const V *own, const V *base) {
    if constexpr (kLive == 3) return GatherCluster<V>{(unsigned)((const char *)own - (const char *)base)};
    else return GatherLive<V>{(const V *)global};
}
// (wait: the barrier after which x may be gathered; false leaves the product out)
template <int kLive, class V, int NV, class G, class W, class F>
__device__ __forceinline__ void ps_product(const MatView<V> &A, const G &gx, const Own &o,
                                           typename Ar<V>::Acc (&acc)[NV], W wait, F f) {
    PsEpi<V, NV, F> epi{f};
#pragma unroll
    for (int j = 0; j < NV; ++j) Ar<V>::acc_zero(acc[j]);
    slice_rows<V, PsEpi<V, NV, F>, NV, kLive, G, W>(A, gx, epi, acc, o.lo + (int)(threadIdx.x >> 5), (int)(blockDim.x >> 5),
                                                o.hi, wait);
}

// scalars of a solve, one copy per CTA
template <class St>
struct PsState {
    St rho, alpha, omega, beta;
    St fac;            // alpha / (omega rho)
    double nb;
    double rel;        // the residual ratio, or, with lazy set,
    double rr;         // the squared residual norm it follows from
    double thr, top;   // squared norms in (thr, top] have not converged and have a finite ratio
    int iter, done, half, status, zero_x, lazy;
    __device__ double ratio() const { return lazy ? sqrt(rr) / nb : rel; }
    // whether a squared norm needs no exact test.  (Every CTA decides the same:
    // nothing that only one of them has, the history for one, enters.)
    __device__ bool clear(double ss) const { return ss > thr && ss <= top; }
};

// the threshold for squared norms of the test rel <= tol: a little above
// (tol nb)^2, so that what passes it is tested exactly
__device__ __forceinline__ double ps_threshold(double tol, double nb) {
    const double t = tol * nb, t2 = t * t * 1.000001;
    return t2 > 1e-290 ? t2 : 1e-290;
}
// squared norms up to it over nb^2 are at most 1e600: the ratio does not overflow
__device__ __forceinline__ double ps_top(double nb) {
    const double t = 1e300 * nb;
    return fmin(t * t, 1.7976931348623157e308);
}

// the BiCGStab iterations from r, rh, p = v = 0 in shared memory until the
// state is done; x is moved.  kOuter: the solve itself (binary64); else the
// inner solve of the refinement.  False when a wait expired.
template <int kLive, class V, bool kOuter>
__device__ bool ps_bicg_loop(const MatView<V> &A, const Ctl &ctl, const Own &o, Grp &g, PsShared &sh,
                             PsState<typename Ar<V>::St> &st, V *x, V *r, V *rh, V *p, V *v, V *s, V *t, V *gp, V *gs,
                             int *total, int in_maxit) {
    using T = Ar<V>;
    using R = typename T::R;
    const bool lead = g.rank == 0;
    const bool hist = kOuter && lead && ctl.hist;
    while (!st.done) {   // (every pass of the body ends in a barrier or leaves)
        const bool broke = cis_zero(st.rho);
        if (threadIdx.x == 0) {
            st.iter += 1;
            if (!kOuter) *total += 1;
            if (broke) { st.status = HZ_BREAKDOWN; st.done = 1; }
        }
        if (broke) break;   // (every thread of every CTA: rho is the same everywhere)
        {   // F1
            const auto beta = st.beta, omega = st.omega;
            o.rows([&](int i) {
                const V q = T::axpy(r[i], beta, T::axmy(p[i], omega, v[i]));
                p[i] = q;
                if constexpr (kLive != 3) gp[i] = q;
            });
        }
        {   // F2
            typename T::Acc acc[2];
            ps_product<kLive, V, 2>(A, ps_gather<kLive>(gp, p, x), o, acc, [&]() { return grp_sync<kLive, R>(g, sh); },
                             [&](int i, V y, auto &a) {
                                 v[i] = y;
                                 T::dotc(a[0], a[1], rh[i], y);
                             });
            if (sh.err) return false;
            const R red[2] = {T::total(acc[0]), T::total(acc[1])};
            if (!grp_reduce<kLive, R, 2, false>(g, sh, red, [&](R(&tot)[2], int lane) {
                    const auto sig = cmk(tot[0], tot[1]);
                    const R q = cdiv_part(st.rho, sig, lane & 1);
                    if (lane == 0 && cis_zero(sig)) { st.status = HZ_BREAKDOWN; st.done = 1; }
                    if (lane == 0) st.alpha.x = q;
                    if (lane == 1) st.alpha.y = q;
                }))
                return false;
        }
        if (st.done) break;
        const auto alpha = st.alpha;
        R ssum[1];
        {   // F3
            typename T::Acc acc[1];
            T::acc_zero(acc[0]);
            o.rows([&](int i) {
                const V q = T::axmy(r[i], alpha, v[i]);
                s[i] = q;
                if constexpr (kLive != 3) gs[i] = q;
                T::nrm2(acc[0], q);
            });
            ssum[0] = T::total(acc[0]);
        }
        typename T::Acc acc4[3];
        ps_product<kLive, V, 3>(   // F4, behind the barrier with ||s||^2
            A, ps_gather<kLive>(gs, s, x), o, acc4,
            [&]() {
                return grp_reduce<kLive, R, 1, true>(g, sh, ssum, [&](R(&tot)[1], int lane) {
                           const double ss = (double)tot[0];
                           if (lane != 0 || st.clear(ss)) return;
                           const double rel = sqrt(ss) / st.nb;
                           if (!finite_d(rel)) { st.status = HZ_ERR_NAN; st.done = 1; st.rel = rel; st.lazy = 0; }
                           else if (kOuter ? rel <= ctl.tol : (float)rel <= ctl.inner_tol) {
                               st.half = 1; st.rel = rel; st.lazy = 0; st.status = HZ_OK; st.done = 1;
                           }
                       }) &&
                       !st.done;
            },
            [&](int i, V y, auto &a) {
                t[i] = y;
                T::dotc(a[0], a[1], y, s[i]);
                T::nrm2(a[2], y);
            });
        if (sh.err) return false;
        if (st.done) {   // half-step exit: x += alpha p
            if (st.half) {
                o.rows([&](int i) { x[i] = T::axpy(x[i], alpha, p[i]); });
                if (hist && threadIdx.x == 0) ctl.hist[st.iter] = st.rel;
            }
            break;
        }
        {
            const R red[3] = {T::total(acc4[0]), T::total(acc4[1]), T::total(acc4[2])};
            if (!grp_reduce<kLive, R, 3, false>(g, sh, red, [&](R(&tot)[3], int lane) {
                    const R q = (lane & 1 ? tot[1] : tot[0]) / tot[2];
                    if (lane == 0 && tot[2] == R(0)) { st.status = HZ_BREAKDOWN; st.done = 1; }
                    if (lane == 0) st.omega.x = q;
                    if (lane == 1) st.omega.y = q;
                }))
                return false;
        }
        if (st.done) break;
        const auto omega = st.omega;
        {   // F5
            // beta = rn (alpha / (omega rho)): the last warp forms the factor
            // beside the pass, so that the barrier waits for no division
            if ((threadIdx.x >> 5) == (blockDim.x >> 5) - 1) {
                const int lane = threadIdx.x & 31;
                const R q = cdiv_part(cdiv_pair(alpha, omega, lane), st.rho, lane & 1);
                if (lane == 0) st.fac.x = q;
                if (lane == 1) st.fac.y = q;
            }
            typename T::Acc acc[3];
#pragma unroll
            for (int j = 0; j < 3; ++j) T::acc_zero(acc[j]);
            o.rows([&](int i) {
                const V si = s[i];
                x[i] = T::axpy(T::axpy(x[i], alpha, p[i]), omega, si);
                const V ri = T::axmy(si, omega, t[i]);
                r[i] = ri;
                T::dotc(acc[0], acc[1], rh[i], ri);
                T::nrm2(acc[2], ri);
            });
            const R red[3] = {T::total(acc[0]), T::total(acc[1]), T::total(acc[2])};
            if (!grp_reduce<kLive, R, 3, false>(g, sh, red, [&](R(&tot)[3], int lane) {
                    const auto rn = cmk(tot[0], tot[1]);
                    const R bq = cmul_part(rn, st.fac, lane & 1);
                    if (lane == 1) st.beta.y = bq;
                    if (lane != 0) return;
                    st.beta.x = bq;
                    st.rho = rn;
                    const double rr = (double)tot[2];
                    const int it = st.iter, maxit = kOuter ? ctl.maxit : in_maxit;
                    const bool last = it >= maxit || (!kOuter && *total >= ctl.maxit);
                    st.rr = rr;
                    st.lazy = 1;
                    const bool go = st.clear(rr) && !last && !cis_zero(omega);
                    if (go && !hist) return;
                    const double rel = sqrt(rr) / st.nb;
                    if (hist) ctl.hist[it] = rel;
                    if (go) return;
                    if (!finite_d(rel)) { st.status = HZ_ERR_NAN; st.done = 1; }
                    else if (kOuter ? rel <= ctl.tol : (float)rel <= ctl.inner_tol) { st.status = HZ_OK; st.done = 1; }
                    else if (cis_zero(omega)) { st.status = HZ_BREAKDOWN; st.done = 1; }
                    else if (last) { st.status = HZ_NOT_CONVERGED; st.done = 1; }
                }))
                return false;
        }
    }
    return true;
}

// start: the iterate from the caller's x0 (a restart keeps it)
__device__ __forceinline__ void ps_start_x(const PsSys &S, const Own &o, double2 *x) {
    const Ctl &c = S.ctl;
    o.rows([&](int i) {
        double2 v;
        if (c.restart) v = S.x[i];
        else if (c.x0_zero) v = make_double2(0.0, 0.0);
        else v = c.pre_d ? cmul(c.x[i], c.pre_d[i]) : c.x[i];
        if (x) x[i] = v;
        S.x[i] = v;
    });
}

// what the start product's reduction decides (tot = ||r||^2, ||b||^2)
__device__ __forceinline__ void ps_start_state(const Ctl &ctl, PsState<double2> &st, double rr, double bb, bool lead) {
    const double nb = sqrt(bb);
    const double2 one = make_double2(1.0, 0.0);
    st.nb = nb;
    st.thr = ps_threshold(ctl.tol, nb);
    st.top = ps_top(nb);
    st.half = 0;
    st.lazy = 0;
    st.rho = make_double2(rr, 0.0);
    st.alpha = one; st.omega = one;
    st.beta = make_double2(0.0, 0.0);
    st.done = 1;
    if (nb == 0.0) {
        st.rel = 0.0; st.status = HZ_OK; st.zero_x = 1;
        if (lead && ctl.hist && !ctl.restart) ctl.hist[0] = 0.0;
        return;
    }
    const double rel = sqrt(rr) / nb;
    st.rel = rel;
    if (lead && ctl.hist && !ctl.restart) ctl.hist[0] = rel;
    if (!finite_d(rel)) st.status = HZ_ERR_NAN;
    else if (rel <= ctl.tol) st.status = HZ_OK;
    else if (st.iter >= ctl.maxit) st.status = HZ_NOT_CONVERGED;
    else { st.status = HZ_NOT_CONVERGED; st.done = 0; }
}

// exit: true residual, info block, copy-out
template <int kLive>
__device__ void ps_finish(const PsSys &S, const MatView<double2> &A, const Own &o, Grp &g, PsShared &sh, const PsState<double2> &st,
                          const double2 *x) {
    const Ctl &c = S.ctl;
    o.rows([&](int i) { S.x[i] = x[i]; });
    double acc[1];
    ps_product<kLive, double2, 1>(A, ps_gather<kLive>(S.x, x, x), o, acc, [&]() { return grp_sync<kLive, double>(g, sh); },
                                  [&](int i, double2 y, auto &a) { Ar<double2>::nrm2(a[0], csub(c.b[i], y)); });
    if (sh.err) return;
    const bool lead = g.rank == 0;
    if (!grp_reduce<kLive, double, 1, true>(g, sh, acc, [&](double(&tot)[1], int lane) {
            if (!lead || lane != 0) return;
            S.info->iters = st.iter;
            S.info->status = st.status;
            S.info->restarts = 0;
            S.info->outer = 0;
            S.info->relres_rec = st.ratio();
            S.info->relres_true = st.zero_x ? 0.0 : sqrt(tot[0]) / st.nb;
            S.info->zero_x = st.zero_x;
        }))
        return;
    if (S.batched) return;   // S.x is the caller's vector
    o.rows([&](int i) {
        const double2 y = S.x[i];
        c.x[i] = st.zero_x ? make_double2(0.0, 0.0) : (c.pre_dinv ? cmul(y, c.pre_dinv[i]) : y);
    });
}

__device__ __forceinline__ const PsSys *ps_setup(const PsSys *sys, int nsys, Own &o, Grp &g, PsShared &sh) {
    int k = 0;
    if (nsys > 1) {   // the system of this CTA: the last one with cta0 <= blockIdx.x
        int hi = nsys - 1;
        while (k < hi) {
            const int mid = (k + hi + 1) >> 1;
            if (sys[mid].cta0 <= (int)blockIdx.x) k = mid;
            else hi = mid - 1;
        }
    }
    const PsSys *S = sys + k;
    g.lines = S->lines;
    g.err = S->err;
    g.rank = (int)blockIdx.x - S->cta0;
    g.size = S->ncta;
    g.epoch = 0ull;
    o.n = S->A.n;
    o.lo = (int)((int64_t)S->A.nsl * g.rank / g.size);
    o.hi = (int)((int64_t)S->A.nsl * (g.rank + 1) / g.size);
    if (threadIdx.x == 0) sh.err = 0;
    __syncthreads();
    return S;
}

extern __shared__ __align__(16) unsigned char ps_smem[];

// rows of a vector's part in shared memory (the same in every CTA of a cluster)
template <int kLive>
__device__ __forceinline__ int ps_rows(const Own &o, const Grp &g, int nsl) {
    return 32 * (kLive == 3 ? (nsl + g.size - 1) / g.size : o.hi - o.lo);
}

// The own slices of the stream in shared memory behind `at` (kLive 2), where
// they and the Krylov vectors fit there: a view that reads them from there.
// Between a barrier and its gathers there is then no other latency, and
// neither the columns nor the values are read through L2 in every pass (the
// fences of the barriers empty L1).
template <int kLive, class V>
__device__ __forceinline__ MatView<V> ps_stage(const MatView<V> &A, const Own &o, const Grp &g, void *at) {
    MatView<V> M = A;
    if constexpr (kLive >= 2) {
        const int b0 = A.sl_base[o.lo], cnt = 32 * (A.sl_base[o.hi] - b0), ns = o.hi - o.lo;
        const size_t off = (size_t)32 * b0;
        unsigned long long *mask = (unsigned long long *)at;
        char *q = (char *)(mask + ns);
        if constexpr (std::is_same<V, double2>::value) {
            double *re = (double *)q, *im = re + cnt;
            q = (char *)(im + cnt);
            for (int i = threadIdx.x; i < cnt; i += blockDim.x) {
                re[i] = A.sl_re[off + i];
                im[i] = A.sl_im[off + i];
            }
            for (int i = threadIdx.x; i < ns; i += blockDim.x) mask[i] = A.sl_mask[o.lo + i];
            M.sl_re = re - off;
            M.sl_im = im - off;
            M.sl_mask = mask - o.lo;
        } else {
            float2 *v = (float2 *)q;
            q = (char *)(v + cnt);
            for (int i = threadIdx.x; i < cnt; i += blockDim.x) v[i] = A.sl_val32[off + i];
            M.sl_val32 = v - off;
        }
        int *col = (int *)q, *base = col + cnt;
        for (int i = threadIdx.x; i < cnt; i += blockDim.x) {
            int c = A.sl_col[off + i];
            if (kLive == 3 && c >= 0) {   // the address of the first vector's entry c in the CTA that owns it
                const int r = (int)(((int64_t)((c >> 5) + 1) * g.size - 1) / A.nsl);
                const int lo = (int)((int64_t)A.nsl * r / g.size);
                c = (int)cluster_map(smem_addr(ps_smem) + (unsigned)(c - 32 * lo) * (unsigned)sizeof(V), r);
            }
            col[i] = c;
        }
        for (int i = threadIdx.x; i <= ns; i += blockDim.x) base[i] = A.sl_base[o.lo + i];
        M.sl_col = col - off;
        M.sl_base = base - o.lo;
        __syncthreads();
    }
    return M;
}

// BiCGStab in binary64
template <int kLive>
__global__ void __launch_bounds__(kPsMaxWarps * 32, 1) k_ps_bicg(const PsSys *sys, int nsys) {
    __shared__ PsShared sh;
    __shared__ PsState<double2> st;
    Own o;
    Grp g;
    const PsSys &S = *ps_setup(sys, nsys, o, g, sh);
    const Ctl &ctl = S.ctl;
    const int m = ps_rows<kLive>(o, g, S.A.nsl);
    // vectors indexed by row: each points 32 lo entries before its part
    double2 *base = reinterpret_cast<double2 *>(ps_smem) - 32 * o.lo;
    double2 *x = base, *r = base + m, *rh = base + 2 * m, *p = base + 3 * m, *v = base + 4 * m, *s = base + 5 * m,
            *t = base + 6 * m;
    const MatView<double2> M = ps_stage<kLive>(S.A, o, g, reinterpret_cast<double2 *>(ps_smem) + 7 * m);
    if (threadIdx.x == 0) {
        st.iter = ctl.restart ? S.info->iters : 0;
        st.zero_x = 0;
    }
    ps_start_x(S, o, x);
    double acc[2];
    ps_product<kLive, double2, 2>(M, ps_gather<kLive>(S.x, x, x), o, acc, [&]() { return grp_sync<kLive, double>(g, sh); },
                           [&](int i, double2 y, auto &a) {
                               const double2 bi = ctl.b[i], ri = csub(bi, y);
                               r[i] = ri;
                               rh[i] = ri;
                               p[i] = make_double2(0.0, 0.0);
                               v[i] = make_double2(0.0, 0.0);
                               Ar<double2>::nrm2(a[0], ri);
                               Ar<double2>::nrm2(a[1], bi);
                           });
    if (sh.err) return;
    if (!grp_reduce<kLive, double, 2, true>(g, sh, acc, [&](double(&tot)[2], int lane) {
            if (lane == 0) ps_start_state(ctl, st, tot[0], tot[1], g.rank == 0);
        }))
        return;
    if (!ps_bicg_loop<kLive, double2, true>(M, ctl, o, g, sh, st, x, r, rh, p, v, s, t, (double2 *)S.g0, (double2 *)S.g1,
                                     nullptr, 0))
        return;
    ps_finish<kLive>(S, M, o, g, sh, st, x);
}

// Mixed precision: outer residuals and x += d in binary64, the inner solve
// on the complex64 copy.  The rules are those of EpiOuter (bicgstab.cu): the
// refinement keeps the iterate with the smallest outer residual and stops
// when a step fails to reduce it.
template <int kLive>
__global__ void __launch_bounds__(kPsMaxWarps * 32, 1) k_ps_mixed(const PsSys *sys, int nsys) {
    __shared__ PsShared sh;
    __shared__ PsState<float2> in;
    struct Outer {
        double rel, best;
        int outer, done, status, zero_x, save, use_best, total;
    };
    __shared__ Outer ou;
    Own o;
    Grp g;
    const PsSys &S = *ps_setup(sys, nsys, o, g, sh);
    const Ctl &ctl = S.ctl;
    const bool lead = g.rank == 0;
    const int m = ps_rows<kLive>(o, g, S.A.nsl);
    float2 *base = reinterpret_cast<float2 *>(ps_smem) - 32 * o.lo;
    float2 *d = base, *r = base + m, *rh = base + 2 * m, *p = base + 3 * m, *v = base + 4 * m, *s = base + 5 * m,
           *t = base + 6 * m;
    const MatView<float2> M = ps_stage<kLive>(S.A32, o, g, reinterpret_cast<float2 *>(ps_smem) + 7 * m);
    if (threadIdx.x == 0) {
        ou.outer = 0; ou.done = 0; ou.status = HZ_NOT_CONVERGED; ou.zero_x = 0;
        ou.best = INFINITY; ou.save = 0; ou.use_best = 0; ou.total = 0;
    }
    ps_start_x(S, o, nullptr);
    for (int run = 0; run <= ctl.max_outer; ++run) {
        double acc[3];
        ps_product<1, double2, 3>(S.A, GatherLive<double2>{S.x}, o, acc, [&]() { return grp_sync<kLive, double>(g, sh); },
                               [&](int i, double2 y, auto &a) {
                                   const double2 bi = ctl.b[i], ri = csub(bi, y);
                                   const float2 r32 = to_c64(ri), z = make_float2(0.f, 0.f);
                                   r[i] = r32;
                                   rh[i] = r32;
                                   p[i] = z;
                                   v[i] = z;
                                   d[i] = z;
                                   Ar<double2>::nrm2(a[0], ri);
                                   Ar<double2>::nrm2(a[1], bi);
                                   Ar<double2>::nrm2(a[2], to_c128(r32));
                               });
        if (sh.err) return;
        if (!grp_reduce<kLive, double, 3, true>(g, sh, acc, [&](double(&tot)[3], int lane) {
                if (lane != 0) return;
                const double nb = sqrt(tot[1]);
                ou.done = 1;
                if (nb == 0.0) {
                    ou.rel = 0.0; ou.status = HZ_OK; ou.zero_x = 1;
                    if (lead && ctl.hist) ctl.hist[ou.outer] = 0.0;
                    return;
                }
                const double rel = sqrt(tot[0]) / nb;
                ou.rel = rel;
                if (lead && ctl.hist) ctl.hist[ou.outer] = rel;
                ou.save = 0;
                if (!finite_d(rel)) { ou.status = HZ_ERR_NAN; ou.use_best = ou.outer > 0; }
                else if (rel <= ctl.tol) ou.status = HZ_OK;
                else if (rel >= ou.best) { ou.status = HZ_NOT_CONVERGED; ou.use_best = 1; }
                else if (ou.outer >= ctl.max_outer || ou.total >= ctl.maxit) ou.status = HZ_NOT_CONVERGED;
                else {
                    ou.done = 0;
                    ou.best = rel;
                    ou.save = 1;
                    ou.outer += 1;
                    const float2 one = make_float2(1.f, 0.f);
                    in.rho = make_float2((float)tot[2], 0.f);
                    in.alpha = one; in.omega = one;
                    in.beta = make_float2(0.f, 0.f);
                    in.nb = (double)sqrtf((float)tot[2]);
                    in.thr = ps_threshold((double)ctl.inner_tol, in.nb);
                    in.top = ps_top(in.nb);
                    in.rel = 1.0; in.lazy = 0;
                    in.iter = 0; in.half = 0; in.status = HZ_NOT_CONVERGED;
                    in.done = in.nb == 0.0 ? 1 : 0;
                }
            }))
            return;
        if (ou.done) break;
        if (!ps_bicg_loop<kLive, float2, false>(M, ctl, o, g, sh, in, d, r, rh, p, v, s, t, (float2 *)S.g0,
                                         (float2 *)S.g1, &ou.total, ctl.inner_maxit))
            return;
        const bool save = ou.save != 0;
        o.rows([&](int i) {
            const double2 xi = S.x[i];
            if (save) S.xbest[i] = xi;
            S.x[i] = Ar<double2>::sub(xi, to_c128(make_float2(-d[i].x, -d[i].y)));
        });
    }
    const bool best = ou.use_best != 0;
    if (lead && threadIdx.x == 0) {
        S.info->iters = ou.total;
        S.info->status = ou.status;
        S.info->outer = ou.outer;
        S.info->relres_rec = S.info->relres_true = best ? ou.best : ou.rel;
        S.info->zero_x = ou.zero_x;
    }
    o.rows([&](int i) {
        const double2 y = best ? S.xbest[i] : S.x[i];
        ctl.x[i] = ou.zero_x ? make_double2(0.0, 0.0) : (ctl.pre_dinv ? cmul(y, ctl.pre_dinv[i]) : y);
    });
}

// TFQMR in binary64 (the passes Q1..Q4 of tfqmr.cu).  The half-step scalars
// are kept as squares: with W = ||w||^2, theta^2 = W / tau^2,
// c^2 = tau^2 / (tau^2 + W), tau^2 <- tau^2 W / (tau^2 + W), so that neither
// square roots nor chains of divisions stand between a barrier and the next
// pass.
struct PsTq {
    double2 eta;            // of the last half step
    double2 coef, etax;     // d and x coefficients of this half step (eta / G)
    double tau2, th2, xs;   // tau^2, theta^2 of the last half step, 1 / G
    double q[5];            // scratch: the five divisions of a half step
    int m, stop, pend;
};

// One half step from W, and beta = rho1 / rho for the second one, by all lanes
// of a warp with one division each: lanes 0, 1 coef = theta^2 eta / alpha,
// 2 c^2, 3 the factor of tau^2, 4 the new theta^2, 5, 6 beta.
__device__ __forceinline__ void ps_tq_half(PsTq &t, double2 alpha, double W, double2 rho1, double2 rho, double2 &beta,
                                           int lane) {
    const bool first = lane < 2;
    const double2 te = make_double2(t.th2 * t.eta.x, t.th2 * t.eta.y);
    const double2 a = first ? te : rho1;
    double2 b = first ? alpha : rho;
    const int part = first ? lane : lane == 6;
    const double tau2 = t.tau2, s = tau2 + W;
    // a / b as cdiv_part, up to the division
    const int e = max(__double2hiint(b.x) & 0x7ff00000, __double2hiint(b.y) & 0x7ff00000) >> 20;
    const double sc = __hiloint2double((2046 - min(2045, max(1, e))) << 20, 0);
    b.x *= sc;
    b.y *= sc;
    const double d = b.x * b.x + b.y * b.y;
    const double y0 = part ? b.x : b.y, y1 = part ? -b.y : b.x;
    const double n = a.y * y0 + a.x * y1;
    const bool mid = lane >= 2 && lane < 5;
    const double num = mid ? (lane == 2 ? tau2 : W) : n, den = mid ? (lane == 4 ? tau2 : s) : d;
    const double q = num / den * (mid ? 1.0 : sc);
    if (lane < 5) t.q[lane] = q;
    if (lane == 5) beta.x = q;
    if (lane == 6) beta.y = q;
    __syncwarp();
    if (lane == 0) {
        const bool z = tau2 == 0.0;
        const double c2 = z ? 1.0 : t.q[2];
        t.coef = make_double2(t.q[0], t.q[1]);
        t.tau2 = z ? 0.0 : tau2 * t.q[3];
        t.th2 = z ? 0.0 : t.q[4];
        t.eta = make_double2(c2 * alpha.x, c2 * alpha.y);
        t.etax = make_double2(t.eta.x * t.xs, t.eta.y * t.xs);
        t.m += 1;
    }
}

template <int kLive>
__global__ void __launch_bounds__(kPsMaxWarps * 32, 1) k_ps_tfqmr(const PsSys *sys, int nsys) {
    using A = Ar<double2>;
    __shared__ PsShared sh;
    __shared__ PsState<double2> st;
    __shared__ PsTq q;
    Own o;
    Grp g;
    const PsSys &S = *ps_setup(sys, nsys, o, g, sh);
    const Ctl &ctl = S.ctl;
    const bool lead = g.rank == 0, hist = lead && ctl.hist;
    const int m = ps_rows<kLive>(o, g, S.A.nsl);
    double2 *base = reinterpret_cast<double2 *>(ps_smem) - 32 * o.lo;
    double2 *x = base, *w = base + m, *u1 = base + 2 * m, *u2 = base + 3 * m, *v = base + 4 * m, *d = base + 5 * m,
            *au1 = base + 6 * m, *au = base + 7 * m, *rh = base + 8 * m;
    double2 *gu1 = (double2 *)S.g0, *gu2 = (double2 *)S.g1;
    const MatView<double2> M = ps_stage<kLive>(S.A, o, g, reinterpret_cast<double2 *>(ps_smem) + 9 * m);
    if (threadIdx.x == 0) {
        st.iter = ctl.restart ? S.info->iters : 0;
        st.zero_x = 0;
    }
    ps_start_x(S, o, x);
    {
        double acc[2];
        ps_product<kLive, double2, 2>(M, ps_gather<kLive>(S.x, x, x), o, acc, [&]() { return grp_sync<kLive, double>(g, sh); },
                               [&](int i, double2 y, auto &a) {
                                   const double2 bi = ctl.b[i], ri = csub(bi, y), z = make_double2(0.0, 0.0);
                                   w[i] = ri;
                                   u1[i] = ri;
                                   gu1[i] = ri;
                                   rh[i] = ri;
                                   d[i] = z;
                                   v[i] = z;
                                   A::nrm2(a[0], ri);
                                   A::nrm2(a[1], bi);
                               });
        if (sh.err) return;
        if (!grp_reduce<kLive, double, 2, true>(g, sh, acc, [&](double(&tot)[2], int lane) {
                if (lane != 0) return;
                q.tau2 = tot[0];
                q.th2 = 0.0;
                q.eta = make_double2(0.0, 0.0);
                q.m = 0;
                q.stop = 0;
                q.pend = 0;
                q.xs = 1.0;
                ps_start_state(ctl, st, tot[0], tot[1], lead);
            }))
            return;
    }
    bool first = true;   // the start's product: u1 is already published
    while (!st.done) {
        {   // Q4: au1 = A u1, v += au1, <r^, v>, ||v||^2 -> alpha
            double acc[3];
            ps_product<kLive, double2, 3>(M, ps_gather<kLive>(gu1, u1, x), o, acc, [&]() { return first || grp_sync<kLive, double>(g, sh); },
                                   [&](int i, double2 y, auto &a) {
                                       au1[i] = y;
                                       const double2 vi = A::add(y, v[i]);
                                       v[i] = vi;
                                       A::dotc(a[0], a[1], rh[i], vi);
                                       A::nrm2(a[2], vi);
                                   });
            first = false;
            if (sh.err) return;
            if (!grp_reduce<kLive, double, 3, false>(g, sh, acc, [&](double(&tot)[3], int lane) {
                    const double2 sig = make_double2(tot[0], tot[1]);
                    const double c = cdiv_part(st.rho, sig, lane & 1);
                    const bool brk = cis_zero(st.rho) || cis_zero(sig);
                    if (lane == 1) st.alpha.y = c;
                    if (lane != 0) return;
                    st.alpha.x = c;
                    if (!(tot[2] < kTqBig) || !(q.tau2 < kTqBig)) q.pend = 1;
                    if (brk) { st.status = HZ_BREAKDOWN; st.done = 1; }
                    else if (st.iter >= ctl.maxit) { st.status = HZ_NOT_CONVERGED; st.done = 1; }
                }))
                return;
        }
        if (st.done) break;
        const double2 alpha = st.alpha;
        double ww[1] = {0.0};
        const bool pend = q.pend != 0;
        o.rows([&](int i) {   // Q1 (with the range guard's scaling)
            double2 u1i = u1[i], vi = v[i], wi = w[i], ai = au1[i];
            if (pend) {
                u1i = A::pow2(u1i, kTqShrink);
                vi = A::pow2(vi, kTqShrink);
                wi = A::pow2(wi, kTqShrink);
                ai = A::pow2(ai, kTqShrink);
                u1[i] = u1i;
                v[i] = vi;
                au1[i] = ai;
                d[i] = A::pow2(d[i], kTqShrink);
            }
            const double2 u = A::axmy(u1i, alpha, vi);
            u2[i] = u;
            if constexpr (kLive != 3) gu2[i] = u;
            wi = A::axmy(wi, alpha, ai);
            w[i] = wi;
            A::nrm2(ww[0], wi);
        });
        double acc[3];
        // Q2, behind the barrier with ||w||^2: au = A u2; d, x and w
        double2 coef, eta;
        ps_product<kLive, double2, 3>(
            M, ps_gather<kLive>(gu2, u2, x), o, acc,
            [&]() {
                const bool ok = grp_reduce<kLive, double, 1, true>(g, sh, ww, [&](double(&tot)[1], int lane) {
                    if (pend && lane == 0) {
                        q.pend = 0;
                        q.tau2 *= kTqShrink * kTqShrink;
                        st.rho = make_double2(st.rho.x * kTqShrink, st.rho.y * kTqShrink);
                        q.xs /= kTqShrink;
                    }
                    __syncwarp();
                    double2 none;
                    ps_tq_half(q, alpha, tot[0], alpha, alpha, none, lane);
                });
                coef = q.coef;
                eta = q.etax;
                return ok;
            },
            [&](int i, double2 y, auto &a) {
                au[i] = y;
                const double2 di = A::axpy(u1[i], coef, d[i]);
                d[i] = di;
                x[i] = A::axpy(x[i], eta, di);
                const double2 wi = A::axmy(w[i], alpha, y);
                w[i] = wi;
                A::nrm2(a[0], wi);
                A::dotc(a[1], a[2], rh[i], wi);
            });
        if (sh.err) return;
        if (!grp_reduce<kLive, double, 3, false>(g, sh, acc, [&](double(&tot)[3], int lane) {
                const double2 rho1 = make_double2(tot[1], tot[2]);
                ps_tq_half(q, alpha, tot[0], rho1, st.rho, st.beta, lane);
                if (lane != 0) return;
                const int it = st.iter + 1;
                st.iter = it;
                st.rho = rho1;
                // squared bound: (m + 1) (tau / G)^2
                const double rr = ((double)q.m + 1.0) * (q.tau2 * q.xs) * q.xs;
                st.rr = rr;
                st.lazy = 1;
                const bool go = st.clear(rr);
                if (go && !hist) return;
                const double rel = sqrt(rr) / st.nb;
                if (hist) ctl.hist[it] = rel;
                if (go) return;
                if (!finite_d(rel)) { st.status = HZ_ERR_NAN; q.stop = 1; }
                else if (rel <= ctl.tol) { st.status = HZ_OK; q.stop = 1; }
            }))
            return;
        const double2 coef2 = q.coef, eta2 = q.etax, beta = st.beta;
        const bool stop = q.stop != 0;
        o.rows([&](int i) {   // Q3
            const double2 ui = u2[i], di = A::axpy(ui, coef2, d[i]);
            d[i] = di;
            x[i] = A::axpy(x[i], eta2, di);
            if (!stop) {
                const double2 u = A::axpy(w[i], beta, ui);
                u1[i] = u;
                if constexpr (kLive != 3) gu1[i] = u;
                v[i] = A::axpy(A::zero(), beta, A::axpy(au[i], beta, v[i]));
            }
        });
        if (stop) break;
    }
    ps_finish<kLive>(S, M, o, g, sh, st, x);
}

// ---------------------------------------------------------------------------
// host side
struct PsMethod {
    void *kern[3];   // the matrix through L2; staged in shared memory; and one cluster
    int vecs;        // Krylov vectors in shared memory
    int elem;        // bytes per element
    int slot;        // bytes per slot of the staged stream
};
static PsMethod ps_method(PsKind k) {
    switch (k) {
        case PS_BICG: return {{(void *)k_ps_bicg<1>, (void *)k_ps_bicg<2>, (void *)k_ps_bicg<3>}, 7, 16, 20};
        case PS_MIXED: return {{(void *)k_ps_mixed<1>, (void *)k_ps_mixed<2>, (void *)k_ps_mixed<3>}, 7, 8, 12};
        default: return {{(void *)k_ps_tfqmr<1>, (void *)k_ps_tfqmr<2>, (void *)k_ps_tfqmr<3>}, 9, 16, 20};
    }
}
constexpr int kPsSmem = 212 * 1024;   // dynamic shared memory of a CTA at most (227 KB less the static part)

static int ps_ctas(const hz_mat *A, int num_sms) { return std::min(std::min(num_sms, kPsMaxCta), A->nsl); }

// the slices one CTA may own
static int ps_slices(PsKind k) {
    const PsMethod m = ps_method(k);
    return kPsSmem / (m.vecs * m.elem * 32);
}

static bool ps_layout(const hz_mat *A) {
    return A->nsl > 0 && !is_ff_kind(A->spmv_kind) && d64_kind(A, A->spmv_kind) == HZ_SPMV_FLAT64P &&
           profile_unroll() <= 0;
}

bool ps_fits(const hz_mat *A, PsKind k) {
    DevInfo d;
    if (!ps_layout(A) || dev_info(&d) != HZ_OK) return false;
    const int c = ps_ctas(A, d.num_sms);
    return (A->nsl + c - 1) / c <= ps_slices(k);
}

// shared memory of the largest CTA of one system on c CTAs, with its part of
// the stream or without
static size_t ps_smem_bytes(const hz_mat *A, const PsMethod &m, int c, bool stage) {
    size_t most = 0;
    for (int r = 0; r < c; ++r) {
        const int lo = (int)((int64_t)A->nsl * r / c), hi = (int)((int64_t)A->nsl * (r + 1) / c);
        size_t b = (size_t)(hi - lo) * 32 * m.vecs * m.elem;
        if (stage) b += (size_t)32 * (A->sl_base_h[hi] - A->sl_base_h[lo]) * m.slot + (size_t)(hi - lo) * 12 + 4;
        most = std::max(most, b);
    }
    return most;
}

// launch `kind` over the systems h[0..ns) on the handles A (device copy
// dsys), whose cta0/ncta are set
static cudaError_t ps_launch(PsKind kind, hz_mat *const *A, const PsSys *h, int ns, PsSys *dsys, cudaStream_t s) {
    const PsMethod m = ps_method(kind);
    int per = 1, grid = 0;
    size_t plain = 0, staged = 0;
    for (int k = 0; k < ns; ++k) {
        per = std::max(per, (h[k].A.nsl + h[k].ncta - 1) / h[k].ncta);
        grid += h[k].ncta;
        plain = std::max(plain, ps_smem_bytes(A[k], m, h[k].ncta, false));
        staged = std::max(staged, ps_smem_bytes(A[k], m, h[k].ncta, true));
    }
    const bool st = staged <= (size_t)kPsSmem;
    const int warps = std::min(kPsMaxWarps, std::max(kPsMinWarps, (per + 3) / 4 * 4));
    void *kern = m.kern[st ? 1 : 0];
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, kPsSmem);
    if (e != cudaSuccess) return e;
    void *args[] = {&dsys, &ns};
    return cudaLaunchCooperativeKernel(kern, dim3(grid), dim3(32 * warps), args, st ? staged : plain, s);
}

// One cluster for the smallest systems: on 16 SMs the gathers and sums go
// through the cluster's shared memory, a pass waits for no L2 latency, but has
// a tenth of the binary64 pipes.  us per iteration, cluster / all SMs:
//   unknowns           512          1.7k         4.1k         5.8k         8k          13.8k
//   BiCGStab    15.4 / 21.0  16.0 / 21.2  17.9 / 22.8  20.7 / 23.9  24.1 / 23.4  24.6* / 24.5
//   TFQMR       15.5 / 19.3  15.1 / 20.4  17.6 / 21.5  20.8 / 22.9  24.4 / 22.8
//   mixed        7.0 /  9.7   6.7 / 10.5   7.3 / 11.9   7.3 / 11.9   7.9 / 12.3   9.0 / 12.5
// (* does not fit).  So up to 12 slices per CTA in binary64, 32 in the mixed
// method, whose passes run on the binary32 pipes, where the staged stream fits
// beside the vectors: with 12 slices rows of up to 22 entries (TFQMR 21), with
// 32 rows of up to 13 (28 slices with rows of 15); wider ones take every SM.
// The CTAs (0: not this way) and their shared memory:
static int ps_cluster(const hz_mat *A, PsKind kind, size_t *smem) {
    const PsMethod m = ps_method(kind);
    if (A->sl_long) return 0;   // (their columns are not staged)
    int c = 1;
    while (c < kPsMaxCluster && c < A->nsl) c *= 2;
    const int per = (A->nsl + c - 1) / c;
    if (per > (kind == PS_MIXED ? 32 : 12)) return 0;
    int steps = 0;
    for (int r = 0; r < c; ++r)
        steps = std::max(steps, A->sl_base_h[(int64_t)A->nsl * (r + 1) / c] - A->sl_base_h[(int64_t)A->nsl * r / c]);
    *smem = (size_t)per * 32 * m.vecs * m.elem + (size_t)32 * steps * m.slot + (size_t)per * 12 + 4;
    return *smem <= (size_t)kPsSmem ? c : 0;
}

// (clusters: how many the device holds at once, asked for at -1)
static cudaError_t ps_launch_cluster(PsKind kind, int ctas, int slices, size_t smem, PsSys *dsys, cudaStream_t s,
                                     int *clusters) {
    void *kern = ps_method(kind).kern[2];
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, kPsSmem);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    if (e != cudaSuccess) return e;
    const int warps = std::min(kPsMaxWarps, std::max(kPsMinWarps, (slices + 3) / 4 * 4));
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(ctas);
    cfg.blockDim = dim3(32 * warps);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = ctas;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    if (*clusters < 0) {
        e = cudaOccupancyMaxActiveClusters(clusters, kern, &cfg);
        if (e != cudaSuccess) { *clusters = -1; return e; }
    }
    if (*clusters == 0) return cudaErrorLaunchOutOfResources;
    int ns = 1;
    void *args[] = {&dsys, &ns};
    return cudaLaunchKernelExC(&cfg, kern, args);
}

// what a launch says that the device has no room for (nothing ran; not sticky)
static bool ps_no_room(cudaError_t e) {
    return e == cudaErrorCooperativeLaunchTooLarge || e == cudaErrorLaunchOutOfResources ||
           e == cudaErrorInvalidClusterSize || e == cudaErrorInvalidConfiguration || e == cudaErrorNotSupported;
}

struct PsSolver {
    int n = 0;
    int clusters = -1;         // clusters of its size that the device holds (-1: not asked)
    void *mem = nullptr;       // lines, err, info, system, vectors
    PsSys *dsys = nullptr;
    Info *dinfo = nullptr;
    double2 *x = nullptr, *xbest = nullptr;
    void *g0 = nullptr, *g1 = nullptr;
    PsLine *lines = nullptr;
    int *err = nullptr;
    PsSys *hsys = nullptr;     // pinned
    struct Back {
        Info info;
        int err;
    } *hback = nullptr;        // pinned
};

void ps_solver_free(void *p) {
    PsSolver *S = (PsSolver *)p;
    if (!S) return;
    cudaFree(S->mem);
    cudaFreeHost(S->hsys);
    cudaFreeHost(S->hback);
    delete S;
}

constexpr size_t kPsLineBytes = sizeof(PsLine) * 2 * kPsMaxCta;
// lines, then the error word and the info block behind them
constexpr size_t kPsErrOff = kPsLineBytes, kPsInfoOff = kPsErrOff + 64, kPsSysOff = kPsInfoOff + 128;

static hz_status ps_get(hz_mat *A, PsKind kind, PsSolver **out) {
    PsSolver *S = (PsSolver *)A->solver_ps[kind];
    if (!S) {
        S = new PsSolver();
        A->solver_ps[kind] = S;   // freed with the handle even if an allocation below fails
        S->n = A->n;
    }
    if (!S->mem) {
        const size_t vb = ((size_t)A->n * 16 + 255) & ~(size_t)255;
        const size_t head = (kPsSysOff + sizeof(PsSys) + 255) & ~(size_t)255;
        if (!S->hsys) HZ_CUDA(cudaMallocHost((void **)&S->hsys, sizeof(PsSys)));
        if (!S->hback) HZ_CUDA(cudaMallocHost((void **)&S->hback, sizeof(PsSolver::Back)));
        char *m = nullptr;
        HZ_CUDA(cudaMalloc((void **)&m, head + vb * (kind == PS_MIXED ? 4 : 3)));
        S->mem = m;
        S->lines = (PsLine *)m;
        S->err = (int *)(m + kPsErrOff);
        S->dinfo = (Info *)(m + kPsInfoOff);
        S->dsys = (PsSys *)(m + kPsSysOff);
        S->x = (double2 *)(m + head);
        S->g0 = m + head + vb;
        S->g1 = m + head + 2 * vb;
        S->xbest = kind == PS_MIXED ? (double2 *)(m + head + 3 * vb) : nullptr;
    }
    *out = S;
    return HZ_OK;
}

hz_status ps_solve(hz_mat *A, PsKind kind, const Ctl &c, Info *out, int *restarts, cudaStream_t s, bool *taken) {
    *taken = true;
    PsSolver *S = nullptr;
    HZ_TRY(ps_get(A, kind, &S));
    DevInfo d;
    HZ_TRY(dev_info(&d));
    PsSys &h = *S->hsys;
    h = PsSys{};
    h.A = mat_view<double2>(A);
    if (kind == PS_MIXED) h.A32 = mat_view<float2>(A);
    h.x = S->x; h.xbest = S->xbest; h.g0 = S->g0; h.g1 = S->g1;
    h.ctl = c;
    h.info = S->dinfo; h.lines = S->lines; h.err = S->err;
    h.cta0 = 0;
    size_t smem = 0;
    const int cl = ps_cluster(A, kind, &smem);
    Way way = cl ? Way::cluster : Way::all_sms;
    *restarts = 0;
    for (int run = 0;; ++run) {
        cudaError_t e = cudaSuccess;
        const bool ok = first_way(way, [&](Way w) {
            h.ncta = w == Way::cluster ? cl : ps_ctas(A, d.num_sms);
            e = cudaMemcpyAsync(S->dsys, &h, sizeof(PsSys), cudaMemcpyHostToDevice, s);
            if (e == cudaSuccess) e = cudaMemsetAsync(S->lines, 0, kPsErrOff + sizeof(int), s);
            if (e != cudaSuccess) return Launch::error;
            e = w == Way::cluster ? ps_launch_cluster(kind, cl, (A->nsl + cl - 1) / cl, smem, S->dsys, s, &S->clusters)
                                  : ps_launch(kind, &A, &h, 1, S->dsys, s);
            if (e == cudaSuccess) return Launch::done;
            if (!ps_no_room(e)) return Launch::error;
            cudaGetLastError();
            // (h is written again only when the copy above has read it)
            e = cudaStreamSynchronize(s);
            return e == cudaSuccess ? Launch::no_room : Launch::error;
        });
        if (!ok) return cuda_fail(e, "hz_zsolve", __FILE__, __LINE__);
        if (way == Way::graph) {
            if (run == 0) { *taken = false; return HZ_OK; }
            return cuda_fail(cudaErrorCooperativeLaunchTooLarge, "hz_zsolve (restart)", __FILE__, __LINE__);
        }
        HZ_CUDA(cudaMemcpyAsync(&S->hback->info, S->dinfo, sizeof(Info), cudaMemcpyDeviceToHost, s));
        HZ_CUDA(cudaMemcpyAsync(&S->hback->err, S->err, sizeof(int), cudaMemcpyDeviceToHost, s));
        HZ_CUDA(cudaStreamSynchronize(s));
        if (S->hback->err) {
            set_error("hz_zsolve: a barrier wait of the persistent solver expired");
            return HZ_ERR_TIMEOUT;
        }
        *out = S->hback->info;
        // the recursive residual met the tolerance, the true one did not: once more from here
        if (kind == PS_MIXED || run || out->status != HZ_OK || !(out->relres_true > c.tol) || out->iters >= c.maxit)
            return HZ_OK;
        *restarts = 1;
        h.ctl.restart = 1;
    }
}

// ---------------------------------------------------------------------------
// a sweep: every system on CTAs of its own
//
// The systems run at their own pace, each with barriers among its own CTAs
// only, instead of advancing together through grid-wide phases
// (batched.cu, 75 to 95 us per iteration for any sweep of small systems).
// CTAs are shared out by rows (sweep_plan).  Twelve boxes of 15^3 to 24^3 unknowns: 10.4 -> 3.8 ms.
struct PsBatch {
    std::atomic_flag busy = ATOMIC_FLAG_INIT;
    void *mem = nullptr;
    size_t bytes = 0;
};

void ps_batch_free(void *p) {
    PsBatch *B = (PsBatch *)p;
    if (!B) return;
    cudaFree(B->mem);
    delete B;
}

bool ps_batch_plan(hz_mat *const *A, int ns, std::vector<int> *ncta) {
    DevInfo d;
    if (dev_info(&d) != HZ_OK) return false;
    std::vector<int> nsl(ns, 0);
    for (int k = 0; k < ns; ++k) {
        if (A[k]->n == 0) continue;
        if (!ps_layout(A[k])) return false;
        nsl[k] = A[k]->nsl;
    }
    return sweep_plan(nsl, d.num_sms, kPsMaxCta, ps_slices(PS_BICG), ncta);
}

hz_status ps_solve_batched(hz_mat *const *A, int ns, const std::vector<int> &ncta, const double2 *const *b,
                           double2 *const *x, double tol, int maxit, Info *out, cudaStream_t s, bool *taken) {
    *taken = true;
    std::vector<hz_mat *> act;
    std::vector<int> idx;
    for (int k = 0; k < ns; ++k) {
        out[k] = Info{};
        if (ncta[k]) { act.push_back(A[k]); idx.push_back(k); }
    }
    const int na = (int)act.size();
    if (na == 0) return HZ_OK;
    auto up = [](size_t v) { return (v + 255) & ~(size_t)255; };
    // error word and info blocks, lines, systems, two vectors per system
    const size_t info_b = up(256 + sizeof(Info) * na);
    size_t line_n = 0, vec_b = 0;
    for (int q = 0; q < na; ++q) {
        line_n += 2 * (size_t)ncta[idx[q]];
        vec_b += 2 * up((size_t)act[q]->n * 16);
    }
    const size_t zero_b = info_b + up(line_n * sizeof(PsLine)), sys_b = up(sizeof(PsSys) * na);
    const size_t bytes = zero_b + sys_b + vec_b;
    // the workspace stays with the first handle; a call that finds it in use
    // (another thread sweeping over the same handles) takes its own
    PsBatch *B;
    {
        static std::mutex mu;   // (the pointer is read under it too: another thread may be setting it)
        std::lock_guard<std::mutex> lk(mu);
        if (!act[0]->ps_batch) act[0]->ps_batch = new PsBatch();
        B = (PsBatch *)act[0]->ps_batch;
    }
    const bool mine = !B->busy.test_and_set(std::memory_order_acquire);
    char *mem = nullptr;
    cudaError_t e = cudaSuccess;
    if (mine) {
        if (B->bytes < bytes) {
            cudaFree(B->mem);
            B->mem = nullptr;
            B->bytes = 0;
            e = cudaMalloc(&B->mem, bytes);
            if (e == cudaSuccess) B->bytes = bytes;
        }
        mem = (char *)B->mem;
    } else {
        e = cudaMalloc((void **)&mem, bytes);
    }
    if (e != cudaSuccess) {
        cudaGetLastError();
        if (mine) B->busy.clear(std::memory_order_release);
        set_error("hz_zsolve_batched: workspace allocation failed");
        return HZ_ERR_ALLOC;
    }
    std::vector<PsSys> h(na);
    char *vec = mem + zero_b + sys_b;
    PsLine *lines = (PsLine *)(mem + info_b);
    PsSys *dsys = (PsSys *)(mem + zero_b);
    int cta = 0;
    for (int q = 0; q < na; ++q) {
        const int k = idx[q];
        PsSys &y = h[q];
        y = PsSys{};
        y.A = mat_view<double2>(act[q]);
        y.x = x[k];
        y.g0 = vec;
        y.g1 = vec + up((size_t)act[q]->n * 16);
        vec += 2 * up((size_t)act[q]->n * 16);
        y.ctl.tol = tol;
        y.ctl.maxit = maxit;
        y.ctl.b = b[k];
        y.ctl.x = x[k];
        y.ctl.op_scale = 1.0;
        y.info = (Info *)(mem + 256) + q;
        y.err = (int *)mem;
        y.lines = lines;
        lines += 2 * (size_t)ncta[k];
        y.cta0 = cta;
        y.ncta = ncta[k];
        y.batched = 1;
        cta += ncta[k];
    }
    std::vector<Info> hi(na);
    int err = 0;
    e = cudaMemsetAsync(mem, 0, zero_b, s);
    if (e == cudaSuccess) e = cudaMemcpyAsync(dsys, h.data(), sizeof(PsSys) * na, cudaMemcpyHostToDevice, s);
    if (e == cudaSuccess) {
        e = ps_launch(PS_BICG, act.data(), h.data(), na, dsys, s);
        if (ps_no_room(e)) {   // the caller's phases take the sweep
            cudaGetLastError();
            e = cudaSuccess;
            *taken = false;
        }
    }
    if (e == cudaSuccess) e = cudaMemcpyAsync(hi.data(), mem + 256, sizeof(Info) * na, cudaMemcpyDeviceToHost, s);
    if (e == cudaSuccess) e = cudaMemcpyAsync(&err, mem, sizeof(int), cudaMemcpyDeviceToHost, s);
    const cudaError_t e2 = cudaStreamSynchronize(s);   // (also after a failure: the workspace is free again)
    if (e == cudaSuccess) e = e2;
    if (mine) B->busy.clear(std::memory_order_release);
    else cudaFree(mem);
    if (e != cudaSuccess) return cuda_fail(e, "hz_zsolve_batched", __FILE__, __LINE__);
    if (!*taken) return HZ_OK;
    if (err) {
        set_error("hz_zsolve_batched: a barrier wait of the persistent solver expired");
        return HZ_ERR_TIMEOUT;
    }
    for (int q = 0; q < na; ++q) out[idx[q]] = hi[q];
    return HZ_OK;
}

}  // namespace hz
