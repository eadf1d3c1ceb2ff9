// A whole CG solve (Fig. 1, or Fig. 2 with Eq. 6 and the updates of Sec. 3.2)
// of a small lattice inside one kernel, one thread-block cluster per system.
//
// An iteration of a small lattice is four kernels of 2 to 3 us whose work is
// a fraction of that; the launches, the grid totals and, between chunks, the
// host are the time.  Here the cluster's CTAs (up to 16) split the sites, the
// barriers between the phases are cluster barriers in hardware (no spinning,
// all CTAs resident by construction), and the sums travel through distributed
// shared memory: every CTA stores its partial into all CTAs' slots before a
// barrier and adds the same slots in the same order after it, so all CTAs
// take the same branches on the same bits.  The true residuals run in place.
// Several systems are several clusters, each at its own pace.
//
// Fields stay in global memory (L2): they are written and read by the CTAs of
// one cluster only, ordered by its barriers, so they are read with plain
// loads, never through the read-only path.
#pragma once

#include <type_traits>

#include "dslash_site.cuh"

namespace stg {

constexpr int kClThreads = 512;
constexpr int kClWarps = kClThreads / 32;
constexpr int kClMaxCtas = 16;
constexpr int kClMaxSystems = 64;
constexpr long long kClBudget = 4096;  // iterations per launch

enum ClStatus { CL_RUNNING = 0, CL_OK, CL_NOT_CONVERGED, CL_BREAKDOWN, CL_BAD_SOURCE, CL_BAD_START };

// one system's parameters and progress (device and pinned host)
struct ClSystem {
    double m2, tol2, trig2;
    long long iter_limit;
    double bb, rr, stop, delta_new, delta_old, rmax2;
    long long iter;
    int updates, breakdowns, status, resume;
};

struct ClArgs {
    Geom g;
    const char *lk[8];  // links of the inner precision, index parity * 4 + mu
    const char *hi[8];  // FP64 links
    const double2 *src; // canonical, Vh * 3 per system
    double2 *x;
    char *x64, *t64, *y, *r, *d, *q, *t;
    size_t f64, fr, fd; // bytes per system of the FP64 / PR / PD fields
    ClSystem *sys;
    int eq6;            // Eq. 6 start after an update and the running maximum of |r|
    int max_breakdowns;
    int write_x;        // store x when the system ends with OK or NOT_CONVERGED
    int lsm;            // k_cg_cluster_one: bytes of links in shared memory (0: read in place)
    FastDiv dper;       // division by the sites per CTA
};

__device__ __forceinline__ unsigned cl_rank()
{
    unsigned r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}

__device__ __forceinline__ unsigned cl_size()
{
    unsigned n;
    asm volatile("mov.u32 %0, %%cluster_nctarank;" : "=r"(n));
    return n;
}

// every thread of the cluster; orders global and shared memory among them
__device__ __forceinline__ void cl_barrier()
{
    asm volatile("barrier.cluster.arrive.release;" ::: "memory");
    asm volatile("barrier.cluster.wait.acquire;" ::: "memory");
}

struct ClShared {
    unsigned long long slot[2][kClMaxCtas];  // every CTA's partial, by rank
    unsigned long long warp[kClWarps];
    double scalar;
    int go;
};

template <bool PAIR> struct ClSum;
template <> struct ClSum<true> {
    typedef FF T;
    __device__ __forceinline__ static T zero() { return FF{0.f, 0.f}; }
    __device__ __forceinline__ static T add(T a, T b) { return ff_add(a, b); }
    __device__ __forceinline__ static unsigned long long bits(T a)
    {
        return ((unsigned long long)__float_as_uint(a.hi) << 32) | __float_as_uint(a.lo);
    }
    __device__ __forceinline__ static T of(unsigned long long b)
    {
        return FF{__uint_as_float((unsigned)(b >> 32)), __uint_as_float((unsigned)b)};
    }
};
template <> struct ClSum<false> {
    typedef double T;
    __device__ __forceinline__ static T zero() { return 0.0; }
    __device__ __forceinline__ static T add(T a, T b) { return a + b; }
    __device__ __forceinline__ static unsigned long long bits(T a) { return (unsigned long long)__double_as_longlong(a); }
    __device__ __forceinline__ static T of(unsigned long long b) { return __longlong_as_double((long long)b); }
};

// The cluster's total of v, in thread 0 of every CTA (the same bits in all),
// through a cluster barrier.  Calls alternate between two slot sets: a set is
// written again only after another barrier.
template <bool PAIR>
__device__ __forceinline__ typename ClSum<PAIR>::T cl_total(typename ClSum<PAIR>::T v, ClShared &sh, int &set)
{
    typedef ClSum<PAIR> S;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v = S::add(v, S::of(__shfl_down_sync(0xffffffffu, S::bits(v), o)));
    if (lane == 0) sh.warp[w] = S::bits(v);
    __syncthreads();
    const unsigned n = cl_size();
    if (w == 0) {
        v = lane < kClWarps ? S::of(sh.warp[lane]) : S::zero();
#pragma unroll
        for (int o = kClWarps / 2; o > 0; o >>= 1) v = S::add(v, S::of(__shfl_down_sync(0xffffffffu, S::bits(v), o)));
        const unsigned long long b = __shfl_sync(0xffffffffu, S::bits(v), 0);
        if (lane < (int)n) {
            unsigned to;
            asm volatile("mapa.shared::cluster.u32 %0, %1, %2;"
                         : "=r"(to) : "r"(smem_addr(&sh.slot[set][cl_rank()])), "r"(lane));
            asm volatile("st.shared::cluster.b64 [%0], %1;" :: "r"(to), "l"(b) : "memory");
        }
    }
    cl_barrier();
    if (w == 0) {
        v = lane < (int)n ? S::of(sh.slot[set][lane]) : S::zero();
#pragma unroll
        for (int o = kClMaxCtas / 2; o > 0; o >>= 1) v = S::add(v, S::of(__shfl_down_sync(0xffffffffu, S::bits(v), o)));
    }
    set ^= 1;
    return v;
}

// The scalars of the inner iterations, kept by thread 0 of every CTA: doubles
// for the plain FP64 iteration, FP32 numbers otherwise (see ff_div).
template <bool PLAIN> struct ClScalars;
template <> struct ClScalars<true> {
    typedef double S;
    typedef double T;
    double delta, delta_old, rmax2, stop, trig2, m2;
    __device__ __forceinline__ void start(const ClSystem &c)
    {
        delta = c.delta_new;
        delta_old = c.delta_old;
        rmax2 = c.rmax2;
        stop = c.stop;
        trig2 = c.trig2;
        m2 = c.m2;
    }
    __device__ __forceinline__ void save(ClSystem &c) const
    {
        c.delta_new = delta;
        c.delta_old = delta_old;
        c.rmax2 = rmax2;
    }
    __device__ __forceinline__ bool alpha(S pAp, T &a) const { return cg_alpha(delta, pAp, m2, a); }
    // after a step: beta, and why the inner iteration stops (iteration limit aside)
    __device__ __forceinline__ int step(S total, bool track, T &beta)
    {
        int f = FLAG_RUN;
        if (!isfinite(total)) f = FLAG_BREAKDOWN;
        else if (total <= stop) f = FLAG_CONVERGED;
        else if (trig2 > 0.0 && total < trig2 * rmax2) f = FLAG_UPDATE;
        beta = total / delta;
        delta_old = delta;
        delta = total;
        if (track && total > rmax2) rmax2 = total;
        return f;
    }
};
template <> struct ClScalars<false> {
    typedef FF S;
    typedef float T;
    F3 delta, delta_old, rmax2, stop, trig;
    double trig2;
    float m2;
    __device__ __forceinline__ void start(const ClSystem &c)
    {
        delta = f3_split(c.delta_new);
        delta_old = f3_split(c.delta_old);
        rmax2 = f3_split(c.rmax2);
        stop = f3_split(c.stop);
        trig2 = c.trig2;
        trig = f3_split(trig2 * c.rmax2);
        m2 = (float)c.m2;
    }
    __device__ __forceinline__ void save(ClSystem &c) const
    {
        c.delta_new = f3_double(delta);
        c.delta_old = f3_double(delta_old);
        c.rmax2 = f3_double(rmax2);
    }
    __device__ __forceinline__ bool alpha(S pAp, T &a) const { return ff_alpha(delta, pAp, m2, a); }
    __device__ __forceinline__ int step(S sum, bool track, T &beta)
    {
        const FF total = ff_norm(sum);
        const int f = f3_stop(total, stop, trig);
        beta = ff_div(total, FF{delta.hi, delta.mid});
        delta_old = delta;
        delta = F3{total.hi, total.lo, 0.f};
        if (track && f3_cmp(total, rmax2) > 0) {
            rmax2 = delta;
            trig = f3_split(trig2 * ((double)total.hi + (double)total.lo));
        }
        return f;
    }
};

// D of parity p in FP64 at site i (one copy for every kernel of the file)
template <int RH>
__device__ __noinline__ Vec3<double> hi_site(const ClArgs &a, int p, const void *in, int i)
{
    return dslash_site<P64, RH | kFixLinks, false>(a.g, a.hi + 4 * p, a.hi + 4 * (1 - p), p, in, i);
}

// PD / R: the inner iterations; RH: the reconstruction of the FP64 links
template <int PD, int R, int RH>
__global__ void __launch_bounds__(kClThreads, 1) k_cg_cluster(const __grid_constant__ ClArgs a)
{
    constexpr bool kPlain = PD == P64;
    constexpr int PR = kPlain ? P64 : P32;
    constexpr int RI = kPlain ? (R | kFixLinks) : R;
    typedef typename Real<PD>::T TD;
    typedef typename Real<PR>::T T;
    __shared__ ClShared sh;
    __shared__ ClSystem cs;  // thread 0 of every CTA keeps its own copy current
    __shared__ ClScalars<kPlain> sc;
    __shared__ typename ClScalars<kPlain>::T step;  // alpha, then beta
    int set = 0;
    const int k = blockIdx.x / cl_size();
    const int vh = a.g.Vh;
    const int per = (vh + (int)cl_size() - 1) / (int)cl_size();
    const int first = (int)cl_rank() * per, last = min(vh, first + per);
    char *const x64 = a.x64 + k * a.f64, *const t64 = a.t64 + k * a.f64;
    char *const y = kPlain ? x64 : a.y + k * a.fr;
    char *const r = a.r + k * a.fr;
    char *const d = a.d + k * a.fd, *const q = a.q + k * a.fd, *const t = a.t + k * a.fd;
    const double2 *const src = a.src + (size_t)k * vh * 3;
    if (threadIdx.x == 0) cs = a.sys[k];
    cl_barrier();  // every CTA runs before any stores into another's slots
    const double m2 = cs.m2;

    // r = b - A x64 (through t64), its FP64 norm in cs.rr
    const auto residual = [&] {
        for (int i = first + (int)threadIdx.x; i < last; i += kClThreads)
            FieldIO<P64>::store(t64, vh, i, hi_site<RH>(a, 1, x64, i));
        cl_barrier();
        double n = 0.0;
        for (int i = first + (int)threadIdx.x; i < last; i += kClThreads) {
            const Vec3<double> dt = hi_site<RH>(a, 0, t64, i);
            const Vec3<double> xv = FieldIO<P64>::load(x64, vh, i);
            Vec3<T> o;
#pragma unroll
            for (int c = 0; c < 3; ++c) {
                const double2 b = src[(size_t)i * 3 + c];
                const double re = b.x - m2 * xv.r[c] + dt.r[c], im = b.y - m2 * xv.i[c] + dt.i[c];
                n += re * re + im * im;
                o.r[c] = T(re);
                o.i[c] = T(im);
            }
            FieldIO<PR>::store(r, vh, i, o);
        }
        const double rr = cl_total<false>(n, sh, set);
        if (threadIdx.x == 0) cs.rr = rr;
    };
    // y = 0 (mixed), d = r + beta d
    const auto reset = [&](double beta) {
        for (int i = first + (int)threadIdx.x; i < last; i += kClThreads) {
            const Vec3<T> rv = FieldIO<PR>::load(r, vh, i);
            if (!kPlain) {
                Vec3<T> z;
#pragma unroll
                for (int c = 0; c < 3; ++c) z.r[c] = z.i[c] = T(0);
                FieldIO<PR>::store(y, vh, i, z);
            }
            Vec3<TD> o;
#pragma unroll
            for (int c = 0; c < 3; ++c) {
                o.r[c] = rv.r[c];
                o.i[c] = rv.i[c];
            }
            if (beta != 0.0) {
                const Vec3<TD> dv = FieldIO<PD>::load(d, vh, i);
#pragma unroll
                for (int c = 0; c < 3; ++c) {
                    o.r[c] = rv.r[c] + T(beta) * T(dv.r[c]);
                    o.i[c] = rv.i[c] + T(beta) * T(dv.i[c]);
                }
            }
            FieldIO<PD>::store(d, vh, i, o);
        }
        cl_barrier();
    };

    if (!cs.resume) {
        double n = 0.0;
        for (int i = first + (int)threadIdx.x; i < last; i += kClThreads) {
            Vec3<double> xv;
#pragma unroll
            for (int c = 0; c < 3; ++c) {
                const double2 v = a.x[((size_t)k * vh + i) * 3 + c], b = src[(size_t)i * 3 + c];
                xv.r[c] = v.x;
                xv.i[c] = v.y;
                n += b.x * b.x + b.y * b.y;
            }
            FieldIO<P64>::store(x64, vh, i, xv);
        }
        const double bb = cl_total<false>(n, sh, set);
        if (threadIdx.x == 0) {
            cs.bb = bb;
            cs.stop = cs.tol2 * bb;
            if (!isfinite(bb)) cs.status = CL_BAD_SOURCE;
        }
        __syncthreads();
        if (cs.status == CL_RUNNING) residual();
        __syncthreads();
        if (threadIdx.x == 0 && cs.status == CL_RUNNING) {
            if (cs.bb == 0.0) cs.status = CL_OK;  // x = 0, stored by the host
            else if (!isfinite(cs.rr)) cs.status = CL_BAD_START;
            else if (cs.rr <= cs.stop) cs.status = CL_OK;
            cs.delta_new = cs.delta_old = cs.rmax2 = cs.rr;
        }
        __syncthreads();
        if (cs.status == CL_RUNNING) reset(0.0);
    }

    if (threadIdx.x == 0) sc.start(cs);
    __syncthreads();
    const TD m2d = TD(m2);
    long long budget = kClBudget;
    while (cs.status == CL_RUNNING && budget > 0) {
        int flag = FLAG_RUN;
        while (flag == FLAG_RUN && budget > 0) {
            --budget;
            // t = D_oe d
            for (int i = first + (int)threadIdx.x; i < last; i += kClThreads)
                FieldIO<PD>::store(t, vh, i, dslash_site<PD, RI, false>(a.g, a.lk + 4, a.lk, 1, d, i));
            cl_barrier();
            // q = m^2 d - D_eo t, d^dag q
            typename ClSum<!kPlain>::T dq = ClSum<!kPlain>::zero();
            for (int i = first + (int)threadIdx.x; i < last; i += kClThreads) {
                const Vec3<TD> v = dslash_site<PD, RI, false>(a.g, a.lk, a.lk + 4, 0, t, i);
                const Vec3<TD> dv = FieldIO<PD>::load(d, vh, i);
                Vec3<TD> o;
#pragma unroll
                for (int c = 0; c < 3; ++c) {
                    o.r[c] = m2d * dv.r[c] - v.r[c];
                    o.i[c] = m2d * dv.i[c] - v.i[c];
                }
                const Vec3<TD> os = FieldIO<PD>::store(q, vh, i, o);
                TD n = TD(0);
#pragma unroll
                for (int c = 0; c < 3; ++c) n += dv.r[c] * os.r[c] + dv.i[c] * os.i[c];
                if constexpr (kPlain) dq += n;
                else dq = ff_add(dq, FF{float(n), 0.f});
            }
            const auto pAp = cl_total<!kPlain>(dq, sh, set);
            if (threadIdx.x == 0) sh.go = sc.alpha(pAp, step);
            __syncthreads();
            if (!sh.go) {
                flag = FLAG_BREAKDOWN;
                break;
            }
            // y += alpha d, r -= alpha q, |r|^2
            const T alpha = T(step);
            typename ClSum<!kPlain>::T nr = ClSum<!kPlain>::zero();
            for (int i = first + (int)threadIdx.x; i < last; i += kClThreads) {
                const Vec3<TD> dv = FieldIO<PD>::load(d, vh, i), qv = FieldIO<PD>::load(q, vh, i);
                Vec3<T> yv = FieldIO<PR>::load(y, vh, i), rv = FieldIO<PR>::load(r, vh, i);
#pragma unroll
                for (int c = 0; c < 3; ++c) {
                    yv.r[c] += alpha * T(dv.r[c]);
                    yv.i[c] += alpha * T(dv.i[c]);
                    rv.r[c] -= alpha * T(qv.r[c]);
                    rv.i[c] -= alpha * T(qv.i[c]);
                }
                FieldIO<PR>::store(y, vh, i, yv);
                const Vec3<T> rs = FieldIO<PR>::store(r, vh, i, rv);
                T n = T(0);
#pragma unroll
                for (int c = 0; c < 3; ++c) n += rs.r[c] * rs.r[c] + rs.i[c] * rs.i[c];
                if constexpr (kPlain) nr += n;
                else nr = ff_add(nr, FF{float(n), 0.f});
            }
            const auto total = cl_total<!kPlain>(nr, sh, set);
            if (threadIdx.x == 0) {
                cs.iter += 1;
                int f = sc.step(total, a.eq6, step);
                if (f == FLAG_RUN && cs.iter >= cs.iter_limit) f = FLAG_MAXITER;
                sh.go = f;
            }
            __syncthreads();
            flag = sh.go;
            if (flag != FLAG_RUN) break;
            // d = r + beta d
            const T beta = T(step);
            for (int i = first + (int)threadIdx.x; i < last; i += kClThreads) {
                const Vec3<T> rv = FieldIO<PR>::load(r, vh, i);
                const Vec3<TD> dv = FieldIO<PD>::load(d, vh, i);
                Vec3<TD> o;
#pragma unroll
                for (int c = 0; c < 3; ++c) {
                    o.r[c] = rv.r[c] + beta * T(dv.r[c]);
                    o.i[c] = rv.i[c] + beta * T(dv.i[c]);
                }
                FieldIO<PD>::store(d, vh, i, o);
            }
            cl_barrier();
        }
        if (flag == FLAG_RUN) break;  // the launch's iterations are used up
        // Sec. 3.2: x += y, r = b - A x
        if (!kPlain) {
            for (int i = first + (int)threadIdx.x; i < last; i += kClThreads) {
                Vec3<double> xv = FieldIO<P64>::load(x64, vh, i);
                const Vec3<T> yv = FieldIO<PR>::load(y, vh, i);
#pragma unroll
                for (int c = 0; c < 3; ++c) {
                    xv.r[c] += double(yv.r[c]);
                    xv.i[c] += double(yv.i[c]);
                }
                FieldIO<P64>::store(x64, vh, i, xv);
            }
        }
        cl_barrier();
        residual();
        if (threadIdx.x == 0) {
            double beta = 0.0;
            cs.updates += 1;
            if (cs.rr <= cs.stop) cs.status = CL_OK;
            else if (!isfinite(cs.rr)) cs.status = CL_BREAKDOWN;
            else if (cs.iter >= cs.iter_limit) cs.status = CL_NOT_CONVERGED;
            else if (flag == FLAG_BREAKDOWN) {
                if (++cs.breakdowns > a.max_breakdowns) cs.status = CL_BREAKDOWN;
            } else if (!kPlain && a.eq6) {
                sc.save(cs);
                beta = cs.rr / cs.delta_old;  // Eq. 6
            }
            sh.scalar = beta;
        }
        __syncthreads();
        if (cs.status != CL_RUNNING) break;
        reset(sh.scalar);
        if (threadIdx.x == 0) {
            cs.delta_new = cs.delta_old = cs.rmax2 = cs.rr;
            sc.start(cs);
        }
        __syncthreads();
    }
    if (a.write_x && (cs.status == CL_OK || cs.status == CL_NOT_CONVERGED) && cs.bb > 0.0)
        for (int i = first + (int)threadIdx.x; i < last; i += kClThreads) {
            const Vec3<double> xv = FieldIO<P64>::load(x64, vh, i);
#pragma unroll
            for (int c = 0; c < 3; ++c) a.x[((size_t)k * vh + i) * 3 + c] = make_double2(xv.r[c], xv.i[c]);
        }
    cl_barrier();  // no CTA leaves while another may still write its slots
    if (cl_rank() == 0 && threadIdx.x == 0) {
        sc.save(cs);
        cs.resume = 1;
        a.sys[k] = cs;
    }
}

// ---------------------------------------------------------------------------
// At most one site per thread (TPS = 1) or per four threads (TPS = 4, one
// direction each).  The inner iterations touch no global memory: y, r and d of
// the thread's site stay in registers, d and t lie in the CTAs' shared memory,
// where the neighbours read them through the cluster, and so do the links of
// both parities where they fit (`lsm` bytes a CTA; in place otherwise).
// Measured on 8^4, FP32/12: 6.2 us an iteration (0.9 us of it the nine true
// residuals' share), 13.5 us as four kernels; 7.4 us with d, t and the links in
// global memory, where the barriers wait for stores to reach L2.  FP32 matrices
// rebuilt once in shared memory instead of the links' records: 3% slower.
// ---------------------------------------------------------------------------
template <int TPS, typename T> __device__ __forceinline__ void sum_lanes(Vec3<T> &v)
{
#pragma unroll
    for (int o = 1; o < TPS; o <<= 1)
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            v.r[c] += __shfl_xor_sync(0xffffffffu, v.r[c], o);
            v.i[c] += __shfl_xor_sync(0xffffffffu, v.i[c], o);
        }
}

// v as a field of precision P holds it; 16-bit records go through slot i of
// `f`, the same record from every lane of the site
template <int P>
__device__ __forceinline__ Vec3<typename Real<P>::T> as_stored(void *f, int n, int i, const Vec3<typename Real<P>::T> &v)
{
    if constexpr (P == P32) return v;
    else return FieldIO<P>::store(f, n, i, v);
}

// the address of this CTA's shared-memory object in CTA `rank`
__device__ __forceinline__ const void *cl_map(const void *p, unsigned rank)
{
    const void *q;
    asm volatile("mapa.u64 %0, %1, %2;" : "=l"(q) : "l"(p), "r"(rank));
    return q;
}

// Hops of the thread's directions first_mu .. first_mu + NM - 1 in FP64 on
// limb links lk (index parity * 4 + mu): nb: the neighbours; bits of sg: the
// row-2 signs.  The 4 / NM lanes of a site decide together between integers and FP64.
template <int RC, int NM>
__device__ __forceinline__ Vec3<double> fix_part(const char *const *lk, int parity, int vh, int first_mu, const void *in,
                                                 int i, const int (&nb)[NM][2], unsigned sg)
{
    FixAcc acc;
    fix_init(acc);
#pragma unroll
    for (int m = 0; m < NM; ++m) {
        const int mu = first_mu + m;
        const int s0 = (sg >> (2 * m)) & 1u ? -1 : 1, s1 = (sg >> (2 * m + 1)) & 1u ? -1 : 1;
        const Vec3<double> vf = FieldIO<P64>::load(in, vh, nb[m][0]), vb = FieldIO<P64>::load(in, vh, nb[m][1]);
        fix_hop<false>(acc, fix_link<RC, false>(lk[parity * 4 + mu], vh, i, s0), vf);
        fix_hop<true>(acc, fix_link<RC, true>(lk[(1 - parity) * 4 + mu], vh, nb[m][1], s1), vb);
    }
    int e = acc.e;
#pragma unroll
    for (int o = 1; o < 4 / NM; o <<= 1) e = max(e, __shfl_xor_sync(0xffffffffu, e, o));
    unsigned t = acc.t >> min(e - acc.e, 31);
#pragma unroll
    for (int o = 1; o < 4 / NM; o <<= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
    if (fix_ok(e, t)) return fix_value(acc);
    Vec3<double> d;
#pragma unroll
    for (int c = 0; c < 3; ++c) d.r[c] = d.i[c] = 0.0;
#pragma unroll
    for (int m = 0; m < NM; ++m)
#pragma unroll
        for (int back = 0; back < 2; ++back) {
            const float s = (sg >> (2 * m + back)) & 1u ? -1.f : 1.f;
            const FixHop h = {lk[(back ? 1 - parity : parity) * 4 + first_mu + m], vh, back ? nb[m][1] : i,
                              in, vh, nb[m][back], s};
            const Vec3<double> v = fix_hop_f64<RC, false>(h, back);
#pragma unroll
            for (int c = 0; c < 3; ++c) {
                d.r[c] += v.r[c];
                d.i[c] += v.i[c];
            }
        }
    return d;
}

template <int PD, int R, int TPS>
__global__ void __launch_bounds__(kClThreads, 1) k_cg_cluster_one(const __grid_constant__ ClArgs a)
{
    constexpr int NM = 4 / TPS;
    extern __shared__ __align__(16) char lsm[];
    __shared__ ClShared sh;
    __shared__ ClSystem cs;
    __shared__ ClScalars<false> sc;
    __shared__ typename ClScalars<false>::T step;  // alpha, then beta
    int set = 0;
    const int k = blockIdx.x / cl_size();
    const int vh = a.g.Vh;
    const int per = (vh + (int)cl_size() - 1) / (int)cl_size();
    const int sub = (int)threadIdx.x % TPS, slot = (int)threadIdx.x / TPS;
    const int i = (int)cl_rank() * per + slot;
    const bool ok = slot < per && i < vh;  // other threads work on site 0 and store nothing
    const int j = ok ? i : 0, sj = ok ? slot : 0;
    const int mu0 = sub * NM;
    char *const x64 = a.x64 + k * a.f64, *const t64 = a.t64 + k * a.f64;
    char *const y = a.y + k * a.fr;
    char *const r = a.r + k * a.fr;
    char *const d = a.d + k * a.fd;
    // this CTA's d, t and (16-bit forms) q, one slot per site and one spare
    // slot for the threads without a site
    const int ns = per + 1;
    const int own = ok ? slot : per;
    const size_t fb = ((size_t)ns * field_site_bytes(PD) + 15) & ~(size_t)15;
    char *const ds = lsm + a.lsm, *const ts = ds + fb, *const qs = ts + fb;
    const double2 *const src = a.src + (size_t)k * vh * 3;
    if (threadIdx.x == 0) cs = a.sys[k];

    // neighbours and row-2 signs of the thread's directions, per output parity
    int nb[2][NM][2];
    unsigned sg[2] = {0u, 0u};
#pragma unroll
    for (int p = 0; p < 2; ++p) {
        const Site s = site_of(a.g, j, p);
#pragma unroll
        for (int mu = 0; mu < 4; ++mu) {
            int f, b;
            float sf, sb;
            neighbours(a.g, s, j, mu, f, b);
            link_signs(a.g, s, mu, sf, sb);
#pragma unroll
            for (int m = 0; m < NM; ++m)
                if (mu == mu0 + m) {
                    nb[p][m][0] = f;
                    nb[p][m][1] = b;
                    sg[p] |= (sf < 0.f ? 1u : 0u) << (2 * m) | (sb < 0.f ? 2u : 0u) << (2 * m);
                }
        }
    }
    // links to shared memory, record by record as they lie in their blocks
    const bool smem = a.lsm != 0;
    const size_t blk = ((size_t)per * link_bytes(PD, R) + 15) & ~(size_t)15;
    if (smem && ok) {
#pragma unroll 1
        for (int p = 0; p < 2; ++p)
#pragma unroll
            for (int m = 0; m < NM; ++m)
#pragma unroll
                for (int back = 0; back < 2; ++back) {
                    const char *from = a.lk[(back ? 1 - p : p) * 4 + mu0 + m];
                    const int n = back ? (p ? nb[1][m][1] : nb[0][m][1]) : j;
                    char *to = lsm + (size_t)(p * 8 + (mu0 + m) * 2 + back) * blk;
                    size_t of = 0, ot = 0;
                    constexpr int n16 = link_bytes(PD, R) / 16, rest = link_bytes(PD, R) % 16;
#pragma unroll
                    for (int e = 0; e < n16; ++e) {
                        *reinterpret_cast<uint4 *>(to + ot + (size_t)slot * 16) =
                            *reinterpret_cast<const uint4 *>(from + of + (size_t)n * 16);
                        of += (size_t)vh * 16;
                        ot += (size_t)per * 16;
                    }
                    if constexpr (rest == 8)
                        *reinterpret_cast<uint2 *>(to + ot + (size_t)slot * 8) =
                            *reinterpret_cast<const uint2 *>(from + of + (size_t)n * 8);
                    if constexpr (rest == 4)
                        *reinterpret_cast<unsigned *>(to + ot + (size_t)slot * 4) =
                            *reinterpret_cast<const unsigned *>(from + of + (size_t)n * 4);
                }
    }
    cl_barrier();  // every CTA runs before any stores into another's slots
    const double m2 = cs.m2;

    // D of parity p at this site from the CTAs' shared field `in`, in every
    // lane of the site
    const auto half = [&](auto parity, const char *in) {
        constexpr int p = decltype(parity)::value;
        Vec3<float> nf[NM][2], v;
#pragma unroll
        for (int m = 0; m < NM; ++m)
#pragma unroll
            for (int w = 0; w < 2; ++w) {
                const int n = nb[p][m][w], rank = (int)a.dper.div((unsigned)n);
                nf[m][w] = FieldIO<PD>::load(cl_map(in, (unsigned)rank), ns, n - rank * per);
            }
#pragma unroll
        for (int c = 0; c < 3; ++c) v.r[c] = v.i[c] = 0.f;
#pragma unroll
        for (int m = 0; m < NM; ++m) {
            const int mu = mu0 + m;
            const char *b = lsm + (size_t)(p * 8 + mu * 2) * blk;
            const float s0 = ((sg[p] >> (2 * m)) & 1u ? -1.f : 1.f) * LinkPost<PD>::row2;
            const float s1 = ((sg[p] >> (2 * m + 1)) & 1u ? -1.f : 1.f) * LinkPost<PD>::row2;
            const Mat3<float> uf = LinkIO<PD, R>::template load<true>(smem ? b : a.lk[p * 4 + mu],
                                                                      smem ? per : vh, smem ? sj : j);
            mul_add<R == 12>(uf, nf[m][0], v, R == 12 ? s0 : 1.f);
            const Mat3<float> ub = LinkIO<PD, R>::template load<true>(
                smem ? b + blk : a.lk[(1 - p) * 4 + mu], smem ? per : vh, smem ? sj : nb[p][m][1]);
            adj_mul_sub(ub, nf[m][1], v, R == 12 ? s1 : 1.f);
        }
        sum_lanes<TPS>(v);
        if (PD == PX16) {
#pragma unroll
            for (int c = 0; c < 3; ++c) {
                v.r[c] *= LinkPost<PX16>::k;
                v.i[c] *= LinkPost<PX16>::k;
            }
        }
        return v;
    };
    const auto half64 = [&](auto parity, const void *in) {
        constexpr int p = decltype(parity)::value;
        Vec3<double> v = fix_part<18, NM>(a.hi, p, vh, mu0, in, j, nb[p], sg[p]);
        sum_lanes<TPS>(v);
        return v;
    };
    typedef std::integral_constant<int, 0> Even;
    typedef std::integral_constant<int, 1> Odd;
    const bool mine = ok && sub == 0;
    Vec3<float> yv, rv;
    Vec3<float> dv;

    // r = b - A x64 (through t64); its FP64 norm in cs.rr
    const auto residual = [&] {
        {
            const Vec3<double> v = half64(Odd{}, x64);
            if (mine) FieldIO<P64>::store(t64, vh, i, v);
        }
        cl_barrier();
        const Vec3<double> dt = half64(Even{}, t64);
        const Vec3<double> xv = FieldIO<P64>::load(x64, vh, j);
        double n = 0.0;
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            const double2 b = src[(size_t)j * 3 + c];
            const double re = b.x - m2 * xv.r[c] + dt.r[c], im = b.y - m2 * xv.i[c] + dt.i[c];
            n += re * re + im * im;
            rv.r[c] = float(re);
            rv.i[c] = float(im);
        }
        const double rr = cl_total<false>(mine ? n : 0.0, sh, set);
        if (threadIdx.x == 0) cs.rr = rr;
    };
    // y = 0, d = r + beta d
    const auto reset = [&](double beta) {
        Vec3<float> o;
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            yv.r[c] = yv.i[c] = float(0);
            o.r[c] = rv.r[c];
            o.i[c] = rv.i[c];
            if (beta != 0.0) {
                o.r[c] = rv.r[c] + float(beta) * float(dv.r[c]);
                o.i[c] = rv.i[c] + float(beta) * float(dv.i[c]);
            }
        }
        dv = as_stored<PD>(ds, ns, own, o);
        if (mine && (PD == P32)) FieldIO<PD>::store(ds, ns, own, dv);
        cl_barrier();
    };

    if (!cs.resume) {
        double n = 0.0;
        Vec3<double> xv;
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            const double2 v = a.x[((size_t)k * vh + j) * 3 + c], b = src[(size_t)j * 3 + c];
            xv.r[c] = v.x;
            xv.i[c] = v.y;
            n += b.x * b.x + b.y * b.y;
        }
        if (mine) FieldIO<P64>::store(x64, vh, i, xv);
        const double bb = cl_total<false>(mine ? n : 0.0, sh, set);
        if (threadIdx.x == 0) {
            cs.bb = bb;
            cs.stop = cs.tol2 * bb;
            if (!isfinite(bb)) cs.status = CL_BAD_SOURCE;
        }
        __syncthreads();
        if (cs.status == CL_RUNNING) residual();
        __syncthreads();
        if (threadIdx.x == 0 && cs.status == CL_RUNNING) {
            if (cs.bb == 0.0) cs.status = CL_OK;  // x = 0, stored by the host
            else if (!isfinite(cs.rr)) cs.status = CL_BAD_START;
            else if (cs.rr <= cs.stop) cs.status = CL_OK;
            cs.delta_new = cs.delta_old = cs.rmax2 = cs.rr;
        }
        __syncthreads();
        if (cs.status == CL_RUNNING) reset(0.0);
    } else if (cs.status == CL_RUNNING) {
        yv = FieldIO<P32>::load(y, vh, j);
        rv = FieldIO<P32>::load(r, vh, j);
        dv = FieldIO<PD>::load(d, vh, j);
        if (mine) {
            if constexpr (PD == P32) FieldIO<PD>::store(ds, ns, own, dv);
            else reinterpret_cast<uint4 *>(ds)[own] = reinterpret_cast<const uint4 *>(d)[i];
        }
        cl_barrier();
    }

    if (threadIdx.x == 0) sc.start(cs);
    __syncthreads();
    const float m2d = float(m2);
    long long budget = kClBudget;
    while (cs.status == CL_RUNNING && budget > 0) {
        int flag = FLAG_RUN;
        while (flag == FLAG_RUN && budget > 0) {
            --budget;
            {  // t = D_oe d
                const Vec3<float> v = half(Odd{}, ds);
                if (mine) FieldIO<PD>::store(ts, ns, own, v);
            }
            cl_barrier();
            // q = m^2 d - D_eo t, d^dag q
            Vec3<float> qv = half(Even{}, ts);
#pragma unroll
            for (int c = 0; c < 3; ++c) {
                qv.r[c] = m2d * dv.r[c] - qv.r[c];
                qv.i[c] = m2d * dv.i[c] - qv.i[c];
            }
            qv = as_stored<PD>(qs, ns, own, qv);
            float n = float(0);
#pragma unroll
            for (int c = 0; c < 3; ++c) n += dv.r[c] * qv.r[c] + dv.i[c] * qv.i[c];
            if (!mine) n = float(0);
            const FF pAp = cl_total<true>(FF{float(n), 0.f}, sh, set);
            if (threadIdx.x == 0) sh.go = sc.alpha(pAp, step);
            __syncthreads();
            if (!sh.go) {
                flag = FLAG_BREAKDOWN;
                break;
            }
            // y += alpha d, r -= alpha q, |r|^2
            const float alpha = float(step);
            float w = float(0);
#pragma unroll
            for (int c = 0; c < 3; ++c) {
                yv.r[c] += alpha * float(dv.r[c]);
                yv.i[c] += alpha * float(dv.i[c]);
                rv.r[c] -= alpha * float(qv.r[c]);
                rv.i[c] -= alpha * float(qv.i[c]);
            }
#pragma unroll
            for (int c = 0; c < 3; ++c) w += rv.r[c] * rv.r[c] + rv.i[c] * rv.i[c];
            if (!mine) w = float(0);
            const FF total = cl_total<true>(FF{float(w), 0.f}, sh, set);
            if (threadIdx.x == 0) {
                cs.iter += 1;
                int f = sc.step(total, a.eq6, step);
                if (f == FLAG_RUN && cs.iter >= cs.iter_limit) f = FLAG_MAXITER;
                sh.go = f;
            }
            __syncthreads();
            flag = sh.go;
            if (flag != FLAG_RUN) break;
            // d = r + beta d
            const float beta = float(step);
#pragma unroll
            for (int c = 0; c < 3; ++c) {
                dv.r[c] = rv.r[c] + beta * float(dv.r[c]);
                dv.i[c] = rv.i[c] + beta * float(dv.i[c]);
            }
            dv = as_stored<PD>(ds, ns, own, dv);
            if (mine && (PD == P32)) FieldIO<PD>::store(ds, ns, own, dv);
            cl_barrier();
        }
        if (flag == FLAG_RUN) break;  // the launch's iterations are used up
        // Sec. 3.2: x += y, r = b - A x
        if (mine) {
            Vec3<double> xv = FieldIO<P64>::load(x64, vh, i);
#pragma unroll
            for (int c = 0; c < 3; ++c) {
                xv.r[c] += double(yv.r[c]);
                xv.i[c] += double(yv.i[c]);
            }
            FieldIO<P64>::store(x64, vh, i, xv);
        }
        cl_barrier();
        residual();
        if (threadIdx.x == 0) {
            double beta = 0.0;
            cs.updates += 1;
            if (cs.rr <= cs.stop) cs.status = CL_OK;
            else if (!isfinite(cs.rr)) cs.status = CL_BREAKDOWN;
            else if (cs.iter >= cs.iter_limit) cs.status = CL_NOT_CONVERGED;
            else if (flag == FLAG_BREAKDOWN) {
                if (++cs.breakdowns > a.max_breakdowns) cs.status = CL_BREAKDOWN;
            } else if (a.eq6) {
                sc.save(cs);
                beta = cs.rr / cs.delta_old;  // Eq. 6
            }
            sh.scalar = beta;
        }
        __syncthreads();
        if (cs.status != CL_RUNNING) break;
        reset(sh.scalar);
        if (threadIdx.x == 0) {
            cs.delta_new = cs.delta_old = cs.rmax2 = cs.rr;
            sc.start(cs);
        }
        __syncthreads();
    }
    if (cs.status == CL_RUNNING) {
        if (mine) {
            FieldIO<P32>::store(y, vh, i, yv);
            FieldIO<P32>::store(r, vh, i, rv);
            if constexpr (PD == P32) FieldIO<PD>::store(d, vh, i, dv);
            else reinterpret_cast<uint4 *>(d)[i] = reinterpret_cast<const uint4 *>(ds)[own];
        }
    } else if (mine && a.write_x && (cs.status == CL_OK || cs.status == CL_NOT_CONVERGED) && cs.bb > 0.0) {
        const Vec3<double> xv = FieldIO<P64>::load(x64, vh, i);
#pragma unroll
        for (int c = 0; c < 3; ++c) a.x[((size_t)k * vh + i) * 3 + c] = make_double2(xv.r[c], xv.i[c]);
    }
    cl_barrier();  // no CTA leaves while another may still write its slots
    if (cl_rank() == 0 && threadIdx.x == 0) {
        sc.save(cs);
        cs.resume = 1;
        a.sys[k] = cs;
    }
}

// ---------------------------------------------------------------------------
// launches
// ---------------------------------------------------------------------------
constexpr int kClSmem = 224 * 1024;  // dynamic shared memory at most

template <class K>
static bool cl_grant(K *kernel, int smem)
{
    if (cudaFuncSetAttribute(kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) == cudaSuccess)
        return !smem || grant_smem(kernel, smem);
    cudaGetLastError();
    return false;
}

// Whether the current device grants the kernel for `per` sites per CTA
// clusters of 16 and its shared memory.
template <int PD, int R>
static bool cl_granted(int per)
{
    constexpr int RH = PD == P64 ? R : 18;
    if constexpr (PD != P64) {
        if (per <= kClThreads / 4) return per_device([] { return cl_grant(k_cg_cluster_one<PD, R, 4>, kClSmem); });
        if (per <= kClThreads) return per_device([] { return cl_grant(k_cg_cluster_one<PD, R, 1>, kClSmem); });
    }
    return per_device([] { return cl_grant(k_cg_cluster<PD, R, RH>, 0); });
}

template <class K>
static cudaError_t cl_launch(K *kernel, const ClArgs &a, int nsys, int ctas, int smem, cudaStream_t s)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(nsys * ctas));
    cfg.blockDim = dim3(kClThreads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = (unsigned)ctas;
    at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kernel, a);
}

template <int PD, int R, int TPS>
static cudaError_t cl_launch_one(ClArgs a, int nsys, int ctas, cudaStream_t s)
{
    const int per = (a.g.Vh + ctas - 1) / ctas;
    const size_t links = 16 * (((size_t)per * link_bytes(PD, R) + 15) & ~(size_t)15);
    const size_t fields = (PD == P32 ? 2 : 3) *
                          (((size_t)(per + 1) * field_site_bytes(PD) + 15) & ~(size_t)15);
    a.lsm = links + fields <= (size_t)kClSmem ? (int)links : 0;
    a.dper = make_fastdiv((unsigned)per);
    return cl_launch(k_cg_cluster_one<PD, R, TPS>, a, nsys, ctas, a.lsm + (int)fields, s);
}

// the kernel for this lattice by the sites each CTA holds (cl_granted)
template <int PD, int R>
static cudaError_t cl_launch_pr(const ClArgs &a, int nsys, int ctas, cudaStream_t s)
{
    constexpr int RH = PD == P64 ? R : 18;
    const int per = (a.g.Vh + ctas - 1) / ctas;
    if constexpr (PD != P64) {  // (limb sums and y, r, d of a site do not fit the registers together)
        if (per <= kClThreads / 4) return cl_launch_one<PD, R, 4>(a, nsys, ctas, s);
        if (per <= kClThreads) return cl_launch_one<PD, R, 1>(a, nsys, ctas, s);
    }
    return cl_launch(k_cg_cluster<PD, R, RH>, a, nsys, ctas, 0, s);
}

// clusters of `ctas` CTAs that run at a time (every kernel here fills an SM's
// registers with one CTA)
template <int PD, int R>
static int cl_active(int ctas)
{
    const auto kernel = k_cg_cluster<PD, R, 18>;
    if (!cl_grant(kernel, 0)) return 0;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)ctas);
    cfg.blockDim = dim3(kClThreads);
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = (unsigned)ctas;
    at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    int n = 0;
    if (cudaOccupancyMaxActiveClusters(&n, kernel, &cfg) != cudaSuccess) {
        cudaGetLastError();
        return 0;
    }
    return n;
}

int cl_active_clusters(int ctas);  // on the current device
bool cl_granted_wide(int pd, int recon, int per);  // FP64, FP32
bool cl_granted_16(int pd, int recon, int per);
cudaError_t cl_dispatch_wide(int pd, int recon, const ClArgs &a, int nsys, int ctas, cudaStream_t s);  // FP64, FP32
cudaError_t cl_dispatch_16(int pd, int recon, const ClArgs &a, int nsys, int ctas, cudaStream_t s);

}  // namespace stg
