// The FP64 Dslash half-pass at one output site on the integer pipe.
//
// This part of the chip multiplies FP64 at 2 per SM and clock but forms
// 32 x 32 + 64-bit integer products (IMAD.WIDE) at 64: 0.60 against 19.1 T/s
// measured.  The 288 FP64 FMAs of a site bound the FP64 half-pass at 2.6
// times its memory time, so the mat-vecs run in fixed point instead, three
// integer products for one FP64 product, 864 a site:
//
//   * A link's numbers lie in memory as two limbs each, u = h 2^-29 + l 2^-57,
//     with the bits that this cuts off beside them (fix_link.cuh).  A link
//     field takes this form only when every link is unitary to 1e-3 and finds
//     room for those bits (k_check_links); others keep doubles and the FP64
//     arithmetic.
//   * A neighbour's colour vector is cut to 57 bits below M = 2^(E - 1022), E the
//     largest FP64 exponent met so far at this site (all limbs of a component
//     carry its sign).  When a later neighbour raises E the sums move right.
//   * hh sums h h' and mm sums h l' + l h' in 64 bits; the l l' terms, below
//     2^-59 M, are left out.  Unit rows give |hh| < 8 sqrt(6) 2^58 < 2^63; |mm| < 48
//     2^56 + 20 2^57 < 2^63.
//   * The total hh + (mm >> 28), up to 62 bits, becomes a double once.
//
// These cuts are relative to M, the size of the site's largest neighbour
// component: a component of the sum is off by at most 20 (neighbours), 28
// (links), 12 (l l') and 2 (moved sums) times 2^-57 M, 3.9 2^-53 M, and one
// rounding.  48 FMAs in FP64 err by up to 48 2^-53 S, S = sum |U_ab| |v_b| over
// that component's own terms.  Where the links hardly mix the colours and
// these differ in scale, S is far below M for the small ones.  So a site's sum
// stands only where M <= 12 T, T a lower bound of S for every component: of six
// numbers of a link's row against six of a neighbour, in any order, the sum of
// products is at least m1 + c (m2 - m1), m1 and m2 the smallest and second
// smallest of the neighbour and c the row's spread; T sums that over the eight
// hops.  The error is then below 48 2^-53 S.  (A rebuilt row 2 errs by up to 3.5
// 2^-57 an entry here, by several 2^-53 in FP64.)  Other sites are recomputed in
// FP64 on the links' own numbers: up to four of a warp by eight lanes each, a hop
// a lane, 3 to 4 us a site; whole warps site by site, some 25 us.  Gaussian
// neighbours on links exp(i eps H) fail the test at below 3e-8 of the sites for eps
// >= 0.3, 8e-7 for 0.2 (with 9 for 12 at 3e-6 for 0.3), on unit links at 3e-4.
// Half-pass on 24^3x48 with unit links, FP64 pipe / this: Gaussian 165 / 79 us (8^4
// 20 / 13), but real numbers only, where every site is recomputed, 165 / 324 us.
//
// Sites whose largest neighbour component is not finite, 2^1017 or more, or
// below 2^-894 are recomputed too (zero vectors, as in a point source's field,
// are skipped there).
//
// Measured (GB300, half-pass, FP64 pipe / this): 32^3x64 18-real 492 / 203 us
// (6.46 TB/s, 0.95 of the measured copy rate), 24^3x48 18-real 168 / 65 us,
// 12-real 326 / 100 us (issue-bound: rebuilding row 2 is 576 more products a
// site), 8^4 20 / 6.2 us.  (Without the test and the bits beside the limbs: 199,
// 62 and 98 us.)  Error of D D chi on Gaussian fields against 64-bit sums: 3.4e-16 ->
// 1.8e-16 (norm), 3.1e-15 -> 1.5e-15 (largest component).
#pragma once

#include "fix_link.cuh"
#include "stg_internal.h"

namespace stg {

// R of the FP64 kernels: the reconstruction, with kFixLinks for limb links
constexpr int kFixLinks = 256;

struct FixLink {
    int h[3][3][2], l[3][3][2];  // [row][column][re, im]
    unsigned c;                  // spread of the rows (columns, for a backward hop), in eighths
};

// v, in units of 2^-58, to limbs in units of 2^-29 and 2^-57
__device__ __forceinline__ void fix_split(long long v, int &h, int &l)
{
    const long long x = (v + 1) >> 1;
    h = (int)((x + (1 << 27)) >> 28);
    l = (int)(x - ((long long)h << 28));
}

template <int N> struct FixDot {  // N products a b, to 2^-58
    long long hh = 0, mm = 0;
    __device__ __forceinline__ void add(int ah, int al, int bh, int bl)
    {
        hh += (long long)ah * bh;
        mm += (long long)ah * bl;
        mm += (long long)al * bh;
    }
};

// row 2 = s conj(r0 x r1) from the limbs of rows 0 and 1
__device__ __forceinline__ void fix_row2(FixLink &u, int s)
{
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        const int b = (a + 1) % 3, c = (a + 2) % 3;
#define STG_L(r_, k_, z_) u.h[r_][k_][z_], u.l[r_][k_][z_]
        FixDot<2> p, n;
        p.add(STG_L(0, b, 0), STG_L(1, c, 0));
        p.add(STG_L(0, c, 1), STG_L(1, b, 1));
        n.add(STG_L(0, b, 1), STG_L(1, c, 1));
        n.add(STG_L(0, c, 0), STG_L(1, b, 0));
        long long re = (p.hh - n.hh) + ((p.mm - n.mm) >> 28);
        FixDot<2> pi, ni;
        pi.add(STG_L(0, b, 0), STG_L(1, c, 1));
        pi.add(STG_L(0, b, 1), STG_L(1, c, 0));
        ni.add(STG_L(0, c, 0), STG_L(1, b, 1));
        ni.add(STG_L(0, c, 1), STG_L(1, b, 0));
#undef STG_L
        long long im = (ni.hh - pi.hh) + ((ni.mm - pi.mm) >> 28);
        if (s < 0) {
            re = -re;
            im = -im;
        }
        fix_split(re, u.h[2][a][0], u.l[2][a][0]);
        fix_split(im, u.h[2][a][1], u.l[2][a][1]);
    }
}

template <int RC, bool BACK>
__device__ __forceinline__ FixLink fix_link(const char *blk, int stride, int i, int s2)
{
    const uint4 *p = reinterpret_cast<const uint4 *>(blk) + i;
    FixLink u;
    constexpr int n = RC == 18 ? 9 : 6;
#pragma unroll
    for (int k = 0; k < n; ++k) {
        const uint4 a = ld_stream(p + (size_t)k * stride);
        u.h[k / 3][k % 3][0] = (int)a.x >> 1;
        u.l[k / 3][k % 3][0] = (int)a.y >> 4;
        u.h[k / 3][k % 3][1] = (int)a.z >> 1;
        u.l[k / 3][k % 3][1] = (int)a.w >> 4;
        if (k == 0) u.c = (BACK ? a.w : a.y) & 15u;
    }
    if (RC == 12) fix_row2(u, s2);
    return u;
}

struct FixAcc {
    long long hh[6], mm[6];  // re, im of colour 0, 1, 2
    int e;                   // FP64 exponent field of the scale
    unsigned t;              // T, in units of 2^-24 M
};

constexpr int kFixExpMin = 128, kFixExpMax = 2040;
constexpr int kFixShared = 4;       // sites of a warp recomputed by eight lanes each
constexpr unsigned kFixSpread = 12;  // the most that keeps 3.9 2^-53 M below 47.5 2^-53 S

__device__ __forceinline__ void fix_init(FixAcc &a)
{
#pragma unroll
    for (int k = 0; k < 6; ++k) a.hh[k] = a.mm[k] = 0;
    a.e = kFixExpMin;
    a.t = 0u;
}

// limbs of v below 2^(e - 1022): v = (h 2^28 + l) 2^(e - 1079), both with the
// sign of v (flipped with NEG); zero where v lies 57 or more bits below
template <bool NEG>
__device__ __forceinline__ void fix_cut(double v, int e, int &h, int &l)
{
    const unsigned hi = (unsigned)__double2hiint(v), lo = (unsigned)__double2loint(v);
    const unsigned wh = __funnelshift_l(lo, hi, 11) | 0x80000000u, wl = lo << 11;
    const unsigned long long w = ((unsigned long long)wh << 32) | wl;
    const int n = e - (int)((hi >> 20) & 0x7ffu) + 7;  // a subnormal (field 0) is shifted out
    unsigned long long x;
    asm("shr.u64 %0, %1, %2;" : "=l"(x) : "l"(w), "r"(n));
    const int m = NEG ? ~((int)hi >> 31) : (int)hi >> 31;
    const int xl = (int)(unsigned)x & 0xfffffff;
    const int xh = (int)__funnelshift_r((unsigned)x, (unsigned)(x >> 32), 28);
    h = (xh ^ m) - m;
    l = (xl ^ m) - m;
}

// the upper half of a double's size as a multiple of 2^-21 M, cut down (subnormals to 0)
__device__ __forceinline__ unsigned fix_size(unsigned hi, int e)
{
    return ((hi & 0xfffffu) | 0x100000u) >> min(e - (int)(hi >> 20), 31);
}

// acc += U v (forward) or acc -= U^dag v (ADJ); v in doubles
template <bool ADJ>
__device__ __forceinline__ void fix_hop(FixAcc &acc, const FixLink &u, const Vec3<double> &v)
{
    unsigned mx = 0u, m1 = ~0u, m2 = ~0u;  // the largest, smallest and second smallest
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        const unsigned a = (unsigned)__double2hiint(v.r[c]) & 0x7fffffffu;
        const unsigned b = (unsigned)__double2hiint(v.i[c]) & 0x7fffffffu;
        const unsigned lo = min(a, b), hi = max(a, b);
        mx = max(mx, hi);
        m2 = min(min(m2, hi), max(m1, lo));
        m1 = min(m1, lo);
    }
    const int e = (int)(mx >> 20);
    if (e > acc.e) {
        const int s = min(e - acc.e, 63);
#pragma unroll
        for (int k = 0; k < 6; ++k) {
            acc.hh[k] >>= s;
            acc.mm[k] >>= s;
        }
        acc.t >>= min(s, 31);
        acc.e = e;
    }
    const unsigned n1 = fix_size(m1, acc.e);
    acc.t += 8u * n1 + u.c * (fix_size(m2, acc.e) - n1);
    // ADJ: w = -v and its negated real parts; forward: v and its negated
    // imaginary parts
    int rh[3], rl[3], ih[3], il[3], nh[3], nl[3];
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        fix_cut<ADJ>(v.r[c], acc.e, rh[c], rl[c]);
        fix_cut<ADJ>(v.i[c], acc.e, ih[c], il[c]);
        nh[c] = ADJ ? -rh[c] : -ih[c];
        nl[c] = ADJ ? -rl[c] : -il[c];
    }
#pragma unroll
    for (int a = 0; a < 3; ++a)
#pragma unroll
        for (int b = 0; b < 3; ++b) {
            const int p = ADJ ? b : a, q = ADJ ? a : b;
            const int xh = u.h[p][q][0], xl = u.l[p][q][0], yh = u.h[p][q][1], yl = u.l[p][q][1];
            long long &hr = acc.hh[2 * a], &mr = acc.mm[2 * a];
            long long &hi = acc.hh[2 * a + 1], &mi = acc.mm[2 * a + 1];
            hr += (long long)xh * rh[b];
            mr += (long long)xh * rl[b];
            mr += (long long)xl * rh[b];
            hi += (long long)xh * ih[b];
            mi += (long long)xh * il[b];
            mi += (long long)xl * ih[b];
            // forward: re -= y i, im += y r; ADJ: re += y w_i, im -= y w_r
            const int ch = ADJ ? ih[b] : nh[b], cl = ADJ ? il[b] : nl[b];
            const int dh = ADJ ? nh[b] : rh[b], dl = ADJ ? nl[b] : rl[b];
            hr += (long long)yh * ch;
            mr += (long long)yh * cl;
            mr += (long long)yl * ch;
            hi += (long long)yh * dh;
            mi += (long long)yh * dl;
            mi += (long long)yl * dh;
        }
}

__device__ __forceinline__ bool fix_ok(int e, unsigned t)
{
    return e < kFixExpMax && e > kFixExpMin && t >= (1u << 24) / kFixSpread;
}

// (hh + (mm >> 28)) 2^(e - 1080), rounded to nearest (half away from zero) by
// integer operations: the conversion instruction runs on the FP64 pipe
__device__ __forceinline__ double fix_double(long long hh, long long mm, int e)
{
    const long long v = hh + (mm >> 28);
    const unsigned long long a = v < 0 ? 0ull - (unsigned long long)v : (unsigned long long)v;
    const int lz = __clzll((long long)a);
    const unsigned long long n = a << (lz & 63);  // leading one at bit 63
    const unsigned long long m = (n >> 11) + ((n >> 10) & 1ull);  // a carry raises the exponent below
    const unsigned long long r = m + ((unsigned long long)(unsigned)(e + 5 - lz) << 52);
    const unsigned hi = (unsigned)(r >> 32) | ((unsigned)(v >> 32) & 0x80000000u);
    return a ? __hiloint2double((int)hi, (int)(unsigned)r) : 0.0;
}

__device__ __forceinline__ Vec3<double> fix_value(const FixAcc &a)
{
    Vec3<double> v;
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        v.r[c] = fix_double(a.hh[2 * c], a.mm[2 * c], a.e);
        v.i[c] = fix_double(a.hh[2 * c + 1], a.mm[2 * c + 1], a.e);
    }
    return v;
}

// One hop's operands: the link record and the neighbour's vector, each by
// base, plane stride and index, and the sign of a 12-real link's row 2.
struct FixHop {
    const char *link;
    int lstride, li;
    const void *f;
    int fstride, fi;
    float s;
};

// One hop in FP64 (the recomputation): U v, or -U^dag v for a backward hop.
// Not inlined: it runs for exceptional sites only, and inlined its registers
// made every site's path spill.
template <int RC, bool NC>
__device__ __noinline__ Vec3<double> fix_hop_f64(const FixHop t, bool back)
{
    const Vec3<double> v = FieldIO<P64>::load<NC>(t.f, t.fstride, t.fi);
    Vec3<double> d;
#pragma unroll
    for (int c = 0; c < 3; ++c) d.r[c] = d.i[c] = 0.0;
    if (v.r[0] == 0.0 && v.i[0] == 0.0 && v.r[1] == 0.0 && v.i[1] == 0.0 && v.r[2] == 0.0 && v.i[2] == 0.0) return d;
    const uint4 *p = reinterpret_cast<const uint4 *>(t.link) + t.li;
    int2 w[RC];
    double n[RC];
#pragma unroll
    for (int k = 0; k < RC / 2; ++k) {
        const uint4 a = ld_stream(p + (size_t)k * t.lstride);
        w[2 * k] = make_int2((int)a.x, (int)a.y);
        w[2 * k + 1] = make_int2((int)a.z, (int)a.w);
    }
    fix_decode<RC>(w, n);
    Mat3<double> u;
#pragma unroll
    for (int k = 0; k < RC / 2; ++k) set_entry(u, k, n[2 * k], n[2 * k + 1]);
    if (RC == 12) reconstruct_row2(u, 1.0);
    const double s = RC == 12 ? (double)t.s : 1.0;
    if (back) adj_mul_sub(u, v, d, s);
    else mul_add<RC == 12>(u, v, d, s);
    return d;
}

// D chi at site i; hop(s, i, mu, back) gives the eight hops' operands.  U: the
// directions unrolled; all four, but two in the 12-real kernels of small
// lattices, whose code (64 KB unrolled) would come from L2 once per launch when
// two of them alternate: A on 8^4 30.2 -> 22.3 us.  Elsewhere two cost 4-8%.
template <int RC, bool NC = true, int U = 4, class H>
__device__ __forceinline__ Vec3<double> fix_site(const Geom &g, int parity, int i, const H &hop)
{
    const Site s = site_of(g, i, parity);
    FixAcc acc;
    fix_init(acc);
#pragma unroll U
    for (int mu = 0; mu < 4; ++mu) {
        {
            const FixHop t = hop(s, i, mu, false);
            const FixLink u = fix_link<RC, false>(t.link, t.lstride, t.li, t.s < 0.f ? -1 : 1);
            fix_hop<false>(acc, u, FieldIO<P64>::load<NC>(t.f, t.fstride, t.fi));
        }
        {
            const FixHop t = hop(s, i, mu, true);
            const FixLink u = fix_link<RC, true>(t.link, t.lstride, t.li, t.s < 0.f ? -1 : 1);
            fix_hop<true>(acc, u, FieldIO<P64>::load<NC>(t.f, t.fstride, t.fi));
        }
    }
    const bool ok = fix_ok(acc.e, acc.t);
    Vec3<double> d = fix_value(acc);
    const unsigned here = __activemask(), bad = __ballot_sync(here, !ok);
    if (bad == 0u) return d;
    // The recomputation: the hops' vectors each by itself, added in their order.
    if (here == 0xffffffffu && __popc(bad) <= kFixShared) {
        // few sites of a full warp: lane k takes hop k of one site after another
        const int k = (int)threadIdx.x & 7;
        for (unsigned m = bad; m != 0u; m &= m - 1u) {
            const int lane = __ffs((int)m) - 1, j = __shfl_sync(0xffffffffu, i, lane);
            const Vec3<double> h = fix_hop_f64<RC, NC>(hop(site_of(g, j, parity), j, k >> 1, k & 1), k & 1);
            Vec3<double> sum;
#pragma unroll
            for (int c = 0; c < 3; ++c) sum.r[c] = sum.i[c] = 0.0;
#pragma unroll 1
            for (int n = 0; n < 8; ++n)
#pragma unroll
                for (int c = 0; c < 3; ++c) {
                    sum.r[c] += __shfl_sync(0xffffffffu, h.r[c], n);
                    sum.i[c] += __shfl_sync(0xffffffffu, h.i[c], n);
                }
            if (((int)threadIdx.x & 31) == lane) d = sum;
        }
        return d;
    }
    if (ok) return d;
    // from the index alone (the empty asm): no neighbour address stays in a
    // register for this branch
    asm volatile("" : "+r"(i));
    const Site z = site_of(g, i, parity);
#pragma unroll
    for (int c = 0; c < 3; ++c) d.r[c] = d.i[c] = 0.0;
#pragma unroll 1
    for (int k = 0; k < 8; ++k) {
        const Vec3<double> h = fix_hop_f64<RC, NC>(hop(z, i, k >> 1, k & 1), k & 1);
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            d.r[c] += h.r[c];
            d.i[c] += h.i[c];
        }
    }
    return d;
}

}  // namespace stg
