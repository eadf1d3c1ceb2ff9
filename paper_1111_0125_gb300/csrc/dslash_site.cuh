// The Dslash half-pass (Eq. 5) at one output site, shared by the one-site-
// per-thread kernels (dslash.cu) and the multi-lattice group launch
// (group.cu): the four forward links at the site, the four backward links at
// the neighbours, the eight neighbour colour vectors, and for FX16 links the
// scale 1/32767 applied once to the sum.  FP64 links held as limbs (R has
// kFixLinks) take the integer form of fix64.cuh.
#pragma once

#include "fix64.cuh"

namespace stg {

// links and fields in floating point; NC: no thread of the kernel writes `in`
template <int P, int R, bool NC = true>
__device__ __forceinline__ Vec3<typename Real<P>::T> dslash_site_fp(const Geom &g, const Site &s,
                                                                    const char *const *lf,
                                                                    const char *const *lb, const void *in, int i)
{
    typedef typename Real<P>::T T;
    const int vh = g.Vh;
    Vec3<T> acc;
#pragma unroll
    for (int c = 0; c < 3; ++c) acc.r[c] = acc.i[c] = T(0);
#pragma unroll
    for (int mu = 0; mu < 4; ++mu) {
        int jf, jb;
        neighbours(g, s, i, mu, jf, jb);
        float sf = 1.f, sb = 1.f;
        if (R == 12) link_signs(g, s, mu, sf, sb);
        const T s2f = (R == 12) ? T(sf * LinkPost<P>::row2) : T(1);
        const T s2b = (R == 12) ? T(sb * LinkPost<P>::row2) : T(1);
        const Mat3<T> uf = LinkIO<P, R>::load(lf[mu], vh, i);
        const Vec3<T> vf = FieldIO<P>::template load<NC>(in, vh, jf);
        mul_add<R == 12>(uf, vf, acc, s2f);
        const Mat3<T> ub = LinkIO<P, R>::load(lb[mu], vh, jb);
        const Vec3<T> vb = FieldIO<P>::template load<NC>(in, vh, jb);
        adj_mul_sub(ub, vb, acc, s2b);
    }
    if (P == PX16) {
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            acc.r[c] *= T(LinkPost<PX16>::k);
            acc.i[c] *= T(LinkPost<PX16>::k);
        }
    }
    return acc;
}

template <int P, int R, bool NC = true, int U = 4>
__device__ __forceinline__ Vec3<typename Real<P>::T> dslash_site(const Geom &g, const char *const *lf,
                                                                 const char *const *lb, int parity,
                                                                 const void *in, int i)
{
    if constexpr (P == P64 && (R & kFixLinks) != 0) {
        constexpr int RC = R & ~kFixLinks;
        return fix_site<RC, NC, U>(g, parity, i, [&](const Site &s, int i, int mu, bool back) {
            int jf, jb;
            neighbours(g, s, i, mu, jf, jb);
            float sf = 1.f, sb = 1.f;
            if (RC == 12) link_signs(g, s, mu, sf, sb);
            return back ? FixHop{lb[mu], g.Vh, jb, in, g.Vh, jb, sb} : FixHop{lf[mu], g.Vh, i, in, g.Vh, jf, sf};
        });
    } else {
        return dslash_site_fp<P, R, NC>(g, site_of(g, i, parity), lf, lb, in, i);
    }
}

}  // namespace stg
