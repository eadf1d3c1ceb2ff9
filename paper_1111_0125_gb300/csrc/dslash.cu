// Staggered Dslash half-pass (Eq. 5) and its fused epilogues.
//
// One thread per output site of parity p.  Per site the kernel reads the
// four forward links U_mu(x) (parity p block, index i), the four backward
// links U_mu(x - mu) (parity 1-p block, at the neighbour's index), and the
// eight neighbour colour vectors of parity 1-p, then writes one colour
// vector.  Every link is read exactly once per half-pass; each neighbour
// vector is shared by eight sites and is served from L1/L2 after its first
// read, so the compulsory HBM traffic is 8 links + 1 input + 1 output per
// site.  The work is bandwidth-bound (0.36 flop/byte in FP64, 0.9 in
// FP32/12), so there are no tensor cores here: the 3x3 complex mat-vecs run
// in registers, on the FP32 pipe or, for FP64, on the integer pipe
// (fix64.cuh; 0.6 T FMA/s of FP64 would take 2.6 times the memory time).
//
// Reductions of FP64 data sum in FP64; those of FP32 / 16-bit data use the
// compensated FP32 pairs of grid_sum_ff (the FP64 pipe is ~1/64 of FP32 here).
//
// Epilogues (all fused into the second half-pass of A, Eq. 3):
//   EPI_NONE  out = D in
//   EPI_GATE  out = D in, skipped when the CG state flag is raised
//   EPI_A     out = m^2 w - D in                     (w = the even input d)
//   EPI_A_DOT as EPI_A, plus Re sum w^dag out in FP64 -> *dot
//   EPI_A_CG  as EPI_A inside CG, with block partials of Re sum w^dag out
//   EPI_RES   out = w - m^2 v + D in = b - A x, plus |out|^2 in FP64 -> *dot
#include "dslash_site.cuh"

namespace stg {

// Limb links (fix64.cuh): two blocks per SM, 128 registers.  Measured at
// 24^3x48, A with its dot, 18-real / 12-real: 145 / 208 us; three blocks (80
// registers, 150-550 bytes spilled) 146 / 224 us; one block (200 registers)
// 193 / 270 us.
//
// Other precisions have two forms with the same arithmetic: one with the
// registers that the compiler wants (118 / 204-218 for FP32/12 and /18, 72 to 96
// for 16 bits: two, one and three blocks per SM, the most loads in flight per
// thread), and a dense one (80 / 128 and 64: three, two and four blocks per SM,
// more loads in flight per SM and larger rounds of blocks).
constexpr int min_blocks(int p, int r, int bs, bool dense)
{
    const int blocks = p == P64 ? (r & kFixLinks ? 2 : 1) : dense ? (p != P32 ? 4 : r == 18 ? 2 : 3) : 1;
    return blocks * (kBlock / bs);
}

// Which form a lattice of `b` blocks of 256 sites takes: a lattice that fits
// one round of the first form is faster there, a larger one where its rounds
// over the 152 SMs are fewer, and FP32, FP16 and BF16 with 18-real links are
// faster in the dense form on nearly all of those.  Measured, A with its dot, us,
// first / dense form:
//   blocks    256         320         375         437         525         756         864         1080        1296        1792
//   FP32/18   14.9 / 13.6 21.4 / 16.6 25.2 / 20.0 28.3 / 23.6 35.0 / 28.3 43.9 / 37.8 48.4 / 42.2 59.0 / 51.4 70.7 / 61.3 91.4 / 81.7
//   FP32/12    9.8 / 13.6 14.2 / 14.4 16.4 / 15.0 18.4 / 16.1 21.3 / 22.7 30.9 / 28.8 33.0 / 31.2 40.4 / 39.4 48.1 / 44.7 61.0 / 60.0
//   FP16/18    9.4 /  9.6 13.3 / 14.9 14.4 / 15.2 16.4 / 15.5 17.5 / 15.3 26.4 / 24.0 28.3 / 26.4 33.8 / 29.8 40.6 / 36.3 51.5 / 46.1
//   BF16/18    9.6 /  9.9 13.9 / 15.6 14.9 / 15.7 16.7 / 16.1 17.8 / 15.7 26.8 / 24.9 28.8 / 27.3 34.2 / 30.2 41.5 / 36.9 52.5 / 46.7
//   FX16/18   12.3 / 10.2 13.0 / 16.0 13.2 / 15.5 13.7 / 16.3 17.5 / 16.3 25.0 / 25.9 26.7 / 28.2 35.5 / 31.0 38.2 / 38.0 50.4 / 48.0
//   FP16/12   12.4 / 10.1 12.8 / 15.4 12.8 / 15.6 12.9 / 15.8 16.8 / 16.2 19.9 / 21.3 23.8 / 22.6 28.2 / 27.6 32.6 / 31.6 41.9 / 40.6
//   BF16/12   12.9 / 10.2 13.3 / 16.0 13.4 / 16.2 13.6 / 16.6 17.5 / 17.0 20.8 / 22.5 24.4 / 23.6 29.1 / 29.0 33.5 / 33.1 43.1 / 42.4
// (links in L2 up to 437 blocks).  With the links from memory the dense form of
// FP16/12 at 256 blocks is the slower one, 13.7 against 13.3 us: not taken there.
static bool dense_pays(int p, int r, int b)
{
    constexpr int sms = 152;
    const auto fewer = [b](int dense, int first) {
        return (b + dense * sms - 1) / (dense * sms) < (b + first * sms - 1) / (first * sms);
    };
    if (p == P64) return false;
    if (p == P32) return r == 18 ? b >= 240 : b >= 350 && fewer(3, 2);
    if (r == 18 && p != PX16) return b >= 425;
    return r == 18 ? fewer(4, 3) : b >= 820;
}

// Threads per block.  Blocks of 128 put a small lattice on twice the SMs and
// even out the last wave of a large one; between, blocks of 256 leave fewer
// partials and share more neighbours in L1.  Measured (us, 256 against 128
// threads): A with its dot on Vh 2048: FP32/12 6.1 / 5.4, FP64/18 18.8 / 14.7;
// 10368: 6.1 / 5.5, 18.8 / 14.7; 20736: 6.5 / 6.5; 49152: 9.3 / 10.0; 65536 BF16/18
// 9.6 / 10.9; half-pass on 331776: FP32/12 20.5 / 20.0, FP32/18 30.5 / 29.4, BF16/18
// 17.6 / 16.7, FP64/18 63.9 / 62.7, but FP64/12 97.6 / 103.8.  Sums keep 256 on
// large lattices: one partial per 256 sites is what their scratch holds.
constexpr int kSmallBlock = 128;
constexpr int kSmallMax = 16384;  // ceil(Vh / 128) partials fit ceil(Vh / 256) + 64 up to here

int dslash_blocks(int vh, int epi, bool limbs12)
{
    const bool sums = epi == EPI_A_DOT || epi == EPI_A_CG || epi == EPI_RES;
    const bool fine = vh <= kSmallMax || (!sums && !limbs12 && vh >= 200000);
    const int bs = fine ? kSmallBlock : kBlock;
    return (vh + bs - 1) / bs;
}

template <typename T> __device__ __forceinline__ T pick_m2(double d, float f);
template <> __device__ __forceinline__ double pick_m2<double>(double d, float) { return d; }
template <> __device__ __forceinline__ float pick_m2<float>(double, float f) { return f; }

template <int P, int R, int EPI, int BS, bool DENSE>
__global__ void __launch_bounds__(BS, min_blocks(P, R, BS, DENSE)) k_dslash(const DslashArgs a)
{
    typedef typename Real<P>::T T;
    constexpr int kUnroll = P == P64 && R == (12 | kFixLinks) && BS == kSmallBlock ? 2 : 4;  // see fix_site
    pdl_wait();
    pdl_trigger();
    if (EPI == EPI_A_CG || EPI == EPI_GATE) {
        if (a.state->flag != FLAG_RUN) return;  // uniform over the grid
        if (EPI == EPI_GATE && blockIdx.x == 0 && threadIdx.x == 0) cg_commit(a.state);
    }
    const int i = blockIdx.x * BS + threadIdx.x;
    const int vh = a.g.Vh;
    T dot = T(0);
    if (i < vh) {
        const Vec3<T> acc = dslash_site<P, R, true, kUnroll>(a.g, a.lf, a.lb, a.parity, a.in, i);
        if (EPI == EPI_NONE || EPI == EPI_GATE) {
            FieldIO<P>::store(a.out, vh, i, acc);
        } else if (EPI == EPI_RES) {
            const Vec3<T> b = FieldIO<P>::load_nc(a.w, vh, i);
            const Vec3<T> x = FieldIO<P>::load_nc(a.v, vh, i);
            const T m2 = pick_m2<T>(a.m2, a.m2f);
            Vec3<T> o;
#pragma unroll
            for (int c = 0; c < 3; ++c) {
                o.r[c] = b.r[c] - m2 * x.r[c] + acc.r[c];
                o.i[c] = b.i[c] - m2 * x.i[c] + acc.i[c];
            }
            const Vec3<T> os = FieldIO<P>::store(a.out, vh, i, o);
#pragma unroll
            for (int c = 0; c < 3; ++c) dot += os.r[c] * os.r[c] + os.i[c] * os.i[c];
        } else {
            const T m2 = (EPI == EPI_A_CG) ? pick_m2<T>(a.state->m2, a.state->m2f) : pick_m2<T>(a.m2, a.m2f);
            const Vec3<T> d = FieldIO<P>::load_nc(a.w, vh, i);
            Vec3<T> o;
#pragma unroll
            for (int c = 0; c < 3; ++c) {
                o.r[c] = m2 * d.r[c] - acc.r[c];
                o.i[c] = m2 * d.i[c] - acc.i[c];
            }
            // d^dag q with q as stored, i.e. as the CG update will read it
            const Vec3<T> os = FieldIO<P>::store(a.out, vh, i, o);
#pragma unroll
            for (int c = 0; c < 3; ++c) dot += d.r[c] * os.r[c] + d.i[c] * os.i[c];
        }
    }
    if constexpr (EPI == EPI_A_CG) {
        if constexpr (P == P64) publish_partial<BS>(double(dot), a.state, a.partials);
        else publish_partial<BS>(FF{float(dot), 0.f}, a.state, a.partials);
    } else if constexpr (EPI == EPI_A_DOT || EPI == EPI_RES) {
        double total;
        bool last;
        if constexpr (P == P64) last = grid_sum<BS>(double(dot), a.partials, a.counter, total);
        else last = grid_sum_ff<BS>(FF{float(dot), 0.f}, reinterpret_cast<float2 *>(a.partials), a.counter, total);
        if (last) *a.dot = total;
    }
}

template <int P, int R, int EPI>
static void launch_bs(const DslashArgs &a, cudaStream_t s, bool pdl)
{
    const int vh = a.g.Vh, grid = dslash_blocks(vh, EPI, P == P64 && R == (12 | kFixLinks));
    const bool coarse = grid == (vh + kBlock - 1) / kBlock;
    if (dense_pays(P, R, (vh + kBlock - 1) / kBlock)) {
        if (coarse) launch_k(k_dslash<P, R, EPI, kBlock, P != P64>, grid, kBlock, 0, s, pdl, a);
        else launch_k(k_dslash<P, R, EPI, kSmallBlock, P != P64>, grid, kSmallBlock, 0, s, pdl, a);
    } else {
        if (coarse) launch_k(k_dslash<P, R, EPI, kBlock, false>, grid, kBlock, 0, s, pdl, a);
        else launch_k(k_dslash<P, R, EPI, kSmallBlock, false>, grid, kSmallBlock, 0, s, pdl, a);
    }
}

template <int P, int R>
static void launch_pr(int epi, const DslashArgs &a, cudaStream_t s, bool pdl)
{
    switch (epi) {
    case EPI_NONE: launch_bs<P, R, EPI_NONE>(a, s, pdl); break;
    case EPI_A: launch_bs<P, R, EPI_A>(a, s, pdl); break;
    case EPI_A_DOT: launch_bs<P, R, EPI_A_DOT>(a, s, pdl); break;
    case EPI_A_CG: launch_bs<P, R, EPI_A_CG>(a, s, pdl); break;
    case EPI_RES: launch_bs<P, R, EPI_RES>(a, s, pdl); break;
    case EPI_GATE: launch_bs<P, R, EPI_GATE>(a, s, pdl); break;
    }
}

stg_status launch_dslash(const Geom &g, int prec, int epi, const DslashLaunch &L, cudaStream_t s)
{
    DslashArgs a;
    a.g = g;
    a.parity = L.out_parity;
    for (int mu = 0; mu < 4; ++mu) {
        a.lf[mu] = L.links->blk(L.out_parity, mu);
        a.lb[mu] = L.links->blk(1 - L.out_parity, mu);
    }
    a.lt = L.links->tiled ? L.links->tiled + (size_t)L.out_parity * L.links->tiled_parity_bytes : nullptr;
    a.grid_cap = L.links->fx_grid_cap;
    a.drop_fill = L.links->fx_drop_fill;
    a.in = L.in;
    a.out = L.out;
    a.w = L.w;
    a.v = L.v;
    a.m2 = L.m2;
    a.m2f = (float)L.m2;
    a.dot = L.dot;
    a.state = L.state;
    a.partials = L.partials;
    a.counter = L.counter;
    const int recon = L.links->recon;
    if (prec != L.links->prec) {
        set_error("dslash: link precision does not match the field precision");
        return STG_ERR_UNSUPPORTED;
    }
    if ((prec == PX16 || prec == P16) && launch_dslash_16(prec, recon, epi, a, s, L.pdl)) {
        STG_CUDA(cudaGetLastError());
        return STG_OK;
    }
    if (prec == P64 && L.links->fix) {  // links as limbs: the integer form
        if (recon == 18) launch_pr<P64, 18 | kFixLinks>(epi, a, s, L.pdl);
        else launch_pr<P64, 12 | kFixLinks>(epi, a, s, L.pdl);
    } else if (prec == P64) {
        if (recon == 18) launch_pr<P64, 18>(epi, a, s, L.pdl);
        else launch_pr<P64, 12>(epi, a, s, L.pdl);
    } else if (prec == P32) {
        if (recon == 18) launch_pr<P32, 18>(epi, a, s, L.pdl);
        else launch_pr<P32, 12>(epi, a, s, L.pdl);
    } else {
        if (prec == PB16) {
            if (recon == 18) launch_pr<PB16, 18>(epi, a, s, L.pdl);
            else launch_pr<PB16, 12>(epi, a, s, L.pdl);
        } else if (prec == PX16) {
            if (recon == 18) launch_pr<PX16, 18>(epi, a, s, L.pdl);
            else launch_pr<PX16, 12>(epi, a, s, L.pdl);
        } else if (recon == 18) {
            launch_pr<P16, 18>(epi, a, s, L.pdl);
        } else {
            launch_pr<P16, 12>(epi, a, s, L.pdl);
        }
    }
    STG_CUDA(cudaGetLastError());
    return STG_OK;
}

}  // namespace stg
