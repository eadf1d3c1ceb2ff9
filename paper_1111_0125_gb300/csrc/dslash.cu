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
#include <atomic>

#include "dslash_site.cuh"

namespace stg {

// Limb links (fix64.cuh): two blocks per SM, 128 registers.  Measured at
// 24^3x48, A with its dot, 18-real / 12-real: 148 / 214 us; before the limbs carried
// all bits of a link 145 / 208 us, against 146 / 224 us with three blocks (80
// registers, 150-550 bytes spilled) and 193 / 270 us with one (200 registers).
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

// Which of these a lattice of `b` blocks of 256 sites takes: a lattice that fits
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

// A third form starts the copy of its eight links to shared memory before it
// waits for the previous kernel, so the links' latency overlaps that kernel's
// end and no link load waits for registers.  It pays where its blocks (shared
// memory for two per SM of FP32/12, one of FP32/18, four of 16 bits with 12
// reals, three with 18) make one round.  Measured, us, other form / this one:
//   blocks            128           256           304           375           437           531
//   A      FP32/12     8.7 /  7.7   12.0 /  9.9   12.2 / 13.0   15.8 / 19.4   16.3 / 21.7
//   A      FP32/18    10.0 /  7.5   14.7 / 16.0   15.1 / 18.7
//   A      FP16/12     6.5 /  6.6   12.3 /  9.0   12.6 /  9.4   12.8 / 13.5   12.9 / 14.1
//   A      FP16/18     8.1 /  7.2   10.7 / 10.0   11.2 / 10.7   16.0 / 12.7   16.2 / 14.4   17.2 / 18.9
//   A pass BF16/18     2.3 /  2.1    4.8 /  3.9    5.2 /  4.1    7.5 /  4.4    7.2 /  6.1    7.8 /  9.2
//   A pass FX16/18     2.4 /  2.2    5.8 /  4.1    6.0 /  4.2    6.2 /  4.5    6.7 /  6.3    8.0 /  9.5
// FP32/12 at 272 blocks: 12.2 / 11.1, at 288: 12.0 / 12.3.
static bool ahead_pays(int p, int r, int b)
{
    if (p == P32) return b <= (r == 18 ? 152 : 280);
    return b <= (r == 18 ? 3 : 2) * 152;
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

constexpr int kFirst = 0, kDense = 1, kAhead = 2;

// The ahead form: every thread copies its site's eight links to its own slots
// of shared memory, one link field of BS sites (the planes of LinkIO) for each
// direction, forward then backward, and one commit group per direction.
constexpr int ahead_bytes(int p, int r, int bs) { return 8 * link_bytes(p, r) * bs; }

template <int N> __device__ __forceinline__ void cp_async(unsigned dst, const char *src)
{
    if constexpr (N == 16) asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" :: "r"(dst), "l"(src) : "memory");
    else asm volatile("cp.async.ca.shared.global [%0], [%1], %2;" :: "r"(dst), "l"(src), "n"(N) : "memory");
}

template <int N> __device__ __forceinline__ void cp_wait() { asm volatile("cp.async.wait_group %0;" :: "n"(N) : "memory"); }

// site s of a link field of vh sites to slot t of one of BS sites
template <int B, int BS>
__device__ __forceinline__ void cp_link(const char *dst, int t, const char *src, size_t vh, int s)
{
    constexpr int n = B / 16, rest = B % 16;
    const unsigned d = smem_addr(dst);
#pragma unroll
    for (int q = 0; q < n; ++q) cp_async<16>(d + (q * BS + t) * 16, src + (q * vh + s) * 16);
    if constexpr (rest != 0) cp_async<rest>(d + n * BS * 16 + t * rest, src + n * vh * 16 + (size_t)s * rest);
}

template <int P, int R, int BS>
__device__ __forceinline__ void ahead_issue(const DslashArgs &a, const char *links, const Site &s, int i)
{
    constexpr int B = link_bytes(P, R);
#pragma unroll
    for (int mu = 0; mu < 4; ++mu) {
        int jf, jb;
        neighbours(a.g, s, i, mu, jf, jb);
        cp_link<B, BS>(links + 2 * mu * B * BS, threadIdx.x, a.lf[mu], a.g.Vh, i);
        cp_link<B, BS>(links + (2 * mu + 1) * B * BS, threadIdx.x, a.lb[mu], a.g.Vh, jb);
        asm volatile("cp.async.commit_group;" ::: "memory");
    }
}

// dslash_site_fp with the links taken from the thread's slots
template <int P, int R, int BS>
__device__ __forceinline__ Vec3<float> ahead_site(const DslashArgs &a, const char *links, const Site &s, int i)
{
    constexpr int B = link_bytes(P, R);
    Vec3<float> acc;
#pragma unroll
    for (int c = 0; c < 3; ++c) acc.r[c] = acc.i[c] = 0.f;
#pragma unroll
    for (int mu = 0; mu < 4; ++mu) {
        int jf, jb;
        neighbours(a.g, s, i, mu, jf, jb);
        float sf = 1.f, sb = 1.f;
        if (R == 12) link_signs(a.g, s, mu, sf, sb);
        const float s2f = R == 12 ? sf * LinkPost<P>::row2 : 1.f, s2b = R == 12 ? sb * LinkPost<P>::row2 : 1.f;
        const Vec3<float> vf = FieldIO<P>::load_nc(a.in, a.g.Vh, jf), vb = FieldIO<P>::load_nc(a.in, a.g.Vh, jb);
        if (mu == 0) cp_wait<3>();
        else if (mu == 1) cp_wait<2>();
        else if (mu == 2) cp_wait<1>();
        else cp_wait<0>();
        mul_add<R == 12>(LinkIO<P, R>::template load<true>(links + 2 * mu * B * BS, BS, threadIdx.x), vf, acc, s2f);
        adj_mul_sub(LinkIO<P, R>::template load<true>(links + (2 * mu + 1) * B * BS, BS, threadIdx.x), vb, acc, s2b);
    }
    if (P == PX16) {
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            acc.r[c] *= LinkPost<PX16>::k;
            acc.i[c] *= LinkPost<PX16>::k;
        }
    }
    return acc;
}

template <int P, int R, int EPI, int BS, int FORM>
__global__ void __launch_bounds__(BS, min_blocks(P, R, BS, FORM == kDense)) k_dslash(const DslashArgs a)
{
    typedef typename Real<P>::T T;
    constexpr int kUnroll = P == P64 && R == (12 | kFixLinks) && BS == kSmallBlock ? 2 : 4;  // see fix_site
    constexpr bool kReadsW = EPI != EPI_NONE && EPI != EPI_GATE;
    extern __shared__ __align__(16) char links_ahead[];
    const int i = blockIdx.x * BS + threadIdx.x;
    const int vh = a.g.Vh;
    Site site = {};
    bool issued = false;
    if constexpr (FORM == kAhead) {
        if (i < vh) site = site_of(a.g, i, a.parity);
        // links are constant, so their copies may overlap the previous kernel.
        // The flag's writer may be that kernel: this read only decides whether
        // to copy early, the check after the wait whether to go on.
        issued = i < vh && ((EPI != EPI_A_CG && EPI != EPI_GATE) || *(volatile const int *)&a.state->flag == FLAG_RUN);
        if (issued) ahead_issue<P, R, BS>(a, links_ahead, site, i);
    }
    pdl_wait();
    pdl_trigger();
    if (EPI == EPI_A_CG || EPI == EPI_GATE) {
        if (a.state->flag != FLAG_RUN) {  // uniform over the grid
            if (FORM == kAhead) cp_wait<0>();
            return;
        }
        if (EPI == EPI_GATE && blockIdx.x == 0 && threadIdx.x == 0) cg_commit(a.state);
    }
    T dot = T(0);
    if (i < vh) {
        Vec3<T> acc, w = {};
        // the ahead form's waits keep later loads behind them
        if (FORM == kAhead && kReadsW) w = FieldIO<P>::load_nc(a.w, vh, i);
        if constexpr (FORM == kAhead) {
            if (!issued) ahead_issue<P, R, BS>(a, links_ahead, site, i);
            acc = ahead_site<P, R, BS>(a, links_ahead, site, i);
        } else {
            acc = dslash_site<P, R, true, kUnroll>(a.g, a.lf, a.lb, a.parity, a.in, i);
        }
        if (EPI == EPI_NONE || EPI == EPI_GATE) {
            FieldIO<P>::store(a.out, vh, i, acc);
        } else if (EPI == EPI_RES) {
            const Vec3<T> b = FORM == kAhead ? w : FieldIO<P>::load_nc(a.w, vh, i);
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
            const Vec3<T> d = FORM == kAhead ? w : FieldIO<P>::load_nc(a.w, vh, i);
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

// The ahead form's shared memory is above the default limit and is granted per
// device; false if it is refused (the other forms need none).  One carve-out
// for all its instantiations: two that differ change the SMs' split between
// consecutive kernels, 4 us more per A of FP16/12 on 16^4.
template <int P, int R, int EPI, int BS>
static bool ahead_granted()
{
    static std::atomic<unsigned long long> granted{0};
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev > 63) return false;
    if (granted.load(std::memory_order_relaxed) >> dev & 1) return true;
    const auto k = k_dslash<P, R, EPI, BS, kAhead>;
    if (cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, ahead_bytes(P, R, BS)) != cudaSuccess ||
        cudaFuncSetAttribute(k, cudaFuncAttributePreferredSharedMemoryCarveout, cudaSharedmemCarveoutMaxShared) !=
            cudaSuccess) {
        cudaGetLastError();
        return false;
    }
    granted.fetch_or(1ull << dev, std::memory_order_relaxed);
    return true;
}

template <int P, int R, int EPI, int BS>
static void launch_form(const DslashArgs &a, int grid, cudaStream_t s, bool pdl)
{
    const int blocks = (a.g.Vh + kBlock - 1) / kBlock;
    if constexpr (P != P64) {
        if (ahead_pays(P, R, blocks) && ahead_granted<P, R, EPI, BS>()) {
            launch_k(k_dslash<P, R, EPI, BS, kAhead>, grid, BS, ahead_bytes(P, R, BS), s, pdl, a);
            return;
        }
    }
    if (dense_pays(P, R, blocks)) launch_k(k_dslash<P, R, EPI, BS, P == P64 ? kFirst : kDense>, grid, BS, 0, s, pdl, a);
    else launch_k(k_dslash<P, R, EPI, BS, kFirst>, grid, BS, 0, s, pdl, a);
}

template <int P, int R, int EPI>
static void launch_bs(const DslashArgs &a, cudaStream_t s, bool pdl)
{
    const int vh = a.g.Vh, grid = dslash_blocks(vh, EPI, P == P64 && R == (12 | kFixLinks));
    if (grid == (vh + kBlock - 1) / kBlock) launch_form<P, R, EPI, kBlock>(a, grid, s, pdl);
    else launch_form<P, R, EPI, kSmallBlock>(a, grid, s, pdl);
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
            launch_pr<PX16, 18>(epi, a, s, L.pdl);  // 12-real: launch_dslash_16
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
