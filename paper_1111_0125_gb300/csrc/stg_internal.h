// Host-side structures shared by the library's translation units.
#pragma once

#include <cuda_runtime.h>

#include <string>
#include <utility>

#include "stg.h"
#include "per_device.h"
#include "stg_common.cuh"

namespace stg {

constexpr int kBlock = 256;  // threads per block of every site-parallel kernel

// Launch with programmatic dependent launch when `pdl`: the kernel may start
// while its predecessor on the stream finishes; it must call pdl_wait()
// before touching anything the predecessor writes (stg_common.cuh).
template <typename... K, typename... A>
static inline cudaError_t launch_k(void (*kernel)(K...), dim3 grid, dim3 block, size_t smem, cudaStream_t s,
                                   bool pdl, A &&...args)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = pdl ? at : nullptr;
    cfg.numAttrs = pdl ? 1 : 0;
    return cudaLaunchKernelEx(&cfg, kernel, std::forward<A>(args)...);
}

// Device copy of the links in one precision / reconstruction.
// Tile-major copy of FX16 or FP16 / 12-real links for the staged Dslash: for output
// parity p, tile k of kFxTile consecutive output sites and direction mu, one
// contiguous block of kFxStageBytes holds the forward links U_mu(x) (uint4
// [kFxTile] then uint2 [kFxTile]) followed by the backward links U_mu(x - mu)
// of the same output sites, each record at the output site's slot; slots past
// Vh are zero.  Every link appears twice (once per parity of output site).
constexpr int kFxTile = 1024;
constexpr unsigned kFxStageBytes = kFxTile * 48u;

// Tile-major copy of FP32 / 12-real and FX16 / 12-real links for the staged
// multi-system Dslash: for output parity p and tile k of kMTile consecutive
// output sites, one contiguous block of kMTile * 8 * L bytes holds, for mu =
// 0..3 and dir = forward, backward, the 12-real records of the tile's sites
// as planes (FP32: three float4 planes; FX16: a uint4 plane then a uint2
// plane); slots past Vh are zero.
constexpr int kMTile = 64;

struct LinkField {
    char *base = nullptr;   // 8 blocks: (parity, mu) -> base + (2 * 4 ... ) see blk()
    int prec = -1;
    int recon = 18;
    bool fix = false;       // FP64: entries held as limbs (fix64.cuh) instead of doubles
    size_t blk_bytes = 0;   // bytes of one (parity, mu) block, 256-aligned
    char *tiled = nullptr;  // FX16 / 12-real only: tile-major copy (kFxTile)
    size_t tiled_parity_bytes = 0;
    char *mtiled = nullptr; // 12-real FP32 / FX16: tile-major copy (kMTile)
    size_t mtiled_parity_bytes = 0, mtile_bytes = 0;
    // test hooks of the staged FX16 kernel, read once when the handle is
    // created (STG_FX16_GRID, STG_FX16_TEST_DROP_FILL): a cap on its CTA
    // count (0 = none) and the withheld fill of the failure-detection test
    int fx_grid_cap = 0;
    int fx_drop_fill = 0;
    const char *blk(int parity, int mu) const { return base + (size_t)(parity * 4 + mu) * blk_bytes; }
};

struct Workspace;

// Workspace of the multi-system CG (mrhs.cu): n systems of every vector.
struct MrhsWs {
    int nrhs = 0, pd = -1;
    size_t f64 = 0, fr = 0, fd = 0;   // bytes of one FP64 / PR / PD field
    size_t pstride = 0;               // reduction partials per system (doubles)
    char *x64 = nullptr, *b64 = nullptr, *r64 = nullptr;
    char *y = nullptr, *r = nullptr, *d = nullptr, *q = nullptr, *t = nullptr;
    double *partials = nullptr;
    CGState *states = nullptr, *states_host = nullptr;
    int *active = nullptr, *active_host = nullptr;  // [0] = count, [1..] = systems
    void *tmp = nullptr;
    cudaGraphExec_t graph = nullptr;
    int graph_iters = 0;
    int shape = 0;                    // autotuned (NB, threads per site) index
    // The iteration's kernels by programmatic dependent launch: for a solve of
    // its own (12^3x24 n = 8 19.6 -> 18.5 ms), not for sessions, which run side by
    // side: waiting blocks keep places that other streams' kernels need.
    // Served stream at 200 requests/s, three runs each, without / with: p99 744,
    // 787, 804 / 979, 1124, 1026 ms (24^3x48 p50 558-604 / 828-945 ms).
    bool pdl = false;
};
void mrhs_free(MrhsWs *m);
void batch_destroy(stg_batch *b);
size_t mrhs_bytes(const Geom &g, int n, int pd);

}  // namespace stg

struct stg_gauge {
    int dims[4];
    stg::Geom geom;
    int device;
    int sloppy;             // stg_prec of the low-precision copy (P64 = none)
    stg::LinkField hi;      // FP64 links
    stg::LinkField lo;      // sloppy links (base == nullptr when sloppy == FP64)
    stg::Workspace *ws;     // lazily created
};

namespace stg {

// per-thread error text
void set_error(const std::string &msg);
stg_status cuda_fail(cudaError_t e, const char *what);

#define STG_CUDA(call)                                                   \
    do {                                                                 \
        cudaError_t e_ = (call);                                         \
        if (e_ != cudaSuccess) return ::stg::cuda_fail(e_, #call);       \
    } while (0)

#define STG_TRY(call)                                                    \
    do {                                                                 \
        stg_status s_ = (call);                                          \
        if (s_ != STG_OK) return s_;                                     \
    } while (0)

Geom make_geom(const int dims[4]);

// The state's scalars in FP32 numbers for the mixed CG's kernels (before a copy
// to the device, inner precision pd), and back (after one from it); all bits
// both ways.
inline void state_put(CGState *h, int pd)
{
    h->ff = pd != P64;
    h->m2f = (float)h->m2;
    h->f_stop = f3_split(h->stop_r2);
    h->f_delta = f3_split(h->delta_new);
    h->f_delta_old = f3_split(h->delta_old);
    h->f_rmax2 = f3_split(h->rmax2);
    h->f_trig = f3_split(h->trig2 * h->rmax2);
}
inline void state_got(CGState *h)
{
    if (!h->ff) return;
    h->delta_new = f3_double(h->f_delta);
    h->delta_old = f3_double(h->f_delta_old);
    h->rmax2 = f3_double(h->f_rmax2);
}

// stg_cg_params defaults for inner iterations in `sloppy` (api.cu)
void cg_params_for(int sloppy, stg_cg_params *p);

const LinkField *links_for(const stg_gauge *g, int prec);

// FP64 links as limbs (gauge.cu): links_check raises *bad (device) where one
// of n canonical links is not unitary or does not fit the form; links_fix
// converts a packed FP64 field in place
stg_status links_check(const double2 *ucan, long n, int recon, int *bad, cudaStream_t s);
stg_status links_fix(const Geom &g, LinkField *lf, cudaStream_t s);

// Reduction scratch: partial sums (one double per block) and the state.
struct Workspace {
    double *partials = nullptr;
    double *rr = nullptr;          // kRrPartials more behind them: |r|^2 of the update
    size_t n_partials = 0;
    CGState *state = nullptr;      // device
    CGState *state_host = nullptr; // pinned mirror for read-back
    void *tmp[kNumPrec] = {};  // odd intermediate per precision
    // CG vectors (allocated by the solver)
    void *x64 = nullptr, *b64 = nullptr, *r64 = nullptr, *t64 = nullptr;
    void *y = nullptr, *r = nullptr, *d = nullptr, *q = nullptr;
    int cg_sloppy = -1;
    // captured chunks of iterations: [0] plain (programmatic dependent
    // launch), [1] with per-kernel events, [2] plain without dependent launch
    cudaGraphExec_t graph[3] = {nullptr, nullptr, nullptr};
    int graph_sloppy[3] = {-1, -1, -1}, graph_iters[3] = {0, 0, 0};
    cudaEvent_t ev[5] = {nullptr, nullptr, nullptr, nullptr, nullptr};  // per-kernel events
    cudaEvent_t ev_chunk[2] = {nullptr, nullptr};                        // around plain chunks
    stg_batch *batch = nullptr;       // session cached for stg_cg_solve_mrhs
    void *cl_dev = nullptr, *cl_host = nullptr;  // systems of cluster_solve (device, pinned)
    void *mrhs_tmp = nullptr;         // odd intermediates of stg_apply_A_mrhs
    size_t mrhs_tmp_bytes = 0;
};

stg_status workspace_get(stg_gauge *g, Workspace **out);
stg_status workspace_tmp(stg_gauge *g, int prec, void **out);
void workspace_free(Workspace *ws);

// kernels (launch only; all on `s`)
enum Epi { EPI_NONE = 0, EPI_A = 1, EPI_A_DOT = 2, EPI_A_CG = 3, EPI_RES = 4, EPI_GATE = 5 };

struct DslashLaunch {
    const LinkField *links;
    int out_parity;
    const void *in;
    void *out;
    const void *w;   // EPI_A*: the even input d (m^2 d term, d^dag q); EPI_RES: b
    const void *v;   // EPI_RES: x
    double m2;
    double *dot;     // EPI_A_DOT: result
    CGState *state;  // EPI_A_CG, EPI_GATE
    double *partials;
    unsigned *counter;
    bool pdl;        // programmatic dependent launch: the kernel's blocks are
                     // placed while the previous kernel of the stream drains
                     // and wait for its end before they touch a field
};

stg_status launch_dslash(const Geom &g, int prec, int epi, const DslashLaunch &a, cudaStream_t s);
// thread blocks (and block partials) of the one-site kernel; limbs12: FP64 / 12-
// real limb links
int dslash_blocks(int vh, int epi, bool limbs12);

// kernel arguments of every Dslash variant
struct DslashArgs {
    Geom g;
    const char *lf[4];  // forward link blocks  (parity p,   mu)
    const char *lb[4];  // backward link blocks (parity 1-p, mu)
    const char *lt;     // tile-major links of output parity p (FX16 / 12), or null
    int grid_cap;       // staged kernel: at most this many CTAs (0 = one per SM)
    int drop_fill;      // tests only: the staged kernel withholds the fill of
                        // its second tile's first stage, so that bounded
                        // wait runs out
    int parity;
    const void *in;
    void *out;
    const void *w;
    const void *v;
    double m2;
    float m2f;          // m2 in FP32: a conversion per thread costs 16 cycles of the FP64 pipe a warp
    double *dot;
    CGState *state;
    double *partials;
    unsigned *counter;
};

// FP16 / FX16 Dslash on packed FP32x2 arithmetic (dslash_fx16.cu); false
// where the one-site kernel of dslash.cu is the faster one
bool launch_dslash_16(int prec, int recon, int epi, const DslashArgs &a, cudaStream_t s, bool pdl);

int grid_for(long n);

// vector-kernel helpers with explicit operands (cg.cu)
// dq: A's block partials of d^dag q, system k's at k times their number per
// system (CGState::n_part); rr: room for kRrPartials doubles a system
constexpr int kRrPartials = 384;
stg_status launch_update_m(int pd, int vh, char *y, char *r, const char *d, const char *q, size_t sr,
                           size_t sd, CGState *states, const double *dq, double *rr, const int *active,
                           const int *nactive, int nslots, bool pdl, cudaStream_t s);
stg_status launch_xpay_m(int pd, int vh, const char *r, char *d, size_t sr, size_t sd, CGState *states,
                         const double *rr, const int *active, const int *nactive, int nslots, bool pdl,
                         cudaStream_t s);
stg_status launch_reset(int pd, int vh, void *y, void *r, void *d, const void *r64, double beta,
                        int copy_r, cudaStream_t s);
stg_status launch_accumulate_x(int pr, int vh, void *x64, const void *y, cudaStream_t s);
stg_status launch_norm2(int prec, int vh, const void *v, CGState *st, double *partials, cudaStream_t s);
stg_status launch_true_residual(stg_gauge *g, const void *x64, const void *b64, void *r64, void *t64,
                                double m2, CGState *st, double *partials, cudaStream_t s);
// whole solves of small lattices in one kernel (cg_cluster.cu)
struct ClFields {
    void *x64, *t64, *y, *r, *d, *q, *t;
};
int cluster_ctas(const stg_gauge *g, int pd, int nsys, bool batch);
stg_status cluster_solve(stg_gauge *g, Workspace *ws, int ctas, int nsys, bool batch, const ClFields &buf, const double *src,
                         double *x, const double *masses, double tol, const stg_cg_params *p, int pd,
                         stg_cg_stats *stats, cudaStream_t s);
stg_status pack_field(const Geom &g, int prec, const double *canon, void *out, cudaStream_t s);
stg_status unpack_field(const Geom &g, int prec, const void *in, double *canon, cudaStream_t s);

}  // namespace stg
