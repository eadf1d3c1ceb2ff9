// Whole solves of small lattices in one kernel (cg_cluster.cuh): where that is
// the faster way, and the host side of stg_cg_solve and stg_cg_solve_mrhs there.
#include <math.h>
#include <string.h>
#include <time.h>

#include <array>

#include "cg_cluster.cuh"

namespace stg {

// Where one kernel per solve is the faster way, and the CTAs per cluster for
// it (0: not).  Microseconds per iteration, its share of the updates included,
// measured on exp(0.5) links at m = 0.02 with FP32 inner iterations:
//   cluster, by sites per CTA: 128: 6.9 (8^4); 256: 8.7; 512: 9.2; 648: 14.2;
//     1296: 20.5; 2592: 35; 4096: 55; 8192: 103;
//   four kernels per iteration, one system: 13.5 (8^4), 12.5 (8^3x16), 14.6
//     (12^4), 13.0 (12^3x24), 17.0 (16^3x32); batches of 2 / 4 / 8 / 16: 20 / 24
//     / 32 / 50 on 8^4, 20 / 28 / 34 / 53 on 12^3x24, 22 / 30 / 45 / 71 on 16^4,
//     25 / - / 57 / 93 on 16^3x32.
// One system takes the cluster up to 512 sites per CTA (12^4, 648: 4.3 against
// 4.2 ms); a batch by the estimates below, with as many CTAs per system as let
// the clusters run side by side (152 SMs: seven clusters of 16 CTAs, eight of
// 12, fifteen of 8, 23 of 6, 36 of 4).  Plain FP64 (limbs, one site per thread):
// 8^4 4.0 against 6.0 ms, 8^3x16 10.7 against 12.7, 12^4 14.8 against 7.9.
static double cluster_us(int per) { return per <= kClThreads / 4 ? 6.9 : per <= kClThreads ? 9.0 : 7.5 + 0.0115 * per; }

int cluster_ctas(const stg_gauge *g, int pd, int nsys, bool batch)
{
    const LinkField *lf = links_for(g, pd);
    const int vh = g->geom.Vh;
    if (!g->hi.fix || !lf || nsys > kClMaxSystems) return 0;
    if (lf->fx_grid_cap > 0 || lf->fx_drop_fill) return 0;  // tests of the staged kernel
    static const int sizes[] = {16, 12, 10, 8, 6, 4};
    const std::array<int, 6> active = per_device([] {
        std::array<int, 6> a;
        for (int z = 0; z < 6; ++z) a[z] = cl_active_clusters(sizes[z]);
        return a;
    });
    if (active[0] < 1) return 0;
    // none where the device does not grant the kernel what it needs
    const auto granted = [&](int ctas) {
        const int per = ctas ? (vh + ctas - 1) / ctas : 0;
        return !ctas ? 0 : (pd == P64 || pd == P32 ? cl_granted_wide(pd, lf->recon, per) : cl_granted_16(pd, lf->recon, per)) ? ctas : 0;
    };
    if (pd == P64) return granted(vh <= 4096 ? 16 : 0);
    if (!batch) return granted(vh <= 16 * kClThreads ? 16 : 0);
    double best = 16.0 + 2.0 * nsys + 3.9e-5 * nsys * (double)vh;  // the four kernels
    int ctas = 0;
    for (int z = 0; z < 6; ++z) {
        if (active[z] < 1) continue;
        const int waves = (nsys + active[z] - 1) / active[z];
        const double us = waves * cluster_us((vh + sizes[z] - 1) / sizes[z]);
        if (us < best) {
            best = us;
            ctas = sizes[z];
        }
    }
    return granted(ctas);
}

// The solves of cg_solve and cg_solve_mrhs for small lattices; buf: the work
// fields (x64, t64, y, r, d, q, t), one per system and consecutive.
// batch: the form of stg_cg_solve_mrhs (x of every system stored, whatever its
// outcome, once none has a bad input).
stg_status cluster_solve(stg_gauge *g, Workspace *ws, int ctas, int nsys, bool batch, const ClFields &buf, const double *src,
                         double *x, const double *masses, double tol, const stg_cg_params *p, int pd,
                         stg_cg_stats *stats, cudaStream_t s)
{
    const std::string who = batch ? "stg_cg_solve_mrhs: " : "stg_cg_solve: ";
    timespec t0, t1;
    clock_gettime(CLOCK_MONOTONIC, &t0);
    const Geom &geo = g->geom;
    const int vh = geo.Vh;
    const bool plain = pd == P64;
    cudaError_t e = cudaSuccess;
    if (!ws->cl_dev) e = cudaMalloc(&ws->cl_dev, kClMaxSystems * sizeof(ClSystem));
    if (e == cudaSuccess && !ws->cl_host) e = cudaMallocHost(&ws->cl_host, kClMaxSystems * sizeof(ClSystem));
    if (e != cudaSuccess) return cuda_fail(e, "cluster workspace");
    ClSystem *h = static_cast<ClSystem *>(ws->cl_host);
    memset(h, 0, nsys * sizeof(ClSystem));
    for (int k = 0; k < nsys; ++k) {
        h[k].m2 = masses[k] * masses[k];
        h[k].tol2 = tol * tol;
        h[k].trig2 = plain ? 0.0 : p->delta * p->delta;
        h[k].iter_limit = p->maxiter > 0 ? p->maxiter : 10L * 3L * vh;
    }
    ClArgs a;
    a.g = geo;
    const LinkField *lf = links_for(g, pd);
    for (int b = 0; b < 8; ++b) {
        a.lk[b] = lf->blk(b / 4, b % 4);
        a.hi[b] = g->hi.blk(b / 4, b % 4);
    }
    a.src = reinterpret_cast<const double2 *>(src);
    a.x = reinterpret_cast<double2 *>(x);
    a.x64 = static_cast<char *>(buf.x64);
    a.t64 = static_cast<char *>(buf.t64);
    a.y = static_cast<char *>(buf.y);
    a.r = static_cast<char *>(buf.r);
    a.d = static_cast<char *>(buf.d);
    a.q = static_cast<char *>(buf.q);
    a.t = static_cast<char *>(buf.t);
    a.f64 = (size_t)vh * 48;
    a.fr = (size_t)vh * field_site_bytes(plain ? P64 : P32);
    a.fd = (size_t)vh * field_site_bytes(pd);
    a.sys = static_cast<ClSystem *>(ws->cl_dev);
    a.eq6 = p->policy == STG_CG_RELIABLE;
    a.max_breakdowns = batch ? 64 : 3;
    a.write_x = !batch;
    a.lsm = 0;
    a.dper = make_fastdiv(1u);
    STG_CUDA(cudaMemcpyAsync(a.sys, h, nsys * sizeof(ClSystem), cudaMemcpyHostToDevice, s));
    long launches = 0;
    for (bool again = true; again;) {
        if (pd == P64 || pd == P32) STG_CUDA(cl_dispatch_wide(pd, lf->recon, a, nsys, ctas, s));
        else STG_CUDA(cl_dispatch_16(pd, lf->recon, a, nsys, ctas, s));
        ++launches;
        STG_CUDA(cudaMemcpyAsync(h, a.sys, nsys * sizeof(ClSystem), cudaMemcpyDeviceToHost, s));
        STG_CUDA(cudaStreamSynchronize(s));
        again = false;
        for (int k = 0; k < nsys; ++k) again = again || h[k].status == CL_RUNNING;
    }
    stg_status worst = STG_OK;
    for (int k = 0; k < nsys && worst == STG_OK; ++k) {
        if (h[k].status == CL_BAD_SOURCE) {
            set_error(who + "the source has non-finite entries");
            worst = STG_ERR_INVALID_ARG;
        } else if (h[k].status == CL_BAD_START) {
            set_error(who + "non-finite residual of the initial guess");
            worst = STG_ERR_INVALID_ARG;
        }
    }
    if (worst != STG_OK) return worst;
    bool stored = false;
    for (int k = 0; k < nsys; ++k) {
        double *xk = x + (size_t)k * vh * 6;
        if (h[k].bb == 0.0) {
            STG_CUDA(cudaMemsetAsync(xk, 0, (size_t)vh * 48, s));
            stored = true;
        } else if (batch) {
            STG_TRY(unpack_field(geo, P64, a.x64 + k * a.f64, xk, s));
            ++launches;
            stored = true;
        }
    }
    if (stored) STG_CUDA(cudaStreamSynchronize(s));
    clock_gettime(CLOCK_MONOTONIC, &t1);
    for (int k = 0; k < nsys; ++k) {
        if (h[k].status != CL_OK && worst == STG_OK) {
            worst = h[k].status == CL_BREAKDOWN ? STG_ERR_BREAKDOWN : STG_ERR_NOT_CONVERGED;
            set_error(who + (worst == STG_ERR_BREAKDOWN ? "d^dag A d <= 0 or a non-finite residual"
                                                        : "maxiter reached before convergence"));
        }
        if (!stats) continue;
        stg_cg_stats st = {};
        if (h[k].bb > 0.0) {
            st.iters = (long)h[k].iter;
            st.sloppy_iters = plain ? 0 : st.iters;
            st.updates = h[k].updates;
            st.true_res = sqrt(h[k].rr / h[k].bb);
            st.iter_res = sqrt(h[k].delta_new / h[k].bb);
            st.launches = launches;
            st.seconds = (t1.tv_sec - t0.tv_sec) + 1e-9 * (t1.tv_nsec - t0.tv_nsec);
        }
        stats[k] = st;
    }
    return worst;
}

}  // namespace stg
