"""Whole solves of small lattices in one kernel (csrc/cg_cluster.cuh) where the
split over CTAs, lanes and systems can go wrong: fewer sites than CTAs, one
site per CTA more or less than a lane layout holds, ragged last CTAs, several
systems of different length, restarted launches, and the refusals."""
import numpy as np
import pytest
import torch

import gen
import oracle
import paper_1111_0125_gb300 as stg
from paper_1111_0125_gb300 import Gauge

pytestmark = pytest.mark.gpu

# Vh = 8 (half the CTAs empty), 192, 2048 = 16 x 128 (four lanes a site), 2160
# (one lane, ragged), 8064 (504 sites a CTA), 10368 (batches only)
DIMS = [(2, 2, 2, 2), (4, 6, 2, 8), (8, 8, 8, 8), (6, 6, 10, 12), (12, 12, 8, 14)]
PRECS = [(stg.STG_FP32, 12), (stg.STG_FP32, 18), (stg.STG_FP16, 12), (stg.STG_FX16, 12), (stg.STG_FX16, 18),
         (stg.STG_BF16, 12), (stg.STG_FP64, 18), (stg.STG_FP64, 12)]


@pytest.fixture(scope="module", autouse=True)
def _oracle():
    oracle.build()


def _check(dims, U, mass, b, x, tol):
    """The true residual with the oracle's A (1% for its own rounding)."""
    r = b - oracle.apply_A(dims, U, mass, x)
    assert np.linalg.norm(r) <= 1.01 * tol * np.linalg.norm(b)


@pytest.mark.parametrize("dims", DIMS)
@pytest.mark.parametrize("prec,recon", PRECS)
def test_solve(dims, prec, recon):
    mass, tol = 0.2, 1e-10
    U = gen.gauge_field(dims, "exp", seed=5, eps=0.4)
    b = gen.source(dims, seed=6)
    x0 = gen.source(dims, seed=7)
    with Gauge(dims, U, sloppy=prec, recon=recon) as g:
        x, st = g.cg_solve(torch.from_numpy(b).cuda(), mass, tol)
        _check(dims, U, mass, b, x.cpu().numpy(), tol)
        assert st["iters"] > 0 and st["updates"] >= 1 and st["true_res"] <= tol
        y, _ = g.cg_solve(torch.from_numpy(b).cuda(), mass, tol, x0=torch.from_numpy(x0))
        _check(dims, U, mass, b, y.cpu().numpy(), tol)
        again, _ = g.cg_solve(torch.from_numpy(b).cuda(), mass, tol)
        assert torch.equal(x, again)


@pytest.mark.parametrize("dims,n", [((2, 2, 2, 2), 64), ((8, 8, 8, 8), 3), ((8, 8, 8, 8), 17), ((12, 12, 12, 12), 8)])
@pytest.mark.parametrize("prec", [stg.STG_FP32, stg.STG_FX16])
def test_batch(dims, n, prec):
    """Masses over two decades: systems of very different length."""
    tol = 1e-10
    U = gen.gauge_field(dims, "exp", seed=8, eps=0.4)
    bs = gen.source(dims, seed=9, nrhs=n)
    masses = np.geomspace(0.02, 2.0, n)
    with Gauge(dims, U, sloppy=prec, recon=12) as g:
        src = torch.from_numpy(bs).cuda()
        src[n // 2] = 0.0
        x = torch.ones_like(src)
        st = stg.stg_cg_solve_mrhs(g.handle, n, src, x, masses, tol)
        for k in range(n):
            if k == n // 2:
                assert not torch.any(x[k]) and st[k]["iters"] == 0
            else:
                _check(dims, U, masses[k], bs[k], x[k].cpu().numpy(), tol)


@pytest.mark.parametrize("policy", [stg.STG_CG_RELIABLE, stg.STG_CG_REFINE])
def test_same_iteration_as_the_kernel_sequence(policy):
    """timing = 1 runs the four-kernel sequence: the same iteration to the
    rounding of the sums, so the counts agree to 5% and both solve."""
    dims, mass, tol = (8, 8, 8, 8), 0.05, 1e-10
    U = gen.gauge_field(dims, "exp", seed=3, eps=0.5)
    b = gen.source(dims, seed=4)
    with Gauge(dims, U, sloppy=stg.STG_FP32, recon=12) as g:
        out = [g.cg_solve(torch.from_numpy(b).cuda(), mass, tol, g.params(timing=t, policy=policy)) for t in (0, 1)]
    for x, _ in out:
        _check(dims, U, mass, b, x.cpu().numpy(), tol)
    (_, s0), (_, s1) = out
    assert abs(s0["iters"] - s1["iters"]) <= 0.05 * s1["iters"] and abs(s0["updates"] - s1["updates"]) <= 2


def test_iteration_limit_and_refusals():
    dims = (8, 8, 8, 8)
    U = gen.gauge_field(dims, "exp", seed=3, eps=0.5)
    b = torch.from_numpy(gen.source(dims, seed=4)).cuda()
    with Gauge(dims, U, sloppy=stg.STG_FP32, recon=12) as g:
        # tol 1e-17 is out of reach of FP64: launches of 4096 iterations are
        # restarted up to maxiter, and x holds the last iterate
        for tol, maxiter, status in ((1e-10, 7, stg.STG_ERR_NOT_CONVERGED), (1e-17, 9000, stg.STG_ERR_NOT_CONVERGED)):
            x = torch.zeros_like(b)
            with pytest.raises(stg.StgError) as e:
                stg.stg_cg_solve(g.handle, b, x, 0.05, tol, g.params(maxiter=maxiter))
            assert e.value.status == status and e.value.stats["iters"] >= maxiter
            assert torch.isfinite(torch.view_as_real(x)).all() and torch.any(x)
        for bad in (float("nan"), float("inf")):
            c = b.clone()
            c[5, 1] = bad
            for src, x in ((c, torch.zeros_like(b)), (b, c)):
                keep = x.clone()
                with pytest.raises(stg.StgError) as e:
                    stg.stg_cg_solve(g.handle, src, x, 0.05, 1e-10)
                assert e.value.status == stg.STG_ERR_INVALID_ARG
                assert torch.equal(torch.view_as_real(x).isnan(), torch.view_as_real(keep).isnan())
                with pytest.raises(stg.StgError) as e:
                    stg.stg_cg_solve_mrhs(g.handle, 2, torch.stack([b, src]), torch.stack([keep, x]), [0.05, 0.1],
                                          1e-10)
                assert e.value.status == stg.STG_ERR_INVALID_ARG
        x = torch.ones_like(b)
        st = stg.stg_cg_solve(g.handle, torch.zeros_like(b), x, 0.05, 1e-10)
        assert not torch.any(x) and st["iters"] == 0


def test_concurrent_streams():
    """Two handles on two streams: each solves as it does alone, bit for bit."""
    dims = (8, 8, 8, 8)
    b = torch.from_numpy(gen.source(dims, seed=4)).cuda()
    gs = [Gauge(dims, gen.gauge_field(dims, "exp", seed=s, eps=0.5), sloppy=stg.STG_FP32, recon=12) for s in (1, 2)]
    try:
        alone = [g.cg_solve(b, 0.05, 1e-10)[0] for g in gs]
        import threading
        got = [None, None]

        def work(k):
            with torch.cuda.stream(torch.cuda.Stream()):
                for _ in range(3):
                    got[k] = gs[k].cg_solve(b, 0.05, 1e-10)[0]

        ts = [threading.Thread(target=work, args=(k,)) for k in range(2)]
        [t.start() for t in ts]
        [t.join() for t in ts]
        torch.cuda.synchronize()
        for k in range(2):
            assert torch.equal(got[k], alone[k])
    finally:
        for g in gs:
            g.close()
