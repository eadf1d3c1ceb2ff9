"""Which kernel a half-pass runs: the 16-bit forms that take the one-site
kernel give the bits of the group launch, which always runs it."""
import functools

import pytest
import torch

import gen
import paper_1111_0125_gb300 as stg

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dims", [(2, 2, 2, 2), (12, 12, 12, 24)])
@pytest.mark.parametrize("prec,recon", [(stg.STG_FP16, 12), (stg.STG_FP16, 18), (stg.STG_FX16, 18)])
def test_one_site_kernel_runs(dims, prec, recon):
    U = gen.gauge_field(dims, "exp", seed=4, eps=0.5)
    chi = torch.from_numpy(gen.source(dims, seed=9)).cuda()
    with stg.Gauge(dims, U, sloppy=prec, recon=recon) as g:
        f = g.pack(chi, prec)
        for parity in (0, 1):
            group = torch.empty_like(f)
            stg.stg_dslash_group([g.handle], [parity], [f], [group], prec)
            assert torch.equal(g.dslash(f, parity, prec), group)


@functools.lru_cache(maxsize=1)
def haar(dims):
    return gen.gauge_field(dims, "haar", seed=5)


@pytest.mark.parametrize("prec,recon", [(stg.STG_FP32, 12), (stg.STG_FP32, 18), (stg.STG_FP16, 12), (stg.STG_FP16, 18),
                                        (stg.STG_BF16, 12), (stg.STG_BF16, 18), (stg.STG_FX16, 18)])
# in blocks of 256 sites: a partial one; 81 of 128 sites; 256; 288; 375; 437.5; 531.25; 864.
# Links copied ahead: FP32/18 up to 152, FP32/12 to 280, 16 bits to 304 (12 reals) and 456.
# Dense: FP32/18 from 240; FP32/12 at 375, 437.5 and 864; FP16/18, BF16/18 from 531.25,
# FX16/18 at 531.25; FP16/12, BF16/12 at 864
@pytest.mark.parametrize("dims", [(2, 2, 2, 6), (12, 12, 12, 12), (16, 16, 16, 32), (16, 16, 18, 32), (20, 20, 20, 24),
                                  (20, 20, 20, 28), (20, 20, 20, 34), (24, 24, 24, 32)])
def test_every_form_gives_the_bits_of_the_group_launch(dims, prec, recon):
    """The forms (first, fewer registers, links copied ahead) run the same
    arithmetic as the group launch's sites; the A with the dot gives the bits
    of the A without, and its dot that of the fields."""
    with stg.Gauge(dims, haar(dims), sloppy=prec, recon=recon) as g:
        f = g.pack(torch.from_numpy(gen.source(dims, seed=9)).cuda(), prec)
        for parity in (0, 1):
            group = torch.empty_like(f)
            stg.stg_dslash_group([g.handle], [parity], [f], [group], prec)
            assert torch.equal(g.dslash(f, parity, prec), group)
        out, dot = torch.empty_like(f), torch.empty(1, dtype=torch.float64, device="cuda")
        stg.stg_apply_A_dot(g.handle, 0.2, f, out, dot, prec)
        assert torch.equal(out, g.apply_A(f, 0.2, prec))
        x, y = g.unpack(f, prec), g.unpack(out, prec)
        want = torch.sum(x.conj() * y).real
        assert abs(dot[0] - want) <= 1e-6 * torch.sum(x.abs() * y.abs())


@pytest.mark.parametrize("prec,recon", [(stg.STG_FP64, 18), (stg.STG_FP32, 12), (stg.STG_FP16, 12)])
def test_early_placed_blocks_wait_for_the_input(prec, recon):
    """The operators' kernels may be placed while their predecessor runs; the
    input's producer is a copy, a memset, another library's kernel or another
    stream's, eagerly and in a captured graph, and the output never changes."""
    dims, mass = (16, 16, 16, 16), 0.1
    with stg.Gauge(dims, gen.gauge_field(dims, "exp", seed=1, eps=0.5), sloppy=prec, recon=recon) as g:
        x = g.pack(torch.from_numpy(gen.source(dims, seed=2)).cuda(), prec)
        f, out, dot = torch.empty_like(x), torch.empty_like(x), torch.empty(1, dtype=torch.float64, device="cuda")
        side = torch.cuda.Stream()

        def call():
            stg.stg_apply_A_dot(g.handle, mass, f, out, dot, prec)

        def produce(kind):
            f.zero_()
            if kind == 0:
                f.copy_(x)
            elif kind == 1:
                f.add_(x)
            else:
                cur = torch.cuda.current_stream()
                side.wait_stream(cur)
                with torch.cuda.stream(side):
                    f.copy_(x)
                cur.wait_stream(side)

        f.copy_(x)
        call()
        want, want_dot = out.clone(), dot.clone()
        for k in range(30):
            produce(k % 3)
            call()
            got = out.clone()
            assert torch.equal(got, want) and torch.equal(dot, want_dot)
        stream, graph = torch.cuda.Stream(), torch.cuda.CUDAGraph()
        stream.wait_stream(torch.cuda.current_stream())
        with torch.cuda.stream(stream), torch.cuda.graph(graph, stream=stream):
            call()
            for kind in range(3):
                produce(kind)
                call()
        for _ in range(5):
            out.zero_()
            graph.replay()
            torch.cuda.synchronize()
            assert torch.equal(out, want) and torch.equal(dot, want_dot)


@pytest.mark.parametrize("n", [1, 2, 3, 4, 5, 7])
@pytest.mark.parametrize("prec,tol", [(stg.STG_FP32, 1e-6), (stg.STG_FX16, 1e-4)])
def test_batches_with_empty_and_odd_groups(n, prec, tol, monkeypatch):
    """The staged multi-system kernel's four site groups share the systems; at
    these sizes some have none or a single last one.  Against the single-system
    A (each within the precision's tolerance of the exact one, so within twice
    that of each other)."""
    dims, mass = (4, 6, 2, 8), 0.3
    monkeypatch.setenv("STG_MRHS_SHAPE", "14")
    chis = torch.from_numpy(gen.source(dims, seed=3, nrhs=n)).cuda()
    with stg.Gauge(dims, gen.gauge_field(dims, "haar", seed=1), sloppy=prec, recon=12) as g:
        buf = torch.cat([g.pack(c, prec) for c in chis])
        out = torch.full_like(buf, 255)
        stg.stg_apply_A_mrhs(g.handle, n, [mass + k for k in range(n)], buf, out, prec)
        size = out.numel() // n
        for k in range(n):
            got = g.unpack(out[k * size:(k + 1) * size], prec)
            want = g.unpack(g.apply_A(g.pack(chis[k], prec), mass + k, prec), prec)
            assert torch.linalg.vector_norm(got - want) <= 2 * tol * torch.linalg.vector_norm(want)
