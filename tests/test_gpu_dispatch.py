"""Which kernel a half-pass runs: the 16-bit forms that take the one-site
kernel give the bits of the group launch, which always runs it."""
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
