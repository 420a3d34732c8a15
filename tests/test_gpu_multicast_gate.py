"""Cluster multicast loads are for one process on one GPU: a rank of a larger job
runs the plain X pass, with the same bits."""
import pytest

import workload

pytestmark = pytest.mark.gpu


# N = 100, 200, 325: one row-tile pair a cluster, and odd tile counts
@pytest.mark.parametrize("name", ["w4", "w8", "w13"])
def test_rank_of_a_larger_job_uses_plain_loads(monkeypatch, name):
    import torch
    import paper_2502_17963_gb300 as bqc
    out = []
    for world in (None, "1", "2"):
        if world is None:
            monkeypatch.delenv("WORLD_SIZE", raising=False)
        else:
            monkeypatch.setenv("WORLD_SIZE", world)
        ctx = bqc.Context(0)
        assert ctx.multicast == (world != "2" and torch.cuda.device_count() == 1)
        basis = bqc.Basis(ctx, workload.molecule_for(name))
        df = bqc.DF(ctx, basis, keep_fp32=bqc.SHADOW_F16)
        g = torch.Generator(device="cuda").manual_seed(9)
        C = torch.randn((basis.nbf, basis.nocc), generator=g, device="cuda", dtype=torch.float64)
        out.append(df.jk(C, bqc.PREC_MIXED_F16X3))
        torch.cuda.synchronize()
    for J, K in out[1:]:
        assert torch.equal(J, out[0][0]) and torch.equal(K, out[0][1])
