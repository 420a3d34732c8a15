"""The Coulomb part of a TF32x3 build adds its aux chunks (of at least 64
functions) in order: a staged SCF's result depends on the last bits of its mixed
builds.  A shard of one chunk is one running sum, and the w_P of a shard are the
whole handle's, so the whole J is the shards' J added up one after the other."""
import pytest

import workload

pytestmark = pytest.mark.gpu


# Naux = 150 (2 chunks of 75), 300 (4), 375 (5)
@pytest.mark.parametrize("name", ["w2", "w4", "w5"])
def test_tf32x3_coulomb_adds_chunks_of_75(gpu_ctx, name):
    import torch
    import paper_2502_17963_gb300 as bqc
    basis = bqc.Basis(gpu_ctx, workload.molecule_for(name))
    g = torch.Generator(device="cuda").manual_seed(3)
    C = torch.randn((basis.nbf, basis.nocc), generator=g, device="cuda", dtype=torch.float64)
    J = bqc.DF(gpu_ctx, basis, keep_fp32=bqc.SHADOW_TF32).jk(C, bqc.PREC_MIXED_TF32X3)[0]
    total = None
    for p in range(0, basis.naux, 75):
        part = bqc.DF(gpu_ctx, basis, keep_fp32=bqc.SHADOW_TF32, aux_range=(p, p + 75))
        one = part.jk(C, bqc.PREC_MIXED_TF32X3)[0]
        total = one if total is None else total + one
    assert torch.equal(J, total)
