"""Split-FP16 MP2 on either side of the size from which its transform is a sliced
product (80 functions): within 2^-18 of the absolute term sum (the bound of the
split pair blocks, 2^-22 a factor) of plain torch FP64 on the same tensor."""
import pytest

import workload

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("name", ["w3", "w4"])  # N = 75 and 100
def test_f16x3_transform_routes(gpu_ctx, name):
    import torch
    import paper_2502_17963_gb300 as bqc
    basis = bqc.Basis(gpu_ctx, workload.molecule_for(name))
    df = bqc.DF(gpu_ctx, basis, keep_fp32=False)
    n, no = basis.nbf, basis.nocc
    r = bqc.scf_run(gpu_ctx, df, keep_arrays=True)
    C, eps = r["C"].contiguous(), r["eps"].contiguous()
    i, j = torch.tril_indices(n, n, device="cuda")
    B = torch.zeros((basis.naux, n, n), dtype=torch.float64, device="cuda")
    B[:, i, j] = df.copy(0)
    B[:, j, i] = B[:, i, j]
    ov = torch.einsum("mi,pmn,na->pia", C[:, :no], B, C[:, no:])
    v = torch.einsum("pia,pjb->iajb", ov, ov)
    den = (eps[:no, None, None, None] - eps[None, no:, None, None]
           + eps[None, None, :no, None] - eps[None, None, None, no:])
    terms = v * (2 * v - v.transpose(1, 3)) / den
    e2 = bqc.mp2(df, C, eps, bqc.PREC_MIXED_F16X3)
    assert abs(e2 - float(terms.sum())) <= 2.0 ** -18 * float(terms.abs().sum())
