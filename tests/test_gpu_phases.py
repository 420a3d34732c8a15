"""Phase times of an FP64 build (bqc_df_phase_ms): [0] the X pass, [1] J, [2] K
with its reduction, also where the build alternates X and K by chunks."""
import pytest

import workload

pytestmark = pytest.mark.gpu


# sliced builds in one chunk and in several (N = 125, 325)
@pytest.mark.parametrize("name", ["w5", "w13"])
def test_k_is_in_its_own_phase(gpu_ctx, name):
    import torch
    import paper_2502_17963_gb300 as bqc
    basis = bqc.Basis(gpu_ctx, workload.molecule_for(name))
    df = bqc.DF(gpu_ctx, basis, keep_fp32=False)
    C = torch.randn((basis.nbf, basis.nocc), device="cuda", dtype=torch.float64)
    df.jk(C, bqc.PREC_FP64)
    df.timing()
    for _ in range(3):
        beg, end = (torch.cuda.Event(enable_timing=True) for _ in range(2))
        beg.record()
        df.jk(C, bqc.PREC_FP64)
        end.record()
        x, j, k, prep = df.phase_ms()
        assert min(x, j, k) > 0 and prep >= 0
        # K is half of X's multiply-adds on operands of half its slices' bytes
        assert 0.1 * x < k < 2 * x
        assert x + j + k + prep <= beg.elapsed_time(end) * 1.01 + 0.01
