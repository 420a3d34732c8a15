"""Device memory stays within what is declared: AUTO mode's limit, the serving
ledger's footprint, and the peak of a shard's build."""
import ctypes

import pytest

import workload

pytestmark = pytest.mark.gpu

MB = 1 << 20


@pytest.fixture()
def tracked():
    """A context whose allocations are summed: live and peak bytes."""
    import torch
    import paper_2502_17963_gb300 as bqc
    from paper_2502_17963_gb300 import _build
    _build.build()
    size, state = {}, {"live": 0, "peak": 0}

    def alloc(nbytes, _):
        p = torch.cuda.caching_allocator_alloc(int(nbytes), 0)
        size[p] = int(nbytes)
        state["live"] += int(nbytes)
        state["peak"] = max(state["peak"], state["live"])
        return p

    def free(ptr, _):
        state["live"] -= size.pop(ptr)
        torch.cuda.caching_allocator_delete(ptr)

    ctx = bqc.Context.__new__(bqc.Context)
    ctx.device, ctx.h = 0, ctypes.c_void_p()
    ctx._afn, ctx._ffn = bqc.ALLOC_FN(alloc), bqc.FREE_FN(free)
    bqc.check(bqc.lib().bqc_ctx_create(0, 0, ctx._afn, ctx._ffn, None, ctypes.byref(ctx.h)),
              "bqc_ctx_create")
    yield torch, bqc, ctx, state
    ctx.close()


# the largest scratch beyond X (N = 100 to 150), none to speak of (N = 26, 325)
@pytest.mark.parametrize("name", ["h2o", "w4", "w6", "w13"])
@pytest.mark.parametrize("shadow", ["NONE", "F16", "TF32"])
def test_auto_mode_holds_no_more_than_its_limit(gpu_ctx, name, shadow):
    """The smallest limit at which AUTO stores the tensor: the handle holds at
    most that (1 MB for the screening plan, which the limit does not count), and
    builds what an unlimited one does to rounding: 16 Naux N nocc 2^-53 of the
    largest products."""
    import torch
    import paper_2502_17963_gb300 as bqc
    basis = bqc.Basis(gpu_ctx, workload.molecule_for(name))
    kw = dict(keep_fp32=getattr(bqc, "SHADOW_" + shadow))
    full = bqc.DF(gpu_ctx, basis, **kw)
    lo, hi = 1, 2 * full.device_bytes
    while hi - lo > 1:
        mid = (lo + hi) // 2
        df = bqc.DF(gpu_ctx, basis, mode=bqc.DF_AUTO, hbm_limit=mid, **kw)
        lo, hi = (lo, mid) if df.mode == bqc.DF_STORED else (mid, hi)
        df.close()
    df = bqc.DF(gpu_ctx, basis, mode=bqc.DF_AUTO, hbm_limit=hi, **kw)
    assert df.mode == bqc.DF_STORED
    assert df.device_bytes <= hi + MB
    g = torch.Generator(device="cuda").manual_seed(2)
    C = torch.randn((basis.nbf, basis.nocc), generator=g, device="cuda", dtype=torch.float64)
    C = C / basis.nbf ** 0.5
    eps = 16 * basis.naux * basis.nbf * basis.nocc * 2.0 ** -53
    D = C @ C.T
    for a, b in list(zip(df.jk(C), full.jk(C))) + [(df.coulomb(D), full.coulomb(D))]:
        assert (a - b).abs().max() <= eps * b.abs().max()


@pytest.mark.parametrize("name", ["h2o", "w2", "w4", "w6", "w13", "w20"])
@pytest.mark.parametrize("prec", ["FP64", "MIXED_F16X3", "MIXED_TF32X3"])
def test_a_solve_stays_within_its_footprint(tracked, name, prec):
    torch, bqc, ctx, state = tracked
    p = getattr(bqc, "PREC_" + prec)
    shadow = {"FP64": bqc.SHADOW_NONE, "MIXED_F16X3": bqc.SHADOW_F16}.get(prec, bqc.SHADOW_TF32)
    basis = bqc.Basis(ctx, workload.molecule_for(name))
    df = bqc.DF(ctx, basis, keep_fp32=shadow)
    bqc.scf_run(ctx, df, prec=p, max_iter=6)
    torch.cuda.synchronize()
    assert state["peak"] <= bqc.serve_footprint(basis.nbf, basis.naux, basis.nocc, p)
    df.close()
    basis.close()


@pytest.mark.parametrize("shadow", ["NONE", "F16"])
def test_peak_of_a_shard_build(tracked, shadow):
    """Rows [520, 700) of 825: integrals of 700 rows, two factors, the shard's B,
    and 4 MB for the plan; or what the finished handle holds, if that is more."""
    torch, bqc, ctx, state = tracked
    basis = bqc.Basis(ctx, workload.molecule_for("w11"))
    before = state["live"]
    state["peak"] = 0
    df = bqc.DF(ctx, basis, keep_fp32=getattr(bqc, "SHADOW_" + shadow), aux_range=(520, 700))
    solve = 8 * (700 * basis.npair + basis.naux ** 2 + 700 ** 2 + 180 * basis.npair)
    assert state["peak"] - before <= max(solve, df.device_bytes) + 4 * MB
    df.close()
    basis.close()
