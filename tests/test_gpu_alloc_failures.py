"""A device allocation that fails in the middle of a call: the call returns
BQC_E_OOM (or does without the memory), what it gives back is not in use by work
still running on its stream, and the same call succeeds afterwards with the same
result."""
import ctypes

import pytest

import workload

pytestmark = pytest.mark.gpu


class FailingAllocator:
    """Allocation callbacks over torch's caching allocator: allocation number
    `fail_at` (from arm()) fails; `busy` counts releases before the stream is idle."""

    def __init__(self, bqc, torch, stream):
        self.fail_at, self.seen, self.busy, self.live = None, 0, 0, set()

        def alloc(nbytes, _):
            self.seen += 1
            if self.fail_at is not None and self.seen == self.fail_at:
                return None
            p = torch.cuda.caching_allocator_alloc(int(nbytes), 0, stream)
            self.live.add(p)
            return p

        def free(ptr, _):
            if self.fail_at is not None and not stream.query():
                self.busy += 1
            self.live.discard(ptr)
            torch.cuda.caching_allocator_delete(ptr)

        self.fns = bqc.ALLOC_FN(alloc), bqc.FREE_FN(free)

    def arm(self, fail_at):
        self.fail_at, self.seen, self.busy = fail_at, 0, 0


@pytest.fixture(scope="module")
def setup():
    import torch
    import paper_2502_17963_gb300 as bqc
    from paper_2502_17963_gb300 import _build
    _build.build()
    stream = torch.cuda.Stream()
    mem = FailingAllocator(bqc, torch, stream)
    ctx = bqc.Context.__new__(bqc.Context)
    ctx.device, ctx.h = 0, ctypes.c_void_p()
    ctx._afn, ctx._ffn = mem.fns
    bqc.check(bqc.lib().bqc_ctx_create(0, 0, ctx._afn, ctx._ffn, None, ctypes.byref(ctx.h)),
              "bqc_ctx_create")
    basis = bqc.Basis(ctx, workload.molecule_for("w3"))
    yield torch, bqc, mem, ctx, basis, stream
    basis.close()
    ctx.close()


def _each(mem, bqc, call, same):
    """call() with every one of its allocations failing in turn."""
    mem.arm(None)
    ref = call()
    count = mem.seen
    assert count > 0
    for k in range(1, count + 1):
        live = len(mem.live)
        mem.arm(k)
        try:
            got = call()
        except bqc.BqcError as e:
            assert e.status == -2, e
            assert len(mem.live) == live  # nothing of the failed call is kept
        else:
            assert same(got, ref)
        assert mem.busy == 0, (k, mem.busy)
    mem.arm(None)
    assert same(call(), ref)


@pytest.mark.parametrize("mode,shadow,shard", [(0, "NONE", None), (0, "F16", None), (0, "TF32", None),
                                               (0, "NONE", (40, 180)), (1, "TF32", None),
                                               (3, "NONE", None)])
def test_build(setup, mode, shadow, shard):
    torch, bqc, mem, ctx, basis, stream = setup

    def call():
        with torch.cuda.stream(stream):
            df = bqc.DF(ctx, basis, mode=mode, keep_fp32=getattr(bqc, "SHADOW_" + shadow),
                        stream=stream, aux_range=shard)
            try:
                return df.copy(0, stream) if mode == 0 else torch.zeros(1, device="cuda")
            finally:
                stream.synchronize()
                df.close()

    # without room for its slices a solve takes another route: equal to rounding
    _each(mem, bqc, call, lambda a, b: bool((a - b).abs().max() <= 1e-11 * b.abs().max()))


def test_int3c(setup):
    torch, bqc, mem, ctx, basis, stream = setup

    def call():
        with torch.cuda.stream(stream):
            out = bqc.int3c(basis, 1e-12, stream)
            stream.synchronize()
        return out

    _each(mem, bqc, call, torch.equal)


@pytest.mark.parametrize("prec", ["FP64", "MIXED_F16X3"])
def test_scf_and_mp2(setup, prec):
    torch, bqc, mem, ctx, basis, stream = setup
    p = getattr(bqc, "PREC_" + prec)
    with torch.cuda.stream(stream):
        df = bqc.DF(ctx, basis, keep_fp32=bqc.SHADOW_F16, stream=stream)
        r = bqc.scf_run(ctx, df, stream=stream, keep_arrays=True)
        C, eps = r["C"].contiguous(), r["eps"].contiguous()
        stream.synchronize()
    try:
        _each(mem, bqc, lambda: bqc.scf_run(ctx, df, prec=p, stream=stream)["energy"],
              lambda a, b: abs(a - b) <= 1e-8)
        _each(mem, bqc, lambda: bqc.mp2(df, C, eps, p, stream=stream),
              lambda a, b: abs(a - b) <= 1e-9)
    finally:
        df.close()
