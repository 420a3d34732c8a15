"""Eigen-decomposition of the SCF's FP64 stage (csrc/eigh.cu): FP32 vectors
refined to FP64, on spectra with pairs of close levels (what symmetric or weakly
coupled fragments give a Fock matrix).

Bounds, with eps = 2^-53 and t the largest eigenvalue: V^T V - 1 is left by the
last orthonormalisation at the rounding of two products of n terms of unit
vectors, sqrt(n) eps each for terms of mixed sign; 16 sqrt(n) eps.  A V - V w and
w carry the rounding of products with |A| <= t, of the accepted off-diagonals
(n 1e-15 t at most), and of the test's own evaluation: 64 n eps t."""
import math

import pytest

pytestmark = pytest.mark.gpu

EPS = 2.0 ** -53


def _matrix(torch, n, gap, pairs, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    w = torch.sort(torch.rand(n, generator=g, device="cuda", dtype=torch.float64) * 62 - 2)[0]
    for p in range(pairs):  # a core-like pair each, gap apart
        w[2 * p] = -20.5 - 0.3 * p
        w[2 * p + 1] = -20.5 - 0.3 * p + gap
    q = torch.linalg.qr(torch.randn((n, n), generator=g, device="cuda", dtype=torch.float64))[0]
    a = (q * w) @ q.T
    return 0.5 * (a + a.T)


def _check(torch, ctx, bqc, A):
    n = len(A)
    w, V, refined = bqc.eigh(ctx, A)
    top = float(torch.linalg.eigvalsh(A).abs().max())
    one = torch.eye(n, device="cuda", dtype=torch.float64)
    assert (V.T @ V - one).abs().max() <= 16 * math.sqrt(n) * EPS
    assert (A @ V - V * w).abs().max() <= 64 * n * EPS * top
    assert (w - torch.linalg.eigvalsh(A)).abs().max() <= 64 * n * EPS * top
    assert (w[1:] >= w[:-1] - 64 * n * EPS * top).all()
    return refined


# orders: the smallest, odd, ragged tiles, sliced products (256 and up), the largest refined
@pytest.mark.parametrize("n", [2, 9, 75, 150, 257, 320])
@pytest.mark.parametrize("gap", [0.0, 1e-13, 1e-12, 1e-11, 6.2e-11, 1e-10, 1e-9, 1e-8, 1e-6, 1e-3])
def test_close_pairs(gpu_ctx, n, gap):
    import torch
    import paper_2502_17963_gb300 as bqc
    A = _matrix(torch, n, gap, 1 if n < 9 else 4, n)
    assert _check(torch, gpu_ctx, bqc, A)


def test_where_the_refinement_does_not_apply(gpu_ctx):
    """A level of more than eight functions, and an order above the refined ones:
    the FP64 decomposition serves."""
    import torch
    import paper_2502_17963_gb300 as bqc
    g = torch.Generator(device="cuda").manual_seed(5)
    q = torch.linalg.qr(torch.randn((60, 60), generator=g, device="cuda", dtype=torch.float64))[0]
    w = torch.arange(60, device="cuda", dtype=torch.float64)
    w[20:32] = 20.0
    A = (q * w) @ q.T
    assert not _check(torch, gpu_ctx, bqc, 0.5 * (A + A.T))
    assert not _check(torch, gpu_ctx, bqc, _matrix(torch, 330, 1e-9, 2, 1))


def test_scf_of_two_distant_fragments(gpu_ctx):
    """Two waters 18 Angstrom apart, one bent by a hair: core levels split by far
    less than FP32 resolves.  C^T S C = 1 to n 2^-50 of |X|^2 |S| (the products'
    rounding, 2^-53 of the same terms each)."""
    import torch
    import numpy as np
    from types import SimpleNamespace as NS
    import paper_2502_17963_gb300 as bqc
    import workload
    one = workload.single_water()
    shift = np.array([34.0, 0.0, 0.0])
    for bend in (0.0, 1e-9, 1e-7):
        second = one.xyz.copy()
        second[1, 2] += bend
        nat = len(one.Z)
        mol = NS(Z=np.concatenate([one.Z, one.Z]), xyz=np.concatenate([one.xyz, second + shift]),
                 orb=[NS(atom=s.atom + k * nat, l=s.l, exps=s.exps, coefs=s.coefs)
                      for k in range(2) for s in one.orb],
                 aux=[NS(atom=s.atom + k * nat, l=s.l, exps=s.exps, coefs=s.coefs)
                      for k in range(2) for s in one.aux])
        basis = bqc.Basis(gpu_ctx, mol)
        df = bqc.DF(gpu_ctx, basis, keep_fp32=False)
        r = bqc.scf_run(gpu_ctx, df, keep_arrays=True)
        assert r["converged"]
        S = bqc.one_electron(basis)[0]
        C, n = r["C"], basis.nbf
        bound = n * 2.0 ** -50 * (C.abs().T @ S.abs() @ C.abs()).max()
        unit = torch.eye(C.shape[1], device="cuda", dtype=C.dtype)
        assert (C.T @ S @ C - unit).abs().max() <= bound
