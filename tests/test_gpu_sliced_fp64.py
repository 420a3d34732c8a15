"""FP64 products assembled from exact FP16 slices (csrc/oz.cu), through the
entry points that use them: the FP64 Fock build, the metric solve of a stored
handle and the MP2 energy.

Bounds.  An operand element is kept to 2^-56 of a power-of-two bound of its row
(at most twice the row's largest element m_a), products of digits from level 8
on are dropped: each term of a product of rows a and b is off by at most about
2^-53 m_a m_b.  X = B C therefore carries N 2^-53 m_B m_C, and K, a product of
X with itself over Naux nocc terms, 2^-52 of the row bounds a term plus the
error of X; the plain FP64 evaluation on the other side rounds at 2^-53 of
its partial sums.  A factor 16 covers both.
"""
import numpy as np
import pytest

import workload

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def bqc():
    import paper_2502_17963_gb300 as m
    return m


def _full(torch, Bp, n):
    r, c = torch.tril_indices(n, n, device="cuda")
    B = torch.zeros((Bp.shape[0], n, n), dtype=torch.float64, device="cuda")
    B[:, r, c] = Bp
    B[:, c, r] = Bp
    return B


# N = 75 (one ragged 128-row tile), 125, 150, 275 (row and column tails), 200
# with orbitals whose columns span twelve orders of magnitude
@pytest.mark.parametrize("name,spread", [("w3", 0), ("w5", 0), ("w6", 0), ("w8", 6), ("w11", 0)])
def test_fp64_fock_build(gpu_ctx, bqc, name, spread):
    import torch
    basis = bqc.Basis(gpu_ctx, workload.molecule_for(name))
    df = bqc.DF(gpu_ctx, basis, keep_fp32=False)
    n, no, naux = basis.nbf, basis.nocc, basis.naux
    B = _full(torch, df.copy(0), n)
    rng = np.random.default_rng(n)
    C = rng.standard_normal((n, no)) * 10.0 ** rng.uniform(-spread, spread, (1, no))
    C = torch.tensor(C, device="cuda")
    J, K = df.jk(C, bqc.PREC_FP64)
    X = B @ C
    w = (X * C).sum((1, 2))
    Kr = torch.einsum("pmi,pni->mn", X, X)
    Jr = torch.einsum("p,pmn->mn", w, B)
    eps = 2.0 ** -53
    mx = X.abs().amax((0, 2))  # by row of K
    ex = n * eps * B.abs().max() * C.abs().amax(0)  # error of X by column
    kb = naux * no * eps * mx[:, None] * mx[None] + naux * mx.max() * ex.sum()
    assert ((K - Kr).abs() <= 16 * kb).all()
    wa = (B.abs() @ C.abs() * C.abs()).sum((1, 2))  # absolute contraction
    ja = torch.einsum("p,pmn->mn", wa, B.abs())
    jb = n * eps * ja + naux * n * (ex * C.abs().amax(0)).sum() * B.abs().max()
    assert ((J - Jr).abs() <= 16 * jb).all()
    assert torch.equal(K, K.T) and torch.equal(J, J.T)


def test_fp64_fock_build_many_occupied(gpu_ctx, bqc):
    """As many occupied orbitals as functions (twelve argon atoms in three s
    and two p shells each, N = nocc = 108): the small build's B_P, C and X_P do
    not fit in shared memory together, and the sliced products take over."""
    import torch
    from types import SimpleNamespace as NS
    k = np.arange(12)
    xyz = 6.0 * np.stack([k % 3, k // 3 % 2, k // 6], axis=1).astype(float)

    def shells(rules):
        return [NS(atom=a, l=l, exps=[e], coefs=[1.0]) for a in range(12) for l, e in rules]

    mol = NS(Z=np.full(12, 18, dtype=np.int32), xyz=xyz,
             orb=shells([(0, 0.3), (0, 1.0), (0, 3.0), (1, 0.4), (1, 1.2)]),
             aux=shells([(0, 0.8), (0, 2.5), (1, 1.0), (2, 1.1)]))
    basis = bqc.Basis(gpu_ctx, mol)
    n, no = basis.nbf, basis.nocc
    assert n == no == 108
    df = bqc.DF(gpu_ctx, basis, keep_fp32=False)
    B = _full(torch, df.copy(0), n)
    rng = np.random.default_rng(3)
    C = torch.tensor(rng.standard_normal((n, no)) / np.sqrt(n), device="cuda")
    J, K = df.jk(C, bqc.PREC_FP64)
    X = B @ C
    Kr = torch.einsum("pmi,pni->mn", X, X)
    Jr = torch.einsum("p,pmn->mn", (X * C).sum((1, 2)), B)
    # N Naux nocc terms of 2^-53 of the largest products, as above
    eps = 16 * 2.0 ** -53
    assert (K - Kr).abs().max() <= eps * basis.naux * no * n * X.abs().max() ** 2
    assert (J - Jr).abs().max() <= eps * basis.naux * no * n * (X.abs().max() * B.abs().max())


def test_fp64_fock_build_nan(gpu_ctx, bqc):
    """A NaN or an infinity in one orbital reaches every element of J and K."""
    import torch
    basis = bqc.Basis(gpu_ctx, workload.molecule_for("w3"))
    df = bqc.DF(gpu_ctx, basis, keep_fp32=False)
    C = torch.randn((basis.nbf, basis.nocc), dtype=torch.float64, device="cuda")
    for bad in (float("nan"), float("inf")):
        Cb = C.clone()
        Cb[7, 3] = bad
        J, K = df.jk(Cb, bqc.PREC_FP64)
        assert not torch.isfinite(J).any() and not torch.isfinite(K).any()
    J, K = df.jk(torch.zeros_like(C), bqc.PREC_FP64)
    assert (J == 0).all() and (K == 0).all()
    J, K = df.jk(C, bqc.PREC_FP64)
    assert torch.isfinite(J).all() and torch.isfinite(K).all()


# Naux = 92 (two blocks, the second ragged), 150, 450, 825 (uneven halving)
@pytest.mark.parametrize("name", ["h2o", "w2", "w6", "w11"])
def test_metric_solve(gpu_ctx, bqc, name):
    """L B equals the raw integrals: the residual of the solve, against
    Naux 2^-50 of the absolute products |L||B| (forward substitution gives
    Naux 2^-53; the diagonal blocks' inverses add their condition, about
    10, for these metrics)."""
    import torch
    basis = bqc.Basis(gpu_ctx, workload.molecule_for(name))
    df = bqc.DF(gpu_ctx, basis, keep_fp32=False)
    B, L = df.copy(0), df.copy(1)
    raw = df.int3c_screened(0, basis.naux)
    bound = basis.naux * 2.0 ** -50 * (L.abs() @ B.abs()).amax()
    assert (L @ B - raw).abs().max() <= bound


# n = 50, 150 (plain small products), 275 and 325 (sliced ones)
@pytest.mark.parametrize("name", ["w2", "w6", "w11", "w13"])
def test_scf_orbitals(gpu_ctx, bqc, name):
    """The SCF's orbitals (refined from an FP32 decomposition): C^T S C = 1,
    with C = X U, to n 2^-50 of |X|^2 |S| (the products' rounding and the
    refinement's, 2^-53 of the same terms each); ascending energies."""
    import torch
    basis = bqc.Basis(gpu_ctx, workload.molecule_for(name))
    df = bqc.DF(gpu_ctx, basis, keep_fp32=bqc.SHADOW_F16)
    r = bqc.scf_run(gpu_ctx, df, prec=bqc.PREC_MIXED_F16X3, keep_arrays=True)
    assert r["converged"]
    S = bqc.one_electron(basis)[0]
    C = torch.as_tensor(r["C"], device="cuda")
    eps = torch.as_tensor(r["eps"], device="cuda")
    n = basis.nbf
    bound = n * 2.0 ** -50 * (C.abs().T @ S.abs() @ C.abs()).max()
    assert (C.T @ S @ C - torch.eye(C.shape[1], device="cuda", dtype=C.dtype)).abs().max() <= bound
    assert (eps[1:] >= eps[:-1]).all()
