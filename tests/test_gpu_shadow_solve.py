"""What mixed Fock builds are made of keeps its last bits.

The stored tensor of a handle with split shadows is forward substitution's,
operation for operation: the shadows keep 22 bits of it, so a solve that is as
accurate but rounds elsewhere gives mixed Fock builds (and staged SCFs) another
result.

The substitution is restated on the host with each multiply-add rounded once:
the library's diagonal blocks of 64 rows subtract L_jl x_l from the row in the
order of l and divide by L_jj, and the rows below a block take away the sum of
its 64 products, accumulated from zero in the same order.  A multiply-add of
doubles is exact in the 113-bit long double of the GPU machine's host before its
one rounding; a long double of fewer bits cannot restate it."""
import numpy as np
import pytest

import workload

pytestmark = pytest.mark.gpu
NB = 64


def _fma(a, b, c):
    q = np.longdouble
    return (a.astype(q) * b.astype(q) + c.astype(q)).astype(np.float64)


def _substitute(L, R):
    X = R.copy()
    n = len(L)
    for k0 in range(0, n, NB):
        k1 = min(n, k0 + NB)
        acc = np.zeros((n - k1, R.shape[1]))
        for j in range(k0, k1):
            X[j] = X[j] / L[j, j]
            X[j + 1:k1] = _fma(-L[j + 1:k1, j, None], X[None, j], X[j + 1:k1])
            acc = _fma(L[k1:, j, None], X[None, j], acc)
        X[k1:] -= acc
    return X


# Naux = 150, 600 and 825 (a ragged last block), a shard of the last
@pytest.mark.parametrize("name,shadow,shard", [("w2", "TF32", None), ("w8", "F16", None),
                                               ("w11", "TF32", None), ("w11", "F16", (520, 700))])
def test_tensor_is_forward_substitution(gpu_ctx, name, shadow, shard):
    import paper_2502_17963_gb300 as bqc
    if np.finfo(np.longdouble).nmant < 106:
        pytest.skip("long double holds no exact product of doubles")
    basis = bqc.Basis(gpu_ctx, workload.molecule_for(name))
    df = bqc.DF(gpu_ctx, basis, keep_fp32=getattr(bqc, "SHADOW_" + shadow), aux_range=shard)
    cols = np.linspace(0, basis.npair - 1, 5).astype(int)
    L = df.copy(1).cpu().numpy()
    R = df.int3c_screened(0, basis.naux).cpu().numpy()[:, cols]
    p0, p1 = shard or (0, basis.naux)
    B = df.copy(0).cpu().numpy()[:, cols]
    assert np.array_equal(B, _substitute(L[:p1, :p1], R[:p1])[p0:p1])
