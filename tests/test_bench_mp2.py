"""Roofline line of `bench.py --mp2`: a share of the rate of the unit that does
the work, for the kernels that run (FP64 as sliced tensor-core products)."""
import os
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
PK = {"bf16_tflops": 1942.0, "bf16_tflops_sustained": 1700.0}


# waters and measured seconds: the DFMA pipe (N = 50), split blocks on a DFMA
# transform (N = 75), both on the tensor cores (N = 250)
@pytest.mark.parametrize("waters,fp64,seconds,unit", [(2, True, 6e-4, "alu"), (3, False, 5.8e-4, "tensor"),
                                                      (10, True, 6.7e-3, "tensor"),
                                                      (10, False, 4e-3, "tensor")])
def test_mp2_roofline_is_a_share(waters, fp64, seconds, unit):
    sys.path.insert(0, ROOT)
    import bench
    n, naux, no = 25 * waters, 75 * waters, 5 * waters
    nv = n - no
    transform = 2.0 * naux * n * n * no + 2.0 * naux * n * no * nv
    pair = 1.0 * naux * (no * nv) ** 2
    r = bench.mp2_roofline(transform, pair, seconds, n, fp64, PK, "test")
    assert r["bound"] == unit
    assert 0 < r["frac"] < 1
    assert r["algorithmic_flop"] == transform + pair
    if unit == "tensor":
        assert r["frac"] < r["frac_issued"] < 1
        issued = (34 if n > 80 else 0) * transform + (34 if fp64 else 3) * pair
        assert r["issued_tensor_flop"] == issued
