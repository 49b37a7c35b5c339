"""FP64 products at the edges of their tiles (sides around 16, 32, 48 and 64) and the split-K
reductions' ragged forms, through the factorizations that use them."""
import numpy as np
import pytest

import oracle as O
from gpu_helpers import oracle_for, rel_max, run_gpu
from paper_1310_7202_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("m,n,k,l", [
    (17, 40, 1, 3), (65, 300, 32, 33), (300, 130, 31, 48), (1001, 515, 33, 49), (260, 2049, 48, 64),
    (5000, 70, 49, 65), (130, 129, 100, 129)])
def test_f64_factors_match_oracle(m, n, k, l):
    A = synth.lowrank_plus_noise(m, n, min(m, n), 1e-2, seed=m + 3 * l)
    g, o = run_gpu(A, k, l, 9, "f64"), oracle_for(A, k, l, 9, "f64")
    assert np.array_equal(g["P"], o["P"]) and np.array_equal(g["Q"], o["Q"])
    assert rel_max(g["L"], o["L"]) <= 1e-10 and rel_max(g["U"], o["U"]) <= 1e-10


@pytest.mark.parametrize("m,n,k,l,prec", [(1001, 1200, 33, 41, "mixed"), (1003, 999, 47, 60, "f32"),
                                          (4099, 1024, 21, 30, "mixed")])
def test_ragged_reductions(m, n, k, l, prec):
    """Y = A G against FP64 on the same G: within FP32 rounding of the sums."""
    A = synth.lowrank_plus_noise(m, n, 2 * l, 1e-2, seed=m, dtype=np.float32)
    g = run_gpu(A, k, l, 4, prec)
    G = g["G"].astype(np.float32)
    if prec == "mixed":  # the tensor cores read G's upper 19 bits
        G = (np.ascontiguousarray(G).view(np.uint32) & np.uint32(0xFFFFE000)).view(np.float32)
    Y = A.astype(np.float64) @ G.astype(np.float64)
    bound = np.abs(A).astype(np.float64) @ np.abs(G).astype(np.float64)
    # n additions of relative 2^-24 at most, and the tensor cores' truncating ones at 2^-23
    assert np.all(np.abs(g["Y"] - Y) <= n * 2.0 ** -23 * bound)
