"""The cluster LU at the edges of its shapes: rows around the sizes where the number of CTAs,
rows per thread or the single-CTA form change, and columns around inner blocks (8), panels and
column blocks. FP64: pivots identical to the oracle's and factors to 1e-10 (max norm); FP32: the
reconstruction error within 1.1 times the oracle's plus 1e-4 ||A||_2, as in the other parity
tests."""
import numpy as np
import pytest

import oracle as O
from gpu_helpers import oracle_for, rel_max, run_gpu
from paper_1310_7202_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("m,n,k,l", [
    (32, 33, 7, 8), (512, 40, 9, 17), (513, 511, 36, 37), (1025, 90, 44, 45),
    (2049, 160, 73, 109), (4097, 120, 72, 80), (8193, 60, 20, 26)])
def test_f64_edges(m, n, k, l):
    A = synth.lowrank_plus_noise(m, n, min(m, n), 1e-3, seed=m + l)
    g, o = run_gpu(A, k, l, 5, "f64"), oracle_for(A, k, l, 5, "f64")
    assert g["info"].tolist() == [0, -1, -1, 0]
    assert np.array_equal(g["P"], o["P"]) and np.array_equal(g["Q"], o["Q"])
    assert rel_max(g["L"], o["L"]) <= 1e-10 and rel_max(g["U"], o["U"]) <= 1e-10


@pytest.mark.parametrize("m,n,k,l", [
    (128, 129, 8, 9), (257, 256, 75, 77), (512, 513, 76, 153), (2048, 2049, 77, 84),
    (4096, 4097, 60, 76), (8192, 600, 81, 229), (8193, 300, 36, 73), (16385, 400, 130, 145)])
def test_f32_edges(m, n, k, l):
    A = synth.lowrank_plus_noise(m, n, min(m, n, 2 * l), 1e-3, seed=m + l, dtype=np.float32)
    g, o = run_gpu(A, k, l, 6, "f32"), oracle_for(A, k, l, 6, "f32")
    assert g["info"][0] == 0 and g["info"][3] == 0
    assert sorted(g["P"].tolist()) == list(range(m)) and sorted(g["Q"].tolist()) == list(range(n))
    A64 = A.astype(np.float64)
    fro, _ = O.reconstruct_error(A64, g["P"], g["Q"], g["L"], g["U"], spectral=False)
    fro_or, _ = O.reconstruct_error(A64, o["P"], o["Q"], o["L"], o["U"], spectral=False)
    assert fro <= 1.1 * fro_or + 1e-4 * O.spectral_norm(A64)


@pytest.mark.parametrize("m,n,k,l", [(16385, 60, 20, 26), (40, 16390, 20, 30)])
def test_f64_tallest_form(m, n, k, l):
    """Eight rows a thread with panels of 8 columns, for the LU of Y and for that of B^T."""
    A = synth.lowrank_plus_noise(m, n, min(m, n), 1e-3, seed=m + l)
    g, o = run_gpu(A, k, l, 5, "f64"), oracle_for(A, k, l, 5, "f64")
    assert g["info"].tolist() == [0, -1, -1, 0]
    assert np.array_equal(g["P"], o["P"]) and np.array_equal(g["Q"], o["Q"])
    assert rel_max(g["L"], o["L"]) <= 1e-10 and rel_max(g["U"], o["U"]) <= 1e-10
