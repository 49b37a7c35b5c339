"""The batch's kernels for k <= 64 at the edges of their tiles: buckets of k (16, 32, 48, 64),
4 x 4 blocks of the Gram, 64-row chunks, 256-row and 128-column blocks, LUs of 48 and 49
columns, and batches whose longest side passes 2048 (one staged column instead of four). Each problem is compared with
the single-problem path, which uses none of these kernels. Both round in FP32, so the error of
the batch's factors stays within 1.1 of the other's plus 1e-4 ||A||_2, the tolerance of the
batch's other tests; a wrong row, column or chunk leaves an error of the order of ||A||. GPU only."""
import numpy as np
import pytest
import torch

from paper_1310_7202_gb300 import rlu, synth
from tests.test_gpu_batched import _padded

pytestmark = pytest.mark.gpu

SHORT = [(64, 64, 1), (65, 64, 4), (127, 65, 15), (128, 127, 16), (129, 128, 17), (255, 129, 32),
         (256, 255, 33), (257, 130, 47), (511, 257, 48), (513, 300, 49), (700, 513, 63),
         (1025, 640, 64)]


@pytest.mark.parametrize("prec", ["f32", "mixed"])
@pytest.mark.parametrize("extra", [[], [(2048, 200, 21)], [(2051, 90, 40), (100, 90, 7)],
                                   [(2100, 2053, 64)],
                                   # LUs of 48 columns and of 49, launched apart
                                   [(600, 560, 38), (601, 550, 39), (300, 280, 48)]])
def test_edges_of_the_small_kernels(prec, extra):
    mats, probs = [], []
    for i, (m, n, k) in enumerate(SHORT + extra):
        sigma = np.exp(-np.arange(1, min(m, n) + 1) / k)
        mats.append(sigma[0])
        A = synth.prescribed_matrix(m, n, sigma, 300 + i, 400 + i, dtype=np.float32)
        probs.append({"A": _padded(A), "k": k, "l": min(k + 10, m, n), "seed": 50 + i})
    b = rlu.Batch(probs, prec)
    b.run()
    torch.cuda.synchronize()
    for p, s0, r, (m, n, k) in zip(probs, mats, b.outs, SHORT + extra):
        s = rlu.factor(p["A"], k, p["l"], p["seed"], prec)
        fro_s, _ = rlu.reconstruct_error(p["A"], s["P"], s["Q"], s["L"], s["U"])
        fro_b, _ = rlu.reconstruct_error(p["A"], r["P"], r["Q"], r["L"], r["U"])
        assert fro_b <= 1.1 * fro_s + 1e-4 * s0, (m, n, k, fro_b, fro_s)
        assert sorted(r["P"].tolist()) == list(range(m))
        assert sorted(r["Q"].tolist()) == list(range(n))
        U = r["U"][:, :n]
        assert torch.equal(U, torch.triu(U))
