"""||PAQ - LU|| in its exact-FP32 and FP64 forms: odd sizes, operands outside the FP32 form's
range, and values that no comparison with a range accepts."""
import numpy as np
import pytest
import torch

from paper_1310_7202_gb300 import rlu

pytestmark = pytest.mark.gpu


def case(m, n, k, dtype, scale, seed):
    rng = np.random.default_rng(seed)
    L = rng.standard_normal((m, k)).astype(np.float32)
    U = (rng.standard_normal((k, n)) * scale).astype(np.float32)
    A = (L.astype(np.float64) @ U.astype(np.float64)
         + 1e-3 * scale * rng.standard_normal((m, n))).astype(np.float32)
    At = torch.from_numpy(A).cuda().to(dtype)
    P, Q = rng.permutation(m).astype(np.int32), rng.permutation(n).astype(np.int32)
    Lt = torch.from_numpy(np.ascontiguousarray(L.T)).cuda().t()
    args = (At, torch.from_numpy(P).cuda(), torch.from_numpy(Q).cuda(), Lt, torch.from_numpy(U).cuda())
    R = At.double().cpu().numpy()[P][:, Q] - L.astype(np.float64) @ U.astype(np.float64)
    return args, R


# the FP32 form drops nothing above 2^-70 of a term; FP64 rounds k additions at 2^-53 of terms
# of order 4 sqrt(k) scale in residuals of order 1e-3 scale or more
@pytest.mark.parametrize("m,n,k,dtype,scale", [
    (1, 1, 1, torch.float32, 1.0), (65, 63, 17, torch.float32, 1.0), (513, 1030, 33, torch.float32, 1.0),
    (5003, 131, 16, torch.float32, 2.0 ** -10), (300, 257, 40, torch.bfloat16, 1.0),
    (200, 190, 20, torch.float32, 2.0 ** 60), (200, 190, 20, torch.float32, 2.0 ** -60)])
def test_norms(m, n, k, dtype, scale):
    args, R = case(m, n, k, dtype, scale, m + n)
    fro, spec = rlu.reconstruct_error(*args, power_iters=300)
    want = np.linalg.norm(R)
    assert abs(float(fro) - want) <= 1e-12 * want
    top = np.linalg.norm(R, 2)
    assert float(spec) <= top * (1 + 1e-12) and float(spec) >= 0.97 * top


@pytest.mark.parametrize("bad", [float("nan"), float("inf")])
def test_nonfinite_reaches_the_result(bad):
    args, _ = case(130, 70, 9, torch.float32, 1.0, 5)
    args[0][17, 33] = bad
    fro, _ = rlu.reconstruct_error(*args, power_iters=2)
    assert not np.isfinite(float(fro))


def test_zero():
    args, _ = case(40, 50, 3, torch.float32, 1.0, 6)
    for t in (args[0], args[3], args[4]):
        t.zero_()
    fro, spec = rlu.reconstruct_error(*args, power_iters=3)
    assert float(fro) == 0.0 and float(spec) == 0.0


# All of one sign, so that y = (PAQ - LU) x adds up: |y| reaches k 2^(2e) sqrt(n), and A y and its
# sums over a chunk of rows leave the FP32 range although A, L and U are far inside it. Tolerances
# as in test_norms; the residual is of the size of L U, so no cancellation loosens them.
@pytest.mark.parametrize("m,n,k,e", [(200, 190, 20, 40), (2000, 1500, 100, 38), (2000, 1500, 100, 36),
                                     (300, 257, 40, 28), (257, 300, 3, 39)])
def test_large_factors_of_one_sign(m, n, k, e):
    rng = np.random.default_rng(m + e)
    L, U, A = (np.ldexp(rng.uniform(0.5, 1.0, s), e).astype(np.float32) for s in ((m, k), (k, n), (m, n)))
    P, Q = rng.permutation(m).astype(np.int32), rng.permutation(n).astype(np.int32)
    Lt = torch.from_numpy(np.ascontiguousarray(L.T)).cuda().t()
    fro, spec = rlu.reconstruct_error(*(torch.from_numpy(x).cuda() for x in (A, P, Q)), Lt,
                                      torch.from_numpy(U).cuda(), power_iters=60)
    R = A.astype(np.float64)[P][:, Q] - L.astype(np.float64) @ U.astype(np.float64)
    want, top = np.linalg.norm(R), np.linalg.norm(R, 2)
    assert abs(float(fro) - want) <= 1e-12 * want
    assert top * 0.97 <= float(spec) <= top * (1 + 1e-12)


# up to one 64 x 64 tile an SM and 16 columns of L the FP64 form runs, without the scan of the
# operands' magnitudes; from there on the FP32 form
@pytest.mark.parametrize("m,n,k,launches", [(300, 257, 16, 2), (300, 257, 17, 3), (640, 576, 16, 2),
                                            (2000, 1200, 16, 3)])
def test_small_problems_take_no_scan(m, n, k, launches):
    args, R = case(m, n, k, torch.float32, 1.0, m + k)
    before = rlu.launch_count()
    fro, _ = rlu.reconstruct_error(*args)
    assert rlu.launch_count() - before == launches
    assert abs(float(fro) - np.linalg.norm(R)) <= 1e-12 * np.linalg.norm(R)
    _, spec = rlu.reconstruct_error(*args, power_iters=300)
    top = np.linalg.norm(R, 2)
    assert top * 0.97 <= float(spec) <= top * (1 + 1e-12)
