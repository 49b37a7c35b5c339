"""Algorithm 2 (the orthogonal-basis range finder, the comparator of the error experiment of
Section 5) on the GPU through rlu_rsvd, against the FP64 oracle's restatement (LAPACK SVD of
Y): the same G bit for bit, the singular values of Y, the subspace of Q, and the rank-k
error ||Q Q^T A - A||. GPU only."""
import numpy as np
import pytest
import torch

import oracle as O
from paper_1310_7202_gb300 import rlu, synth

pytestmark = pytest.mark.gpu


def _run(A, k, l, seed):
    At = torch.from_numpy(np.ascontiguousarray(A)).cuda()
    r = rlu.rsvd(At, k, l, seed)
    torch.cuda.synchronize()
    return At, {x: r[x].cpu().numpy() for x in ("Q", "B", "sigma", "info")}, r


@pytest.mark.parametrize("m,n,k,l,spec", [
    (500, 400, 20, 30, "paper_exp"),
    (600, 700, 37, 47, "inv_square"),     # odd l: a padding index in the eigensolver
    (300, 300, 1, 1, "paper_slow"),       # one vector
    (2000, 1500, 100, 110, "paper_slow"),
    (1200, 900, 250, 260, "paper_slow"),  # many rounds and sweeps
])
def test_rsvd_matches_the_oracle(m, n, k, l, spec):
    sigma = synth.spectrum(spec, min(m, n))
    A = synth.prescribed_matrix(m, n, sigma, 13, 14)
    At, g, _ = _run(A, k, l, 9)
    o = O.randomized_orth(A, k, l, seed=9)
    sy = o["sigma_y"]
    assert np.abs(g["sigma"] - sy).max() <= 1e-9 * sy[0]
    Q = g["Q"]
    assert np.abs(Q.T @ Q - np.eye(k)).max() <= 1e-10
    assert np.abs(g["B"] - Q.T @ A).max() <= 1e-11 * np.abs(A).max() * np.sqrt(m)
    fro_g, _ = O.orth_error(A, Q, g["B"], spectral=False)
    fro_o, _ = O.orth_error(A, o["Q"], spectral=False)
    assert abs(fro_g - fro_o) <= 1e-8 * fro_o, (fro_g, fro_o)
    # the subspaces agree where Y has a gap after its k-th singular value
    if k < l and sy[k] < 0.99 * sy[k - 1]:
        cosines = np.linalg.svd(o["Q"].T @ Q, compute_uv=False)
        assert cosines.min() >= 1 - 1e-8
    assert g["info"].tolist()[0] == 0


def test_rsvd_flags_singular_values_below_the_gram_resolution():
    """sigma_i = e^{-(i-1)/10} with k = 250: sigma_k(Y) / sigma_1(Y) ~ 1e-11, below what the
    eigenvalues of the FP64 Gram matrix resolve (about 1e-7): the unresolved singular values
    come back as 0, their columns of Q as zero, and the status says so; the resolved ones
    still match the oracle's SVD."""
    m, n, k, l = 1200, 900, 250, 260
    sigma = synth.spectrum("paper_exp", n)
    A = synth.prescribed_matrix(m, n, sigma, 13, 14)
    At, g, _ = _run(A, k, l, 9)
    sy = O.randomized_orth(A, k, l, seed=9)["sigma_y"]
    assert g["info"].tolist()[0] == rlu.RLU_EINVAL
    ok = sy > 1e-6 * sy[0]
    assert ok.sum() >= 100
    assert np.abs(g["sigma"][ok] - sy[ok]).max() <= 1e-9 * sy[0]
    assert np.all(g["sigma"][sy < 1e-9 * sy[0]] == 0)


def test_rsvd_exact_rank_and_device_error_measure():
    m, n, k, l = 400, 300, 12, 20
    A = synth.prescribed_matrix(m, n, synth.spectrum("rank_k", min(m, n), k), 3, 4)
    At, g, r = _run(A, k, l, 2)
    fro, _ = O.orth_error(A, g["Q"], g["B"], spectral=False)
    assert fro / np.linalg.norm(A) < 1e-12
    # ||Q B - A|| through the library's error measure with identity permutations
    ident_m = torch.arange(m, dtype=torch.int32, device="cuda")
    ident_n = torch.arange(n, dtype=torch.int32, device="cuda")
    fro_d, _ = rlu.reconstruct_error(At, ident_m, ident_n, r["Q"], r["B"])
    torch.cuda.synchronize()
    assert fro_d.item() / np.linalg.norm(A) < 1e-12


def test_rsvd_and_randomized_lu_on_the_papers_error_shape():
    """The error experiment of Section 5 (3000 x 3000, exponentially decaying singular
    values, l = k + 3): the randomized LU (FP64 path) and Algorithm 2 give errors of the
    same size (the paper: almost identical), both at or above sigma_{k+1}."""
    m = n = 3000
    sigma = synth.spectrum("paper_exp", n)
    A = synth.prescribed_matrix(m, n, sigma, 21, 22)
    At = torch.from_numpy(A).cuda()
    for k in (20, 60):
        r = rlu.rsvd(At, k, k + 3, 4)
        P, Q, L, U, _ = rlu.Factorizer(m, n, k, k + 3, "f64")(At, 4)
        ident_m = torch.arange(m, dtype=torch.int32, device="cuda")
        ident_n = torch.arange(n, dtype=torch.int32, device="cuda")
        _, e_svd = rlu.reconstruct_error(At, ident_m, ident_n, r["Q"], r["B"], power_iters=60)
        _, e_lu = rlu.reconstruct_error(At, P, Q, L, U, power_iters=60)
        torch.cuda.synchronize()
        assert e_svd.item() >= sigma[k] * (1 - 1e-3) and e_lu.item() >= sigma[k] * (1 - 1e-3)
        assert 1 / 3 <= e_lu.item() / e_svd.item() <= 3, (k, e_lu.item(), e_svd.item())


def test_rsvd_rejects_bad_arguments():
    lib = rlu.load_library()
    assert lib.rlu_rsvd_workspace_size(100, 80, 10, 90) == 0     # l > min(m, n)
    assert lib.rlu_rsvd_workspace_size(100, 80, 0, 5) == 0
    A = torch.zeros((64, 48), dtype=torch.float32, device="cuda")
    with pytest.raises(rlu.RluError):
        rlu.rsvd(A, 4, 6, 1)                                     # FP64 only


def test_rsvd_time_does_not_fall_with_l():
    """A problem with fewer vectors is no slower than one with more. The eigensolver's sweeps
    depend on the data (here one of about nine more or less) and its rounds are l - 1, so the
    smaller l gets 20% of slack, less where it is far below the larger."""
    A = torch.randn(600, 500, dtype=torch.float64, device="cuda",
                    generator=torch.Generator("cuda").manual_seed(3))
    ls = list(range(64, 137, 8))
    t = {}
    for l in ls:
        rlu.rsvd(A, l, l, 5)
        best = float("inf")
        for _ in range(4):
            e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            torch.cuda.synchronize()
            e0.record()
            rlu.rsvd(A, l, l, 5)
            e1.record()
            torch.cuda.synchronize()
            best = min(best, e0.elapsed_time(e1))
        t[l] = best
    slow = [(a, b) for a in ls for b in ls if a < b and t[a] > 1.2 * t[b]]
    assert not slow, t


@pytest.mark.parametrize("l", [1, 2, 3, 63, 64, 65, 66, 79, 80, 81, 82, 95, 96, 97, 111, 112, 113])
def test_rsvd_around_the_eigensolvers_sizes(l):
    """One index, one pair, and the sizes around multiples of 16 where the number of CTAs of the
    eigensolver or its form may change; tolerances of test_rsvd_matches_the_oracle."""
    m, n = 300, 260
    A = synth.prescribed_matrix(m, n, synth.spectrum("paper_slow", n), 13, 14)
    k = max(1, l - 3)
    _, g, _ = _run(A, k, l, 9)
    sy = O.randomized_orth(A, k, l, seed=9)["sigma_y"]
    assert g["info"].tolist()[0] == 0
    assert np.abs(g["sigma"] - sy).max() <= 1e-9 * sy[0]
    assert np.abs(g["Q"].T @ g["Q"] - np.eye(k)).max() <= 1e-10


@pytest.mark.parametrize("e", [-250, 250])
@pytest.mark.parametrize("l", [30, 121])
def test_rsvd_far_from_one(l, e):
    """A scaled by 2^e, so that products of two entries of the Gram matrix leave the FP64 range:
    the factors scale along (a power of two rounds nothing)."""
    m, n = 300, 260
    A = synth.prescribed_matrix(m, n, synth.spectrum("paper_slow", n), 13, 14)
    _, one, _ = _run(A, l, l, 9)
    _, g, _ = _run(np.ldexp(A, e), l, l, 9)
    assert g["info"].tolist()[0] == 0
    want = np.ldexp(one["sigma"], e)
    assert np.abs(g["sigma"] - want).max() <= 1e-9 * want[0]
    assert np.abs(g["Q"].T @ g["Q"] - np.eye(l)).max() <= 1e-10
