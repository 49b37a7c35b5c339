"""The calls that users of the randomized LU library make, as timed cases.

Every case goes through the Python binding (paper_1310_7202_gb300.rlu) the way a program
does: the plan (a Factorizer, Batch, FastFactorizer or Server) is made once for a size, the
matrix is on the GPU, and one pass is one call. Kinds:

  factor    Algorithm 1 on one matrix, any precision, with or without power iterations
  batch     Algorithm 1 on many small problems of uneven sizes at once
  serve     a burst of requests of mixed sizes and precisions through the serving loop
  fast      Algorithm 4 (the SRFT form, complex factors)
  lstsq     Algorithm 3 on the factors of a matrix
  residual  ||PAQ - LU|| in both norms, the check of a factorization
  rsvd      Algorithm 2, which the paper compares against

Matrices are low rank plus noise: A = X diag(exp(-i/k)) W^T / sqrt(r) + 1e-3 E with Gaussian
X, W and E and r = min(m, n, 4k), the exp(-i/k) decay of the batched workload without its QR.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_1310_7202_gb300 import rlu

_DTYPE = {"f64": torch.float64, "f32": torch.float32, "mixed": torch.float32,
          "bf16": torch.bfloat16}


def _factor(name, prec, m, n, k, l, q=0, normalized=False):
    return {"name": name, "kind": "factor", "prec": prec, "m": m, "n": n, "k": k, "l": l, "q": q,
            "normalized": normalized}


def listed():
    return [
        # the smallest whole call: the FP64 parity workload of the benchmark, where launches
        # and the pivot chain are everything
        _factor("f64_512", "f64", 512, 512, 20, 25),
        # an everyday tall matrix in the plain single precision; sizes that divide nothing
        _factor("f32_3001x1203", "f32", 3001, 1203, 61, 71),
        # a mid-size wide matrix on the mixed path, ragged against every tile
        _factor("mixed_2900x5196", "mixed", 2900, 5196, 127, 137),
        # the benchmark's headline workload: 8192 x 8192, k = 200, l = 210
        _factor("mixed_8192", "mixed", 8192, 8192, 200, 210),
        # the precision workload, the largest call: a 1 GB matrix in BF16
        _factor("bf16_32768x16384", "bf16", 32768, 16384, 512, 532),
        # one LU-normalised power iteration, the option for slowly decaying spectra
        _factor("power_6000x4000", "mixed", 6000, 4000, 100, 110, 1, True),
        # the batched form: 512 problems drawn as the batched workload draws them
        {"name": "batch_512", "kind": "batch", "prec": "mixed", "count": 512, "shapes": 4},
        # the served form: a burst of 12 requests, sizes and classes as the serving workload
        # draws them, 8 in flight
        {"name": "serve_12", "kind": "serve", "count": 12, "shapes": 7, "largest": 16384},
        # the fast randomized LU at the paper's timing shape, l = 3 log2(n)^2
        {"name": "fast_4096", "kind": "fast", "m": 4096, "n": 4096, "k": 256, "l": 432},
        # least squares with a few right-hand sides on the headline workload's factors
        {"name": "lstsq_8192", "kind": "lstsq", "dtype": "f32", "m": 8192, "n": 8192, "k": 200,
         "nrhs": 16},
        # the error of the headline workload's factors, as the benchmark reports it
        {"name": "residual_8192", "kind": "residual", "dtype": "f32", "m": 8192, "n": 8192,
         "k": 200, "iters": 100},
        # the comparison method at the size of the paper's error experiment
        {"name": "rsvd_3000", "kind": "rsvd", "m": 3000, "n": 3000, "k": 40, "l": 43},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["factor"] * 6 + ["batch", "serve", "fast", "lstsq", "residual", "rsvd"])
    if kind == "factor":
        prec = rng.choice(["f64", "f32", "mixed", "mixed", "bf16", "bf16"])
        top = {"f64": 2048, "f32": 8192, "mixed": 16384, "bf16": 16384}[prec]
        m, n = _log_int(rng, 256, top), _log_int(rng, 256, top)
        if prec == "bf16":
            n = (n + 7) // 8 * 8  # its rows start on 16-byte boundaries
        elif prec == "mixed" and rng.random() < 0.75:
            n = (n + 3) // 4 * 4  # likewise, where the caller can; else its other route
        kmax = min(m, n) - 10
        k = min(kmax, rng.randint(16, 64 if prec == "f64" else 256))
        q = 1 if prec != "f64" and max(m, n) <= 8192 and rng.random() < 0.2 else 0
        c = _factor("", prec, m, n, k, k + 10, q, q == 1 and rng.random() < 0.7)
    elif kind == "batch":
        c = {"kind": "batch", "prec": rng.choice(["mixed", "mixed", "f32"]),
             "count": _log_int(rng, 24, 700), "shapes": rng.randrange(1 << 20)}
    elif kind == "serve":
        c = {"kind": "serve", "count": rng.randint(3, 12), "shapes": rng.randrange(1 << 20),
             "largest": _log_int(rng, 1024, 16384)}
    elif kind == "fast":
        n = rng.choice([512, 600, 1000, 1024, 1536, 2048, 3000, 4096])
        m = _log_int(rng, 512, 4096)
        l = min(m, n, rng.randint(40, 432))
        c = {"kind": "fast", "m": m, "n": n, "k": min(256, rng.randint(l // 2, l - 4)), "l": l}
    elif kind == "lstsq":
        k = rng.randint(16, 256)
        c = {"kind": "lstsq", "dtype": rng.choice(["f32", "f32", "f64"]),
             "m": _log_int(rng, 512, 16384), "n": _log_int(rng, 512, 16384), "k": k,
             "nrhs": rng.choice([1, 1, 3, 16])}
    elif kind == "residual":
        dtype = rng.choice(["f32", "f32", "bf16", "f64"])
        top = 4096 if dtype == "f64" else 8192
        c = {"kind": "residual", "dtype": dtype, "m": _log_int(rng, 256, top),
             "n": _log_int(rng, 256, top), "k": rng.randint(16, 200),
             "iters": rng.choice([0, 60, 100])}
    else:
        k = rng.choice([10, 20, 40])
        c = {"kind": "rsvd", "m": _log_int(rng, 300, 3000), "n": _log_int(rng, 300, 3000), "k": k,
             "l": k + 3}
    c.pop("name", None)
    return c


# ---- inputs ---------------------------------------------------------------------------------


def _device():
    return "cuda" if torch.cuda.is_available() else "cpu"


def _generator(seed):
    g = torch.Generator(device=_device())
    g.manual_seed(seed)
    return g


def _matrix(m, n, k, dtype, g):
    work = torch.float64 if dtype == torch.float64 else torch.float32
    r = min(m, n, 4 * k)
    X = torch.randn(m, r, generator=g, device=_device(), dtype=work)
    W = torch.randn(n, r, generator=g, device=_device(), dtype=work)
    decay = torch.exp(-torch.arange(1, r + 1, device=_device(), dtype=work) / k) / math.sqrt(r)
    A = torch.randn(m, n, generator=g, device=_device(), dtype=work).mul_(1e-3)
    A.addmm_(X * decay, W.t())
    return A.to(dtype).contiguous()


def _log_uniform(rng, lo, hi):
    return int(math.exp(rng.uniform(math.log(lo), math.log(hi))))


def _batch_shapes(case):
    """m log-uniform in [64, 2048], n log-uniform in [64, 1024] and at most m, k uniform in
    8..64, l = k + 10."""
    rng = np.random.default_rng(case["shapes"])
    out = []
    for _ in range(case["count"]):
        m = _log_uniform(rng, 64, 2048)
        n = min(_log_uniform(rng, 64, 1024), m)
        k = int(rng.integers(8, min(64, n - 10) + 1))
        out.append((m, n, k, k + 10))
    return out


def _serve_shapes(case):
    """m, n log-uniform in [256, largest], k uniform in 16..256, l = k + 10; half the requests
    in each accuracy class."""
    rng = np.random.default_rng(case["shapes"])
    out = []
    for _ in range(case["count"]):
        m, n = _log_uniform(rng, 256, case["largest"]), _log_uniform(rng, 256, case["largest"])
        k = int(rng.integers(16, min(256, min(m, n) - 10) + 1))
        out.append((m, n, k, k + 10, "bf16" if rng.random() < 0.5 else "mixed"))
    return out


def _srft_params(case, seed):
    rng = np.random.default_rng(seed)
    theta = torch.from_numpy(rng.random(case["n"], dtype=np.float32))
    s = torch.from_numpy(rng.permutation(case["n"])[:case["l"]].astype(np.int32))
    return theta.to(_device()), s.to(_device())


def _pivoted_lu(Y):
    """(perm, unit lower, upper) of a tall Y, FP64 or complex128, by LAPACK."""
    lu, piv = torch.linalg.lu_factor(Y.cpu())
    m, c = Y.shape
    perm = np.arange(m)
    for j, p in enumerate(piv.numpy() - 1):
        perm[[j, p]] = perm[[p, j]]
    lo = torch.tril(lu, -1)
    lo[torch.arange(c), torch.arange(c)] = 1
    return torch.from_numpy(perm), lo, torch.triu(lu[:c])


def _column_pivoted_lu(B):
    """(perm, L_b, U_b, the LU of B^T) of a wide B: that LU with the scaling moved to L_b's
    side."""
    perm, lo, up = _pivoted_lu(B.t())
    d = torch.diagonal(up)
    return perm, up.t() / d, d[:, None] * lo.t(), (lo, up)


def _factors(case, seed, dtype):
    """P, Q, L, U laid out as the library returns them, from LUs of Gaussian matrices."""
    g = _generator(seed)
    m, n, k = case["m"], case["n"], case["k"]
    kw = dict(generator=g, device=_device(), dtype=torch.float64)
    P, Ly, _ = _pivoted_lu(torch.randn(m, k, **kw))
    Q, Lb, U, _ = _column_pivoted_lu(torch.randn(k, n, **kw))
    dev = _device()
    L = (Ly @ Lb).to(dtype).t().contiguous().to(dev).t()
    return (P.to(torch.int32).to(dev), Q.to(torch.int32).to(dev), L,
            U.to(dtype).contiguous().to(dev), g)


def _lstsq_inputs(case, seed):
    dtype = _DTYPE[case["dtype"]]
    P, Q, L, U, g = _factors(case, seed, dtype)
    b = torch.randn(case["nrhs"], case["m"], generator=g, device=_device(), dtype=dtype).t()
    return P, Q, L, U, b[:, 0].contiguous() if case["nrhs"] == 1 else b


def _residual_inputs(case, seed):
    """A = P^T (L U + 1e-3 E) Q^T: the factors of A up to a residual of the noise's size."""
    adt = _DTYPE[case["dtype"]]
    P, Q, L, U, g = _factors(case, seed, torch.float64 if case["dtype"] == "f64" else
                             torch.float32)
    m, n = case["m"], case["n"]
    R = torch.randn(m, n, generator=g, device=_device(), dtype=L.dtype).mul_(1e-3)
    R.addmm_(L, U)
    A = torch.empty_like(R)
    A[P.long()[:, None], Q.long()[None, :]] = R
    return A.to(adt).contiguous(), P, Q, L, U


def _philox_seed(seed):
    return (seed * 2654435761 + 12345) % (1 << 48)


def prepare(case, seed):
    kind = case["kind"]
    g = _generator(seed)
    st = {"kind": kind, "seed": _philox_seed(seed)}
    if kind == "factor":
        st["A"] = _matrix(case["m"], case["n"], case["k"], _DTYPE[case["prec"]], g)
        st["plan"] = rlu.Factorizer(case["m"], case["n"], case["k"], case["l"], case["prec"],
                                    case["q"], case["normalized"])
    elif kind == "batch":
        problems = []
        for i, (m, n, k, l) in enumerate(_batch_shapes(case)):
            # rows padded to 16 bytes, which the mixed form asks for
            A = torch.empty(m, (n + 3) // 4 * 4, device="cuda")[:, :n]
            A.copy_(_matrix(m, n, k, torch.float32, g))
            problems.append({"A": A, "k": k, "l": l, "seed": st["seed"] + i})
        st["plan"] = rlu.Batch(problems, case["prec"])
        outs = st["plan"].outs
        st["flat"] = {x: [(o[x].t() if x == "L" else o[x]).reshape(-1) for o in outs]
                      for x in ("P", "Q", "L", "U", "info")}
    elif kind == "serve":
        shapes = _serve_shapes(case)
        big = max(max(s[:2]) for s in shapes)
        A = _matrix(big, (big + 7) // 8 * 8, 128, torch.float32, g)
        st["A"] = {"mixed": A, "bf16": A.to(torch.bfloat16)}
        st["requests"] = shapes
        st["plan"] = rlu.Server(budget_bytes=24 << 30, max_inflight=8)
    elif kind == "fast":
        st["A"] = _matrix(case["m"], case["n"], case["k"], torch.float32, g)
        st["theta"], st["s"] = _srft_params(case, seed)
        st["plan"] = rlu.FastFactorizer(case["m"], case["n"], case["k"], case["l"])
    elif kind == "lstsq":
        st["args"] = _lstsq_inputs(case, seed)
    elif kind == "residual":
        st["args"], st["iters"] = _residual_inputs(case, seed), case["iters"]
    else:
        st["A"] = _matrix(case["m"], case["n"], case["k"], torch.float64, g)
        st["k"], st["l"] = case["k"], case["l"]
    return st


# ---- one pass -------------------------------------------------------------------------------


def run(st):
    kind = st["kind"]
    if kind == "factor":
        P, Q, L, U, info = st["plan"](st["A"], st["seed"])
        return {"P": P, "Q": Q, "L": L, "U": U, "info": info}
    if kind == "batch":
        st["plan"].run()  # and the factors packed, as a program ships them off
        return {x: torch.cat(v) for x, v in st["flat"].items()}
    if kind == "serve":
        srv = st["plan"]
        ids = [srv.submit(st["A"][prec], k, l, st["seed"] + i, prec, m=m, n=n)
               for i, (m, n, k, l, prec) in enumerate(st["requests"])]
        srv.wait_all()
        out = []
        for rid in ids:
            r = srv.result(rid)
            out.append({x: r[x] for x in ("P", "Q", "L", "U", "info")})
            srv.release(rid)
        return out
    if kind == "fast":
        return st["plan"].run(st["A"], st["theta"], st["s"])
    if kind == "lstsq":
        return rlu.lstsq(*st["args"])
    if kind == "residual":
        fro, spec = rlu.reconstruct_error(*st["args"], power_iters=st["iters"])
        return {"fro": fro} if spec is None else {"fro": fro, "spec": spec}
    r = rlu.rsvd(st["A"], st["k"], st["l"], st["seed"])
    return {x: r[x] for x in ("Q", "B", "sigma", "info")}


# ---- what a pass cannot do without ----------------------------------------------------------


def _factor_work(m, n, k, l, esz, osz, q=0):
    """A read once, the factors and permutations written; the method's operations."""
    flops = (2 * m * n * l * (1 + 2 * q) + m * l * l + m * k * k + 2 * m * n * k + 2 * k * k * n
             + n * k * k + m * k * k + k ** 3 // 3)
    return {"bytes": m * n * esz + (m * k + k * n) * osz + 4 * (m + n), "flops": flops}


def _sum(works):
    works = list(works)
    return {x: sum(w[x] for w in works) for x in ("bytes", "flops")}


def work(case):
    kind = case["kind"]
    if kind == "factor":
        esz = {"f64": 8, "bf16": 2}.get(case["prec"], 4)
        return _factor_work(case["m"], case["n"], case["k"], case["l"], esz,
                            8 if case["prec"] == "f64" else 4, case["q"])
    if kind == "batch":
        return _sum(_factor_work(*s, 4, 4) for s in _batch_shapes(case))
    if kind == "serve":
        return _sum(_factor_work(*s[:4], 2 if s[4] == "bf16" else 4, 4)
                    for s in _serve_shapes(case))
    m, n, k = case["m"], case["n"], case["k"]
    if kind == "fast":  # complex multiply-adds as four real ones
        l = case["l"]
        flops = (5 * m * n * math.log2(n) + 4 * (m * l * l + 2 * m * k * l + 2 * k * l * n / 2
                                                 + 2 * k * k * n + n * k * k + m * k * k))
        return {"bytes": 4 * m * n + 8 * (m * k + k * n) + 4 * (m + 2 * n + l), "flops": int(flops)}
    if kind == "lstsq":
        esz = 8 if case["dtype"] == "f64" else 4
        r = case["nrhs"]
        return {"bytes": esz * (m * k + k * k + m * r + n * r) + 4 * (m + n),
                "flops": m * k * k + k ** 3 // 3 + 2 * m * k * r + 3 * k * k * r}
    if kind == "residual":
        asz = {"f64": 8, "f32": 4, "bf16": 2}[case["dtype"]]
        esz = 8 if case["dtype"] == "f64" else 4
        return {"bytes": asz * m * n + esz * (m * k + k * n) + 4 * (m + n) + 16,
                "flops": 2 * m * n * k + 2 * m * n + case["iters"] * 4 * (m * n + m * k + k * n)}
    l = case["l"]
    return {"bytes": 8 * (m * n + m * k + k * n + l),
            "flops": 2 * m * n * l + m * l * l + 2 * m * l * k + 2 * m * n * k + 10 * l ** 3}


# ---- 64-bit values --------------------------------------------------------------------------


def _gaussian(seed, n, l, prec, lda):
    """G (n x l) from the library's stated generator: Philox4x32-10, element e = j n + i of
    counter e / 4, Box-Muller on 32-bit (FP64 path) or 24-bit uniforms. The FP64 deviates are
    rounded to what the path's product reads: FP32, its TF32 part, or BF16."""
    dev, mask = _device(), 0xFFFFFFFF
    count = (n * l + 3) // 4
    c0 = torch.arange(count, device=dev, dtype=torch.int64)
    c = [c0 & mask, c0 >> 32, torch.zeros_like(c0), torch.zeros_like(c0)]
    k0, k1 = seed & mask, (seed >> 32) & mask
    for r in range(10):
        a, b = c[0] * 0xD2511F53, c[2] * 0xCD9E8D57  # low 64 bits; halves taken unsigned
        c = [((b >> 32) & mask) ^ c[1] ^ k0, b & mask, ((a >> 32) & mask) ^ c[3] ^ k1, a & mask]
        k0, k1 = (k0 + 0x9E3779B9) & mask, (k1 + 0xBB67AE85) & mask
    z = []
    for xa, xb in ((c[0], c[1]), (c[2], c[3])):
        if prec == "f64":
            u, t = (xa.double() + 1) * 2.0 ** -32, xb.double() * 2.0 ** -32
        else:
            u, t = ((xa >> 8).double() + 1) * 2.0 ** -24, (xb >> 5).double() * 2.0 ** -27
        r = torch.sqrt(-2 * torch.log(u))
        z += [r * torch.cos(2 * math.pi * t), r * torch.sin(2 * math.pi * t)]
    G = torch.stack(z, 1).reshape(-1)[:n * l].reshape(l, n).t()
    if prec == "f64":
        return G
    G = G.float()
    if prec == "bf16":
        return G.bfloat16().double()
    if prec == "mixed" and lda % 4 == 0:  # the tensor cores read the upper 19 bits
        G = (G.contiguous().view(torch.int32) & ~0x1FFF).view(torch.float32)
    return G.double()


# Where the two largest candidates of a pivot step are nearer to each other than the path's
# rounding, either is a right pivot and the factors have no one value.
_NEAR = {"f64": 1e-11, "f32": 1e-4, "mixed": 1e-3, "bf16": 5e-3, "fast": 1e-3}


def _near_tie(lo, up, tol):
    """Whether a step of the pivoted LU lo, up (unit lower, upper) had two near candidates."""
    below = torch.tril(lo, -1) * torch.diagonal(up)
    mag = below.abs()
    top = torch.diagonal(up).abs()
    if lo.is_complex():
        mag, top = below.real.abs() + below.imag.abs(), (
            torch.diagonal(up).real.abs() + torch.diagonal(up).imag.abs())
    return bool((mag.max(dim=0).values > (1 - tol) * top).any())


def _settled(L, U, *steps):
    """run()'s outputs from the 64-bit factors; None where a pivot was a near tie."""
    if any(_near_tie(*s) for s in steps):
        return None
    return {"P": None, "Q": None, "L": L, "U": U, "info": None}


def _exact_factor(A, k, l, seed, prec, q=0):
    lda = A.stride(0)
    A64 = A.double()
    Y = A64 @ _gaussian(seed, A.shape[1], l, prec, lda)
    for _ in range(q):  # the normalisation changes no pivot and no factor
        Y = A64 @ (A64.t() @ Y)
    P, Lf, Uf = _pivoted_lu(Y)
    Ly = Lf[:, :k].to(A.device)
    Lt = torch.empty_like(Ly)
    Lt[P.to(A.device)] = Ly
    B = torch.linalg.solve(Lt.t() @ Lt, Lt.t() @ A64)
    Q, Lb, U, second = _column_pivoted_lu(B)
    tol = _NEAR[prec]
    return _settled(Ly @ Lb.to(A.device), U, (Lf, Uf, tol), (*second, tol))


def _exact_fast(case, seed, A):
    theta, s = _srft_params(case, seed)
    n, k, l = case["n"], case["k"], case["l"]
    d = torch.polar(torch.ones(n, dtype=torch.float64, device=A.device),
                    2 * math.pi * theta.double())
    Y = torch.fft.fft(A.double() * d, dim=1)[:, s.long()] / math.sqrt(n)
    P, Lf, Uf = _pivoted_lu(Y)
    first = (Lf, Uf, _NEAR["fast"])
    P, Lf = P.to(A.device), Lf.to(A.device)
    J = P[:l]
    PX = torch.linalg.solve_triangular(Lf[:l], Lf, upper=False, left=False, unitriangular=True)
    Ly = Lf[:, :k]
    B = torch.linalg.solve(Ly.mH @ Ly, (Ly.mH @ PX) @ A.double()[J].to(Lf.dtype))
    Q, Lb, U, second = _column_pivoted_lu(B)
    return _settled(Ly @ Lb.to(A.device), U, first, (*second, _NEAR["fast"]))


def exact(case, seed):
    kind = case["kind"]
    g = _generator(seed)
    if kind == "factor":
        A = _matrix(case["m"], case["n"], case["k"], _DTYPE[case["prec"]], g)
        return _exact_factor(A, case["k"], case["l"], _philox_seed(seed), case["prec"], case["q"])
    if kind == "batch":
        out = []
        for i, (m, n, k, l) in enumerate(_batch_shapes(case)):
            A = _matrix(m, n, k, torch.float32, g)
            A = torch.nn.functional.pad(A, (0, -n % 4))[:, :n]
            out.append(_exact_factor(A, k, l, _philox_seed(seed) + i, case["prec"]))
        # packed as run() packs them; one unsettled problem leaves a pack without a value
        if any(o is None for o in out):
            return None
        return {"P": None, "Q": None, "L": torch.cat([o["L"].t().reshape(-1) for o in out]),
                "U": torch.cat([o["U"].reshape(-1) for o in out]), "info": None}
    if kind == "serve":
        shapes = _serve_shapes(case)
        big = max(max(s[:2]) for s in shapes)
        A = _matrix(big, (big + 7) // 8 * 8, 128, torch.float32, g)
        out = []
        for i, (m, n, k, l, prec) in enumerate(shapes):
            block = (A.bfloat16() if prec == "bf16" else A)[:m, :n]
            out.append(_exact_factor(block, k, l, _philox_seed(seed) + i, prec))
        if all(o is None for o in out):
            return None
        return [o or {x: None for x in ("P", "Q", "L", "U", "info")} for o in out]
    if kind == "fast":
        A = _matrix(case["m"], case["n"], case["k"], torch.float32, g)
        return _exact_fast(case, seed, A)
    if kind == "lstsq":
        P, Q, L, U, b = _lstsq_inputs(case, seed)
        L, U, k = L.double(), U.double(), case["k"]
        y = torch.linalg.solve(L.t() @ L, L.t() @ b.double()[P.long()].reshape(case["m"], -1))
        x = torch.zeros(case["n"], y.shape[1], device=y.device, dtype=y.dtype)
        x[Q.long()[:k]] = torch.linalg.solve_triangular(U[:, :k], y, upper=True)
        return x[:, 0] if b.dim() == 1 else x
    if kind == "residual":
        A, P, Q, L, U = _residual_inputs(case, seed)
        R = A.double()[P.long()][:, Q.long()] - L.double() @ U.double()
        # the spectral norm is an estimate after a stated number of iterations
        return {"fro": torch.linalg.norm(R), **({"spec": None} if case["iters"] else {})}
    A = _matrix(case["m"], case["n"], case["k"], torch.float64, g)
    Y = A @ _gaussian(_philox_seed(seed), case["n"], case["l"], "f64", 0)
    return {"Q": None, "B": None, "sigma": torch.linalg.svdvals(Y), "info": None}
