"""Several host threads in the library at once, each on its own stream with its own plan: calls
of different sizes that use the same kernels with different amounts of shared memory. Every call
succeeds and every result is the one that the plan gives alone, to the bit. GPU only."""
import threading

import pytest
import torch

from paper_1310_7202_gb300 import rlu, synth

pytestmark = pytest.mark.gpu


def _matrix(m, n, seed, dtype=torch.float32):
    g = torch.Generator("cuda").manual_seed(seed)
    return torch.randn(m, n, generator=g, device="cuda", dtype=torch.float64).to(dtype)


def _factor(m, n, k, l, prec="mixed", dtype=torch.float32):
    A = _matrix(m, n, m + k, dtype)
    plan = rlu.Factorizer(m, n, k, l, prec)

    def call():
        return list(plan(A, 7)[:4])
    return call


def _rsvd(m, n, k, l):
    A = _matrix(m, n, m + k, torch.float64)

    def call():
        r = rlu.rsvd(A, k, l, 7)
        return [r[x] for x in ("Q", "B", "sigma")]
    return call


def _fast(m, n, k, l):
    A = _matrix(m, n, m + k)
    theta, s = (torch.from_numpy(x).cuda() for x in synth.srft_params(n, l, 3))
    plan = rlu.FastFactorizer(m, n, k, l)
    out = plan.run(A, theta, s)

    def call():
        o = plan.run(A, theta, s, out)
        return [o[x] for x in ("P", "Q", "L", "U")]
    return call


def _batch(shapes):
    probs = [{"A": _matrix(m, n, m + k), "k": k, "l": k + 4, "seed": 7} for m, n, k in shapes]
    b = rlu.Batch(probs, "f32")

    def call():
        b.run()
        return [o[x] for o in b.outs for x in ("P", "Q", "L", "U")]
    return call


# pairs of calls that share kernels: panels of other widths (LU), other k (LDL^T, solves), other
# l (eigensolver), other n (row transform), longer problems (batched gathers)
@pytest.mark.parametrize("makers", [
    (lambda: _factor(2000, 1900, 12, 16), lambda: _factor(2000, 1900, 70, 76)),
    (lambda: _factor(1000, 1900, 30, 40), lambda: _factor(1000, 1900, 200, 230)),
    (lambda: _factor(1500, 900, 10, 12, "f64", torch.float64),
     lambda: _factor(1500, 900, 60, 64, "f64", torch.float64)),
    (lambda: _rsvd(90, 80, 6, 8), lambda: _rsvd(90, 80, 50, 56)),
    (lambda: _fast(200, 128, 10, 16), lambda: _fast(200, 1024, 30, 64)),
    (lambda: _batch([(900, 300, 12)]), lambda: _batch([(300, 200, 60), (2000, 600, 60)]))],
    ids=["panel", "solve", "f64", "rsvd", "fast", "batch"])
def test_two_threads(makers):
    calls = [mk() for mk in makers]
    alone = [[x.clone() for x in c()] for c in calls]
    torch.cuda.synchronize()
    failed = []

    def work(call):
        try:
            with torch.cuda.stream(torch.cuda.Stream()):
                for i in range(200):
                    out = call()
                    if i % 20 == 19:
                        torch.cuda.current_stream().synchronize()
                last.append((call, [x.clone() for x in out]))
                torch.cuda.current_stream().synchronize()
        except Exception as e:  # noqa: BLE001  (reported by the main thread)
            failed.append(e)
    last = []
    threads = [threading.Thread(target=work, args=(c,)) for c in calls]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    torch.cuda.synchronize()
    assert not failed, failed
    for call, out in last:
        for x, y in zip(alone[calls.index(call)], out):
            assert torch.equal(x, y)
