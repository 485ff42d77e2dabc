"""Contexts are independent: host threads, each with its own context and a problem size that needs its
own amount of shared memory, get the results a single thread gets."""
import threading

import numpy as np
import pytest

from paper_2410_01752_gb300 import inputs

pytestmark = pytest.mark.gpu


def _together(*work):
    """Runs the callables in threads of their own; what they raised."""
    raised = []
    start = threading.Barrier(len(work))

    def body(f):
        start.wait()
        try:
            f()
        except Exception as e:                      # noqa: BLE001 (handed to the test)
            raised.append(e)

    threads = [threading.Thread(target=body, args=(f,)) for f in work]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    return raised


def _gram(n, N, seed):
    r = np.random.default_rng(seed)
    Z = r.normal(size=(n, N))
    Z -= Z.mean(1, keepdims=True)
    Z /= Z.std(1, keepdims=True)
    y = Z[0] - 2 * Z[n // 2] + Z[-1] + 0.3 * r.normal(size=N)
    y -= y.mean()
    return Z @ Z.T / N, Z @ y / N, float(y @ y / N)


# two sizes, each above the 48 KB that need no opt-in, on two threads each: the FP64 pairs (D = 2), the
# CTA-shared prefix (D = 4), the two-pass form (FP64 precision)
@pytest.mark.parametrize("D,n,prec,calls", [(2, (1300, 1900), 1, 400), (4, (200, 320), 1, 1000), (3, (270, 400), 0, 600)])
def test_searches_on_several_threads(D, n, prec, calls):
    from paper_2410_01752_gb300 import sisso as S
    N = 100
    r = np.random.default_rng(0)
    X, y = r.uniform(1, 5, size=(N, 3)), r.normal(size=N)

    def search(size):
        G, b, syy = _gram(size, N, size)
        gid = np.arange(size, dtype=np.int64)
        with S.Sisso(X, y, 1, 1, 2, 1) as c:
            first = c.l0_search(G, b, syy, D, gid, prec)
            for _ in range(calls):
                assert c.l0_search(G, b, syy, D, gid, prec) == first

    assert _together(*(lambda size=size: search(size) for size in n * 2)) == []


def test_fits_on_several_threads():
    """Fits of two steps: the keys of the second one (their operand tiles depend on the space)."""
    from paper_2410_01752_gb300 import sisso as S

    def fits(d, rung, g, count):
        r = np.random.default_rng(d)
        X = np.exp(r.normal(0, 0.4, size=(40, d)))
        y = X[:, 0] * X[:, 1] + X[:, 2] / X[:, 3] + 0.1 * r.normal(size=40)
        with S.Sisso(X, y, inputs.OPS9, rung, 5, 2, grammar=g) as c:
            first = None
            for _ in range(count):
                dims = c.fit()
                got = [g.ids for g in dims], [c.sis(t + 1) for t in range(len(dims))]
                assert first is None or got == first
                first = got

    assert _together(*[lambda: fits(5, 3, 1, 700), lambda: fits(4, 2, 0, 1200)] * 2) == []
