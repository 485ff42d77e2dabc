"""Keys of pairs whose terms nearly cancel: differences and quotients of operands that agree to
1e-4 .. 1e-7, and quotients of operands that span many decades together.  Every key lies within the
screening margin of the oracle's score, for a context's first target and for a later one."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

MARGIN = 2e-4      # the selection's bound on |key - FP64 score|


def _check(orc, X, targets, names, rung, prec):
    from paper_2410_01752_gb300 import sisso as S
    m = orc.opmask(*[orc.OP_NAMES.index(n) for n in names])
    sp = orc.Space(X.shape[1], m, rung, 0)
    with S.Sisso(X, targets[0], m, rung, 2, 1, precision=prec, screen=S.SCREEN_TENSOR) as c:
        keys = [c.score_all(y, prec).astype(np.float64) for y in targets]
    for y, got in zip(targets, keys):
        ref, valid = sp.scores(X, y)
        lost = np.flatnonzero((got < 0) & valid)
        assert lost.size == 0, [(sp.expr(int(i)), ref[i]) for i in lost[:5]]
        err = np.where(valid, np.abs(got - ref), 0.0)
        i = int(err.argmax())
        assert err[i] <= MARGIN, (sp.expr(i), got[i], ref[i])


@pytest.mark.parametrize("delta", [1e-4, 1e-5, 3e-6, 1e-6, 3e-7, 1e-7])
@pytest.mark.parametrize("N,rung", [(100, 1), (1000, 1), (1000, 2), (5000, 1)])
@pytest.mark.parametrize("prec", [1, 2, 3])
def test_nearly_equal_operands(orc, delta, N, rung, prec):
    r = np.random.default_rng([N, rung])
    x, n = r.uniform(1, 5, size=N), r.normal(size=N)
    X = np.stack([x, x + delta * n, r.uniform(1, 5, size=N)], 1)
    targets = [n + 0.1 * r.normal(size=N), n / x + 0.1 * r.normal(size=N)]
    _check(orc, X, targets, ["+", "-", "*", "/"], rung, prec)


@pytest.mark.parametrize("seed", range(6))
@pytest.mark.parametrize("N", [60, 500, 5000])
@pytest.mark.parametrize("prec", [1, 3])
def test_operands_over_many_decades(orc, seed, N, prec):
    r = np.random.default_rng([N, seed])
    x = 10.0 ** r.uniform(-9, 9, size=N)
    a, b = r.normal(size=N), r.normal(size=N)
    X = np.stack([x, x * np.exp(0.1 * a), np.exp(0.1 * b) / x], 1)
    _check(orc, X, [a + 0.3 * b, b - a], ["*", "/"], 1, prec)
