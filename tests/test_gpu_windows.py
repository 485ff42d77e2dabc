"""Screening windows narrowed before their FP64 work, ranked and sorted in their several sizes, and
the batched form's later steps and integer Grams: the selections and models of the oracle and of
explicitly sized windows."""
import numpy as np
import pytest

from paper_2410_01752_gb300 import inputs

pytestmark = pytest.mark.gpu


def _problem(N, d, seed, copies=0):
    """Lognormal primaries, the last `copies` nearly equal to the first (duplicates to walk over)."""
    r = np.random.default_rng([N, d, seed])
    X = np.exp(r.normal(0, 0.5, size=(N, d)))
    for q in range(copies):
        X[:, d - 1 - q] = X[:, q] * (1 + 1e-13 * r.normal(size=N))
    y = X[:, 0] * X[:, 1] / (1 + X[:, 2 % d]) + np.log(X[:, 0]) + 0.05 * r.normal(size=N)
    return X, y


# samples on either side of the long-sample kernels (4096); windows: the default (narrowed), as
# large as the space (every candidate), past the counted ranks (32768) and the staged walk
@pytest.mark.parametrize("N,d,k,copies", [(40, 5, 5, 0), (333, 8, 40, 3), (4096, 7, 30, 0), (4097, 7, 30, 2), (5000, 10, 20, 4)])
@pytest.mark.parametrize("prec", [0, 1, 3])
def test_narrowed_windows_select_the_same(N, d, k, copies, prec):
    from paper_2410_01752_gb300 import sisso as S
    X, y = _problem(N, d, 0, copies)
    out = []
    for survivors in (0, 7000, 40000):
        with S.Sisso(X, y, inputs.OPS9, 2, k, 2, precision=prec, survivors=survivors) as c:
            dims = c.fit()
            out.append(([c.sis(t + 1) for t in range(len(dims))], [g.ids for g in dims]))
            if survivors == 0 and N > 40 and copies == 0:      # (copies: walks long enough to repeat a step)
                assert c.stats()["survivors_rescored"] < 2 * 4096
    assert out[0] == out[1] == out[2]


# samples: a sample chunk's edges, the integer Gram's range (256 to 4096) and its change of scale
# (1024); operators: all, + and - alone (no sample loop in the later steps), products alone
@pytest.mark.parametrize("N", [20, 31, 32, 33, 255, 256, 257, 1024, 1025, 4096, 4097])
@pytest.mark.parametrize("names,d", [(None, 3), (["+", "-"], 9), (["*"], 8), (["-", "/", "^2"], 4)])
def test_batch_later_steps_equal_the_oracle(orc, N, names, d):
    from paper_2410_01752_gb300 import sisso as S
    m = inputs.OPS9 if names is None else orc.opmask(*[orc.OP_NAMES.index(n) for n in names])
    X, y = _problem(N, d, 1)
    sp = orc.Space(d, m, 2)
    ref = orc.fit(X, y, sp, 12, 3)
    with S.Batch([(X, y)], m, 2, 12, 3) as b:
        b.run()
        status, dims = b.results()[0]
    assert status == 0 and len(dims) == len(ref.dims)
    for g, r in zip(dims, ref.dims):
        assert g.ids == list(r.ids)
        np.testing.assert_allclose(g.coef, r.coef, rtol=1e-6, atol=1e-9 * np.abs(y).max())
        assert abs(g.rmse - r.rmse) <= 1e-6 * r.rmse + 1e-9 * y.std()
