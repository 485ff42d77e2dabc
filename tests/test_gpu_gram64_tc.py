"""The FP64 Gram from exact tensor-core integer products against extended-precision sums, at the
edges of its tiles, sample blocks and runs, and a fit that takes it against the FP64 kernel."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _rows(n, N, seed):
    """Rows of several shapes: normal, heavy-tailed (one sample dominates), two-valued (the leading
    digit at its largest in every sample), uniform, and one zero row."""
    r = np.random.default_rng([n, N, seed])
    Z = r.normal(size=(n, N))
    Z[1::5] = np.exp(6 * r.normal(size=Z[1::5].shape))
    Z[2::5] = np.where(r.random(Z[2::5].shape) < 0.5, -0.9999999, 0.9999999)
    Z[3::5] = r.random(Z[3::5].shape)
    if n > 4:
        Z[4] = 0.0
    sd = np.sqrt((Z * Z).mean(1, keepdims=True))
    return Z / np.where(sd > 0, sd, 1.0)


# samples: less than a block of 64, its edges, several runs; rows: one, the 64-wide and 128-high
# tiles' edges, several tiles both ways
@pytest.mark.parametrize("n,N", [(1, 3), (5, 63), (7, 64), (33, 65), (63, 1000), (64, 129), (65, 8193), (127, 640), (128, 512),
                                 (129, 1027), (70, 20011), (300, 577)])
def test_gram_error_against_extended_sums(n, N):
    from paper_2410_01752_gb300 import sisso as S
    Z = _rows(n, N, 0)
    y = np.random.default_rng(n).normal(size=N)
    G, b = S.gram_fp64(Z, y)
    L = Z.astype(np.longdouble)
    ref = (L @ L.T) / N
    # q rounds a row to half of 2^(e - 54); products of weight 8 and above are dropped; one
    # rounding of the sum, the division and the conversion
    e = np.exp2(np.ceil(np.log2(np.maximum(np.abs(Z).max(1), 1e-300)) + 1e-9))
    m1 = np.abs(Z).mean(1)
    tol = (2.0 ** -51 * np.abs(ref).astype(float) + 2.0 ** -55 * (np.outer(e, m1) + np.outer(m1, e))
           + 2.0 ** -59 * np.outer(e, e))
    err = np.abs((G - ref).astype(float))
    assert np.all(err <= tol), (err / tol).max()
    assert np.array_equal(G, G.T)
    assert np.abs(b - (L @ y) / N).max() <= 1e-13 * np.sqrt((y * y).mean())


def test_long_fit_takes_it(orc):
    """8192 samples and 90 features a step (over the rule's line): the oracle's selections,
    descriptors and coefficients."""
    from paper_2410_01752_gb300 import inputs
    from paper_2410_01752_gb300 import sisso as S
    P = inputs.workload3(2, N=8192, sis_size=180, max_dim=2)
    sp = orc.Space(12, P.op_set, 2)
    ref = orc.fit(P.X, P.y, sp, 180, 2)
    with S.Sisso(P.X, P.y, P.op_set, 2, 180, 2) as c:
        for t, (g, r) in enumerate(zip(c.fit(), ref.dims)):
            assert c.sis(t + 1) == ref.sis[t]
            assert g.ids == r.ids
            np.testing.assert_allclose(g.coef, r.coef, rtol=1e-6, atol=1e-9 * np.abs(P.y).max())
