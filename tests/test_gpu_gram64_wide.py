"""The exact tensor-core Gram of rows whose largest value is many deviations (a spike, reciprocals near
zero): entries no further from extended-precision sums than FP64 sums are."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N", [65, 8192, 65536])
def test_rows_with_a_wide_range(N):
    from paper_2410_01752_gb300 import sisso as S
    r = np.random.default_rng(N)
    spike = np.arange(N) == 7
    Z = np.stack([r.normal(size=N), 1e-3 * r.normal(size=N) + spike, 1 / r.normal(size=N), r.standard_cauchy(size=N),
                  np.exp(2 * r.normal(size=N)), 1e-3 * r.normal(size=N) + spike, r.uniform(size=N)])
    Z -= Z.mean(1, keepdims=True)
    Z /= Z.std(1, keepdims=True)
    G, _ = S.gram_fp64(Z, r.normal(size=N))
    L = Z.astype(np.longdouble)
    ref = (L @ L.T) / N
    # an FP64 sum by 256 threads: N / 256 roundings each, of random sign, and a few for the rest
    u = 2.0 ** -53
    tol = (np.sqrt(N / 256) + 8) * u * np.sqrt(np.outer(np.diag(ref), np.diag(ref)).astype(float))
    err = np.abs((G - ref).astype(float))
    assert np.all(err <= tol), (err / u).max()
