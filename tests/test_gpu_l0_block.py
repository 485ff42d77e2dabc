"""The l0 enumerations by dimension -- FP64 pairs (D = 2 and 3), and a prefix eliminated once per
CTA (D = 4 and 5): the winner, its RSS
and the number of subsets examined equal the FP64 enumeration's at the sizes where its split,
row groups and launches change."""
import math

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _gram(n, N, seed, twins):
    """Gram and moments of n standardised features, the last `twins` nearly equal to the first."""
    r = np.random.default_rng(seed)
    F = r.normal(size=(n, N)) + 0.5 * r.normal(size=N)
    for q in range(twins):
        F[n - 1 - q] = F[q] + 1e-4 * r.normal(size=N)
    Z = F - F.mean(1, keepdims=True)
    Z /= Z.std(1, keepdims=True)
    terms = min(4, n)
    c = r.uniform(1, 3, size=terms)
    pick = r.choice(n, size=terms, replace=False)
    y = c @ Z[pick] + 0.05 * r.normal(size=N)
    y -= y.mean()
    return Z @ Z.T / N, Z @ y / N, float(y @ y / N)


# D = 2, 3: smallest, a warp's and a CTA's edge, several slices of rows; the FP64 form's largest
# subset count (1063 features at D = 3), beyond which the tiled kernel runs.  D = 4, 5:
# smallest; one row group and its edge; two sweeps of six groups (193 rows); either side of the
# line between the two launches (150 features right of the prefix) and of the shared-memory
# capacity (320), beyond which the tiled kernel runs
@pytest.mark.parametrize("D,n", [(2, 2), (2, 3), (2, 33), (2, 257), (2, 700), (3, 3), (3, 4), (3, 33), (3, 34), (3, 65),
                                 (3, 130), (3, 258), (3, 1063), (3, 1064), (4, 4), (4, 5),
                                 (4, 34), (4, 36), (4, 67), (4, 151), (4, 152), (4, 196), (4, 321), (4, 322),
                                 (5, 5), (5, 6), (5, 35), (5, 37), (5, 70), (5, 100)])
@pytest.mark.parametrize("twins", [0, 3])
def test_block_search_equals_fp64_search(D, n, twins):
    from paper_2410_01752_gb300 import sisso as S
    N = 200
    G, b, syy = _gram(n, N, 100 * D + n, min(twins, n // 2))
    gid = np.random.default_rng(n).permutation(5 * n)[:n].astype(np.int64)
    r = np.random.default_rng(1)
    with S.Sisso(r.uniform(1, 5, size=(N, 3)), r.normal(size=N), 1, 1, 2, 1) as c:
        got = c.l0_search(G, b, syy, D, gid, S.PREC_FP32)
        ref = c.l0_search(G, b, syy, D, gid, S.PREC_FP64)
    assert got[2] == ref[2] == math.comb(n, D)
    assert got[0] == ref[0]
    assert got[1] == pytest.approx(ref[1], rel=1e-9, abs=1e-9 * syy * N)
