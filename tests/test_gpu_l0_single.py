"""The l0 search where all but one subset are singular, so that neither the greedy bound nor the first
candidates of any feature give a bound: the one subset is found."""
import math

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("D,n,members", [(4, 60, (5, 17, 30, 44)), (5, 40, (3, 9, 14, 22, 30)), (4, 60, (0, 1, 2, 3)),
                                         (4, 60, (56, 57, 58, 59)), (3, 90, (7, 40, 61))])
def test_the_one_regular_subset(D, n, members):
    """Unit correlations but among the members, which are uncorrelated; another feature has the largest
    moment, so that a greedy search takes it and finds every extension singular."""
    from paper_2410_01752_gb300 import sisso as S
    N = 100
    G = np.ones((n, n))
    for i in members:
        for j in members:
            G[i, j] = float(i == j)
    b = np.full(n, 0.01)
    b[list(members)] = 0.3
    b[12] = 0.9
    r = np.random.default_rng(0)
    gid = np.arange(n, dtype=np.int64)
    with S.Sisso(r.uniform(1, 5, size=(N, 3)), r.normal(size=N), 1, 1, 2, 1) as c:
        for prec in (S.PREC_FP64, S.PREC_FP32):
            pos, rss, examined = c.l0_search(G, b, 1.0, D, gid, prec)
            assert pos == list(members) and examined == math.comb(n, D)
            assert rss == pytest.approx(N * (1.0 - D * 0.09), rel=1e-12)
