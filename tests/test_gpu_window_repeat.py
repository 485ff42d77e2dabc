"""A selection step is repeated with the same candidates only after its window was narrowed: where
the default window is too large to be narrowed (k above 256), a step does the work of an explicit
window of its size."""
import numpy as np
import pytest

from paper_2410_01752_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,k,window", [(333, 300, 9600), (90, 257, 8224)])
def test_no_step_repeated_unchanged(N, k, window):
    """Primaries in nearly equal copies: the walk passes over so many duplicates that the first window
    proves nothing."""
    from paper_2410_01752_gb300 import sisso as S
    r = np.random.default_rng(N)
    X = np.exp(r.normal(0, 0.5, size=(N, 8)))
    for q in range(2, 8):
        X[:, q] = X[:, q % 2] * (1 + 1e-13 * r.normal(size=N))
    y = X[:, 0] * X[:, 1] + 0.05 * r.normal(size=N)
    seen = []
    for survivors in (0, window):
        with S.Sisso(X, y, inputs.OPS9, 2, k, 1, survivors=survivors) as c:
            ids = c.fit()[0].ids
            st = c.stats()
            seen.append((ids, c.sis(1), st["survivors_rescored"], st["window_grown"]))
    assert seen[0][3] > 0
    assert seen[0] == seen[1]
