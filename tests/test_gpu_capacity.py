"""What fits the device, and what a call leaves behind when it does not."""
import numpy as np
import pytest

from paper_2410_01752_gb300 import inputs

pytestmark = pytest.mark.gpu


def _problem(N, d, seed=0):
    r = np.random.default_rng([N, d, seed])
    X = np.exp(r.normal(0, 0.4, size=(N, d)))
    return X, X[:, 0] * X[:, 1] + np.log(X[:, -1]) + 0.05 * r.normal(size=N)


def test_a_failed_creation_leaves_no_error():
    """A space far too large is refused for its memory; the next context is not."""
    from paper_2410_01752_gb300 import sisso as S
    X, y = _problem(50, 40)
    with pytest.raises(S.SissoError):
        S.Sisso(X, y, inputs.OPS9, 3, 5, 2)
    Y, z = _problem(50, 3)
    with S.Sisso(Y, z, inputs.OPS9, 2, 5, 2) as c:
        assert len(c.fit()) >= 1
