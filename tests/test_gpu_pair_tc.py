"""The tensor-core pair screening at the edges of its tiles and sample runs: the keys of a
context's first target (five sums per pair) and of a later one (one sum, kept deviations)
against the oracle's scores."""
import numpy as np
import pytest

from paper_2410_01752_gb300 import inputs

pytestmark = pytest.mark.gpu

TOL = 2e-4      # the FP32 screening margin: keys within it of the 64-bit scores select the same windows
NAMES = {"all": inputs.OPS9, "sub": ["-"], "mul": ["*"], "div-sq": ["/", "^2"], "pm-exp": ["+", "-", "exp"]}


def _problem(N, d, seed):
    r = np.random.default_rng([N, d, seed])
    X = np.exp(r.normal(0, 0.4, size=(N, d))) * np.where(r.random(d) < 0.3, -1.0, 1.0)
    return X, X[:, 0] * X[:, -1] + 0.1 * r.normal(size=N), X[:, 0] - X[:, -1] + r.normal(size=N)


# samples: one run of 64 and its edges, the register-kept rows' limits (256, 1024), the one-chunk
# limit (2048), many chunks; rung 1 operands: the smallest, one 48-wide and one 128-wide tile and
# their edges, the widest i tile and its edge
CASES = [(N, 5, "all", 2, 0) for N in (4, 63, 64, 65, 256, 257, 1024, 1025, 2048, 2049, 9000)]
CASES += [(90, d, "all", 1, 0) for d in (2, 47, 48, 49, 127, 128, 129, 240, 241, 300)]
CASES += [(130, 6, ops, 2, 0) for ops in ("sub", "mul", "div-sq", "pm-exp")]
CASES += [(70, 2, "pm-exp", 3, 0), (70, 3, "pm-exp", 3, 1), (2200, 2, "div-sq", 3, 1)]


@pytest.mark.parametrize("N,d,ops,rung,g", CASES)
@pytest.mark.parametrize("prec", [1, 2, 3])
def test_keys_of_first_and_later_targets(orc, N, d, ops, rung, g, prec):
    from paper_2410_01752_gb300 import sisso as S
    X, y0, y1 = _problem(N, d, rung)
    m = NAMES[ops]
    if not isinstance(m, int):
        m = orc.opmask(*[orc.OP_NAMES.index(n) for n in m])
    sp = orc.Space(d, m, rung, g)
    with S.Sisso(X, y0, m, rung, 2, 1, precision=prec, grammar=g, screen=S.SCREEN_TENSOR) as c:
        keys = [c.score_all(y, prec).astype(np.float64) for y in (y0, y1)]
    for y, got in zip((y0, y1), keys):
        ref, valid = sp.scores(X, y)
        assert not np.any((got < 0) & valid)
        assert np.abs(got[valid] - ref[valid]).max(initial=0.0) <= TOL
