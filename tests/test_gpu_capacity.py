"""What fits the device: buffers that only make a fit faster are left out where the memory left does
not hold them, with the same results; and what a call leaves behind when it does not fit."""
import numpy as np
import pytest

from paper_2410_01752_gb300 import inputs

pytestmark = pytest.mark.gpu

GB = 1 << 30


class _Held:
    """All of the device's free memory but `leave` bytes, while the block lasts."""

    def __init__(self, S, leave):
        self.S, self.leave = S, leave

    def __enter__(self):
        import torch
        self.S.release_memory(0)
        torch.cuda.empty_cache()
        free = torch.cuda.mem_get_info(0)[0]
        self.block = torch.empty(max(0, free - int(self.leave)), dtype=torch.uint8, device="cuda:0")

    def __exit__(self, *_):
        import torch
        self.block = None
        torch.cuda.empty_cache()


def _memory_of(S, make):
    """Device memory that a new context of an emptied pool takes."""
    import torch
    S.release_memory(0)
    before = torch.cuda.mem_get_info(0)[0]
    with make():
        return before - torch.cuda.mem_get_info(0)[0]


def _fit(c):
    d = c.fit()
    return d, [c.sis(t + 1) for t in range(len(d))]


def _same(a, b):
    assert [g.ids for g in a[0]] == [g.ids for g in b[0]] and a[1] == b[1]
    for g, h in zip(a[0], b[0]):
        np.testing.assert_allclose(g.coef, h.coef, rtol=1e-9, atol=1e-12)


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


def test_deviations_that_do_not_fit():
    """Rung 3 over phi_2 x phi_2: 6.5e8 candidates, 2.6 GB of scores; the deviations kept for later
    steps are 5.2 GB more."""
    from paper_2410_01752_gb300 import sisso as S
    X, y = _problem(40, 5)
    with S.Sisso(X, y, inputs.OPS9, 3, 5, 2) as c:
        ref = _fit(c)
    with _Held(S, 5.5 * GB), S.Sisso(X, y, inputs.OPS9, 3, 5, 2) as c:
        _same(_fit(c), ref)


def test_pair_buffers_that_cannot_be_allocated():
    """234 operands over 65 536 samples with room for half of the pair stage's 0.8 GB."""
    from paper_2410_01752_gb300 import sisso as S
    X, y = _problem(65536, 9)

    def make(screen):
        return S.Sisso(X, y, inputs.OPS9, 2, 20, 2, precision=S.PREC_MIXED_FP16, screen=screen)

    with make(S.SCREEN_AUTO) as c:
        ref = _fit(c)
        assert c.stats()["screen_tc"] == 1
    base = _memory_of(S, lambda: make(S.SCREEN_CORES))
    pair = _memory_of(S, lambda: make(S.SCREEN_AUTO)) - base
    assert pair > GB // 2
    with _Held(S, base + pair // 2), make(S.SCREEN_AUTO) as c:
        _same(_fit(c), ref)
        assert c.stats()["screen_tc"] == 0


def test_partial_sums_in_bounded_batches():
    """2355 operands over 16 384 samples: the partial sums of all tiles together are 1.5 GB.  They are
    taken in batches, and the keys are those of the CUDA-core kernel."""
    from paper_2410_01752_gb300 import sisso as S
    X, y = _problem(16384, 30)

    def make(screen):
        return S.Sisso(X, y, inputs.OPS9, 2, 5, 1, precision=S.PREC_MIXED_FP16, screen=screen)

    keys = {}
    for screen in (S.SCREEN_CORES, S.SCREEN_AUTO):
        with make(screen) as c:
            keys[screen] = [c.score_all(t, S.PREC_MIXED_FP16) for t in (y, X[:, 0] + y)]
            assert c.stats()["screen_tc"] == (screen == S.SCREEN_AUTO)
    for a, b in zip(keys[S.SCREEN_CORES], keys[S.SCREEN_AUTO]):
        both = (a >= 0) & (b >= 0)
        assert both.mean() > 0.5 and np.mean((a >= 0) != (b >= 0)) < 1e-3
        assert np.abs(a[both] - b[both]).max() <= 4e-4          # each within 2e-4 of the 64-bit score
    # rows, target rows, FP32 values and deviations of the pair stage, one batch of sums, and slack
    cells, K = 2355, 16384
    room = 28 * cells * K + 20 * cells * cells + GB + GB // 4
    assert _memory_of(S, lambda: make(S.SCREEN_AUTO)) - _memory_of(S, lambda: make(S.SCREEN_CORES)) <= room


def test_gram_digits_that_do_not_fit():
    """600 features over 65 536 samples: 0.55 GB of digits for the exact Gram, asked for in the fit."""
    from paper_2410_01752_gb300 import sisso as S
    X, y = _problem(65536, 3)
    with S.Sisso(X, y, inputs.OPS9, 2, 200, 3) as c:
        ref = _fit(c)
    with S.Sisso(X, y, inputs.OPS9, 2, 200, 3) as c, _Held(S, GB // 3):
        _same(_fit(c), ref)


def test_batch_values_that_do_not_fit():
    """The deviations that a batch keeps for later steps take most of what its other buffers leave."""
    from paper_2410_01752_gb300 import sisso as S
    problems = [_problem(2000, 9, seed) for seed in range(96)]

    def make():
        return S.Batch(problems, inputs.OPS9, 2, 20, 2)

    with make() as b:
        b.run()
        ref = b.results()
    base = _memory_of(S, make)
    inputs_bytes = 96 * 2000 * 10 * 8
    with _Held(S, base - inputs_bytes // 2), make() as b:
        b.run()
        for (st0, a), (st1, g) in zip(ref, b.results()):
            assert st0 == st1 == 0 and [m.ids for m in a] == [m.ids for m in g]
