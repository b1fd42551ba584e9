"""A tuned schedule is no slower in a solve than the default it replaces.

The tuner times passes alone, where a chained pass overlaps its own copy; the passes
together decide.  3 % is left for the timing of short solves (repeats differ by 0.5 %).
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape", [(16, 16, 16), (64, 64, 64), (64, 64, 128)])
def test_tuned_iterations_are_not_slower(shape):
    from paper_1305_6497_gb300 import binding as B
    t = B.Target(np.ones(shape[::-1], np.uint8), None, [1.4 + 0.05j], method="CM")
    kw = dict(npol=2, tol=1e-30, max_iter=48, precision="fp32", want_P=False, want_famp=False)

    def iteration():
        return min(o["t_solve_ms"] / max(o["iters"]) for o in
                   (t.solve(0.2, [[1.0, 0, 0]], [[0, 1.0, 0]], **kw) for _ in range(8)))

    default, s = iteration(), t.schedule("fp32")
    t.autotune(0.2, 2)
    tuned = iteration()
    t.set_schedule(s, "fp32")
    assert tuned <= 1.03 * min(default, iteration())
    t.close()
