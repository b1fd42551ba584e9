"""Chained launches against ordinary ones.

The kernels of an iteration may start while their predecessor still runs
(waiting for it before they touch its results); a profiled solve records events
between the passes and launches them one after the other instead.  Both run the
same kernels on the same numbers, so everything they return has to be the same
to the last bit: a kernel that read too early would show.  Sizes: boxes of a
few sites (a pass is shorter than a launch), register and shared-memory passes,
batches whose right-hand sides converge at different iterations.
"""
import numpy as np
import pytest

from dda_inputs import workloads as W

pytestmark = pytest.mark.gpu

CASES = [
    ((3, 4, 5), "fp32_refined", "bicgstab", 1),
    ((16, 16, 16), "fp64", "bicgstab", 1),
    ((9, 12, 7), "fp64", "bicgstab2", 2),
    ((20, 24, 18), "fp32_refined", "bicgstab", 5),
    ((20, 24, 18), "fp32_refined", "bicgstab2", 3),
    ((15, 25, 45), "fp32_refined", "qmr", 2),
    ((22, 17, 12), "fp32_refined", "gpbicg", 1),
    ((14, 10, 12), "fp32_refined", "petrkp", 1),
    ((48, 40, 36), "fp32_refined", "bicgstab", 2),
]


@pytest.mark.parametrize("box,precision,solver,n_inc", CASES)
def test_chained_launches_give_the_same_bits(box, precision, solver, n_inc):
    from paper_1305_6497_gb300 import binding as B
    w = W.small_ellipsoid(*box, m=1.4 + 0.05j, kd=0.25, method="LDR", n_orient=n_inc, seed=3)
    t = B.Target(w.occ, w.comp, w.m, method="LDR")
    kw = dict(yhat=w.yhat, precision=precision, solver=solver, max_iter=400,
              tol=1e-9 if precision == "fp64" else 1e-10)
    ref = t.solve(w.kd, w.khat, w.e01, profile=True, **kw)
    for _ in range(3):
        out = t.solve(w.kd, w.khat, w.e01, **kw)
        assert list(out["iters"]) == list(ref["iters"])
        np.testing.assert_array_equal(out["P"], ref["P"])
        np.testing.assert_array_equal(out["Qext"], ref["Qext"])
    t.close()
