"""The register z pass where a CTA runs several passes (rows and right-hand sides).

A CTA asks for the next pass's columns while the present one still uses the
shared memory they land in.  Ten right-hand sides on these grids give a CTA two
to seven passes (one right-hand side alone gives it one), for every odd plan and
an even one, with pairs of columns copied at a time (even x length) and with plain
loads (odd).  Every right-hand side does the same arithmetic alone and in a
batch, so the results have to be the same to the last bit; against the
shared-memory kernel they agree to what the refinement leaves.
"""
import numpy as np
import pytest

from dda_inputs import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape", [
    # z lengths 15, 25, 27, 45, 75, 81, 135, 225
    (64, 64, 8), (64, 50, 13), (60, 50, 14), (64, 32, 23), (64, 32, 38), (50, 27, 41),
    (48, 20, 68), (33, 20, 113),
    # odd x length (81): z lengths 45, 81; even z lengths 72 and 128
    (41, 40, 23), (41, 40, 41), (50, 40, 36), (41, 40, 64)])
def test_batches_equal_their_right_hand_sides(shape):
    from paper_1305_6497_gb300 import binding as B
    w = W.small_ellipsoid(*shape, m=1.4 + 0.05j, kd=0.2, method="LDR", n_orient=5, seed=4)
    t = B.Target(w.occ, w.comp, w.m, method="LDR")
    # a given inner tolerance: the adaptive one depends on the whole batch
    kw = dict(tol=1e-9, inner_tol=1e-5, max_iter=300, precision="fp32_refined")
    for _ in range(2):
        a = t.solve(w.kd, w.khat, w.e01, yhat=w.yhat, npol=2, **kw)
        assert a["status"] == B.DDA_OK
        assert t.schedule("fp32")["z_stage_ghat"] & 15 == 8
        for i in range(5):
            one = t.solve(w.kd, w.khat[i:i + 1], w.e01[i:i + 1], yhat=w.yhat[i:i + 1], npol=1,
                          **kw)
            assert one["iters"][0] == a["iters"][2 * i]
            np.testing.assert_array_equal(one["P"][0], a["P"][2 * i])
    t.set_schedule(dict(t.schedule("fp32"), z_tile=4, z_pitch=13, z_stage_ghat=0, z_threads=128),
                   "fp32")
    b = t.solve(w.kd, w.khat, w.e01, yhat=w.yhat, npol=2, **kw)
    assert np.abs(b["P"] - a["P"]).max() <= 1e-7 * np.abs(a["P"]).max()
    t.close()
