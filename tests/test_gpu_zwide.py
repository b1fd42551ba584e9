"""The FP64 / double-float register z pass: products against the one-tile FP64 kernel
and the direct sum, at the edges of its plans, and the magnetic near field."""
import numpy as np
import pytest

from dda_inputs import targets as tg
from dda_inputs import workloads as W
from oracle import dda as O

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nz", [9, 10, 11, 12, 15, 16, 17, 24, 26, 27, 30, 31, 36, 39, 40, 42, 48,
                                54, 60, 64, 69, 73, 76, 81, 90, 96, 97, 108, 114, 128, 129, 144,
                                150, 160, 168, 192, 217, 240, 251, 256])
def test_products_match(nz):
    from paper_1305_6497_gb300 import binding as B
    occ, comp = tg.rect_prism(7 if nz % 2 else 6, 5, nz)
    flat, pos = O.site_positions(occ)
    x = O.box_to_sites(W.random_polarization(occ, 19)[0], flat)
    t = B.Target(occ, comp, [1.5 + 0.1j], method="CM")
    y = t.matvec(0.4, x)
    s = t.schedule("fp64")
    assert (s["z_stage_ghat"] == 8) == (nz <= 40)
    t.set_schedule(dict(s, z_tile=4, z_pitch=13, z_stage_ghat=0, z_threads=128), "fp64")
    y0 = t.matvec(0.4, x)
    # six transforms of at most nine radix-2 levels, each rounding to 2^-53
    top = np.abs(y0).max()
    assert np.abs(y - y0).max() <= 2 * 6 * 9 * 2.0 ** -53 * top
    # double-float: 2^-48 and a few operations a level
    assert np.abs(t.matvec(0.4, x, precision="df64") - y0).max() <= 4 * 6 * 9 * 2.0 ** -48 * top
    if s["z_stage_ghat"] != 8:   # FP64 takes it on request, too
        t.set_schedule(dict(s, z_tile=4, z_pitch=12, z_stage_ghat=8, z_threads=192), "fp64")
        assert t.schedule("fp64")["z_stage_ghat"] == 8
        assert np.abs(t.matvec(0.4, x) - y0).max() <= 2 * 6 * 9 * 2.0 ** -53 * top
    rows = np.arange(0, len(flat), max(1, len(flat) // 30))
    ainv = O.site_alpha_inverse(comp.reshape(-1)[flat], [1.5 + 0.1j], "CM", 0.4)
    ref = O.matvec_direct(x, pos, ainv, 0.4, "CM", rows=rows)
    assert np.abs(y[rows] - ref).max() <= 1e-10 * np.abs(ref).max()
    t.close()


def test_magnetic_near_field_on_short_lines():
    from paper_1305_6497_gb300 import binding as B
    w = W.small_ellipsoid(4, 6, 6, m=1.5 + 0.1j, kd=0.4, method="CM")
    t = B.Target(w.occ, w.comp, w.m, method="CM")
    rng = np.random.default_rng(3)
    P = rng.standard_normal((2, t.num_dipoles, 3)) + 1j * rng.standard_normal((2, t.num_dipoles, 3))
    ext = np.full(6, 0.5)
    a = t.nearfield(w.kd, w.khat, w.e01, P, ext, want=("E_sca", "B_sca"))
    ref = O.nearfield(w.occ, w.comp, w.m, w.kd, w.khat[0], w.e01[0], "CM", P[0], ext)
    for k in ("E_sca", "B_sca"):
        got, want = a[k][0], np.asarray(ref[k]).reshape(a[k][0].shape)
        assert np.abs(got - want).max() <= 1e-9 * np.abs(want).max(), k
    t.close()
