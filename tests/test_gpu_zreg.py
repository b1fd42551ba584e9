"""The two-step register passes (z kind 8, + 16 for the x and + 32 for the y passes; the FP32 default):
the same product as the general kernels and the FP64 one, at the edges of their
plans."""
import numpy as np
import pytest

from dda_inputs import targets as tg
from dda_inputs import workloads as W
from oracle import dda as O

pytestmark = pytest.mark.gpu

# z extents at both ends of a plan (full lines, and the shortest box of a length),
# plans whose first step leaves part of a warp idle (9, 11, 26), 4 and 8 column
# tiles, odd Lx (no asynchronous copies), fewer columns than a tile, odd Ly
SHAPES = [(2, 3, 9), (3, 5, 11), (13, 8, 12), (8, 13, 16), (14, 9, 26), (9, 11, 32), (10, 7, 33),
          (7, 10, 64), (13, 6, 76), (5, 9, 96), (12, 5, 97), (6, 7, 128), (3, 9, 129),
          (10, 4, 144), (5, 6, 168), (13, 4, 162), (4, 6, 200), (5, 4, 216), (4, 5, 225),
          (6, 4, 251), (5, 5, 256),
          # odd z lengths 15 .. 225, both ends of their boxes, with and without copies
          (9, 3, 7), (7, 5, 8), (13, 4, 13), (10, 3, 14), (9, 5, 21), (14, 4, 23), (6, 7, 37),
          (37, 3, 38), (11, 9, 41), (5, 4, 65), (13, 3, 68), (9, 4, 109), (3, 5, 113)]


@pytest.mark.parametrize("shape", SHAPES)
def test_register_z_kernel_matches(shape):
    from paper_1305_6497_gb300 import binding as B
    occ, comp = tg.rect_prism(*shape)
    flat, pos = O.site_positions(occ)
    x = O.box_to_sites(W.random_polarization(occ, 11)[0], flat)
    t = B.Target(occ, comp, [1.5 + 0.1j], method="GKDLDR")
    kh, e = np.array([0.36, 0.48, 0.8]), [0.8, -0.6, 0]
    sch = t.schedule("fp32") if t.matvec(0.4, x, kh, e, "fp32") is not None else None
    assert sch["z_stage_ghat"] & 15 == 8
    y8 = t.matvec(0.4, x, kh, e, "fp32")
    y64 = t.matvec(0.4, x, kh, e, "fp64")
    t.set_schedule(dict(sch, z_tile=4, z_pitch=13, z_stage_ghat=0, z_threads=128), "fp32")
    y0 = t.matvec(0.4, x, kh, e, "fp32")
    # six transforms of at most nine radix-2 levels, each rounding to 2^-24
    tol = 6 * 9 * 2.0 ** -24
    top = np.abs(y64).max()
    assert np.abs(y8 - y64).max() <= tol * top
    assert np.abs(y8 - y0).max() <= 2 * tol * top
    rows = np.arange(0, len(flat), max(1, len(flat) // 40))
    ainv = O.site_alpha_inverse(comp.reshape(-1)[flat], [1.5 + 0.1j], "GKDLDR", 0.4, kh)
    ref = O.matvec_direct(x, pos, ainv, 0.4, "GKDLDR", rows=rows)
    assert np.abs(y8[rows] - ref).max() <= tol * top
    t.set_schedule(sch, "fp32")
    assert t.schedule("fp32")["z_stage_ghat"] & 15 == 8
    assert np.array_equal(t.matvec(0.4, x, kh, e, "fp32"), y8)
    t.close()


# x extents at the ends of the plans, several rows per warp, a last warp with fewer
# rows than it holds, one composition byte per site unaligned
X_SHAPES = [(9, 3, 2), (10, 5, 3), (11, 4, 5), (15, 7, 3), (17, 5, 4), (26, 3, 5), (28, 5, 3),
            (33, 6, 3), (42, 3, 4), (51, 4, 3), (64, 7, 5), (73, 3, 2), (82, 5, 3), (91, 2, 5),
            (101, 3, 4), (114, 4, 3), (126, 3, 5), (129, 5, 2), (136, 3, 3), (145, 2, 4),
            (151, 3, 3), (161, 3, 2), (168, 2, 3), (189, 3, 3), (193, 2, 2), (204, 3, 2),
            (217, 2, 3), (226, 3, 2), (251, 2, 3), (256, 3, 3),
            (7, 5, 3), (8, 3, 2), (13, 4, 5), (14, 3, 3), (21, 5, 2), (23, 3, 4), (37, 4, 3),
            (38, 3, 5), (41, 7, 3), (65, 3, 2), (68, 2, 3), (109, 3, 3), (113, 2, 2)]


@pytest.mark.parametrize("nx,ny", [(3, 9), (2, 10), (9, 11), (5, 16), (17, 26), (9, 33),
                                   (4, 64), (5, 73), (9, 82), (3, 101), (17, 128), (3, 129),
                                   (5, 136), (2, 145), (9, 150), (3, 168), (2, 189), (5, 193),
                                   (9, 204), (2, 225), (3, 240), (9, 251), (2, 256),
                                   (3, 7), (17, 8), (2, 13), (9, 14), (5, 21), (4, 23), (9, 37),
                                   (2, 38), (17, 41), (3, 65), (9, 68), (2, 109), (5, 113)])
def test_register_y_passes_match(nx, ny):
    """Column tiles with one column, a partial tile and several tiles."""
    from paper_1305_6497_gb300 import binding as B
    occ, comp = tg.rect_prism(nx, ny, 4)
    flat, pos = O.site_positions(occ)
    x = O.box_to_sites(W.random_polarization(occ, 13)[0], flat)
    t = B.Target(occ, comp, [1.5 + 0.1j], method="CM")
    y = t.matvec(0.4, x, precision="fp32")
    s = t.schedule("fp32")
    assert s["z_stage_ghat"] & 32
    y64 = t.matvec(0.4, x, precision="fp64")
    tol = 6 * 9 * 2.0 ** -24
    top = np.abs(y64).max()
    assert np.abs(y - y64).max() <= tol * top
    for kind in (s["z_stage_ghat"] - 32, s["z_stage_ghat"] & 15):
        t.set_schedule(dict(s, z_stage_ghat=kind), "fp32")
        assert np.abs(t.matvec(0.4, x, precision="fp32") - y).max() <= 2 * tol * top
    t.close()


@pytest.mark.parametrize("shape", X_SHAPES)
def test_register_x_passes_match(shape):
    from paper_1305_6497_gb300 import binding as B
    w = W.two_material_brick(*shape, seed=5)
    flat, pos = O.site_positions(w.occ)
    x = O.box_to_sites(W.random_polarization(w.occ, 12)[0], flat)
    kh, e = np.array([0.36, 0.48, 0.8]), [0.8, -0.6, 0]
    t = B.Target(w.occ, w.comp, w.m, method="GKDLDR")
    y = t.matvec(0.4, x, kh, e, "fp32")
    s = t.schedule("fp32")
    assert s["z_stage_ghat"] & 16
    y64 = t.matvec(0.4, x, kh, e, "fp64")
    tol = 6 * 9 * 2.0 ** -24
    top = np.abs(y64).max()
    assert np.abs(y - y64).max() <= tol * top
    t.set_schedule(dict(s, z_stage_ghat=s["z_stage_ghat"] - 16), "fp32")
    assert not t.schedule("fp32")["z_stage_ghat"] & 16
    assert np.abs(t.matvec(0.4, x, kh, e, "fp32") - y).max() <= 2 * tol * top
    # the fused prologues and epilogues of every method against the general passes
    for solver in ("bicgstab", "qmr", "bicgstab2", "gpbicg", "petrkp"):
        q = []
        for z in (s["z_stage_ghat"], s["z_stage_ghat"] - 16):
            t.set_schedule(dict(s, z_stage_ghat=z), "fp32")
            q.append(t.solve(0.4, kh, e, npol=2, tol=1e-9, max_iter=4000, precision="fp32_refined",
                             solver=solver))
        assert q[0]["status"] == B.DDA_OK
        assert np.abs(q[0]["P"] - q[1]["P"]).max() <= 1e-7 * np.abs(q[1]["P"]).max(), solver
    t.close()


def test_batches_and_frozen_right_hand_sides():
    """Several right-hand sides, some converged before others, with one and with
    several passes per CTA."""
    from paper_1305_6497_gb300 import binding as B
    for shape, n_orient in (((9, 12, 11), 3), ((40, 64, 64), 5)):
        w = W.small_ellipsoid(*shape, m=1.5 + 0.1j, kd=0.3, method="LDR", n_orient=n_orient, seed=9)
        t = B.Target(w.occ, w.comp, w.m, method="LDR")
        kw = dict(yhat=w.yhat, npol=2, tol=1e-9, precision="fp32_refined")
        a = t.solve(w.kd, w.khat, w.e01, **kw)
        assert t.schedule("fp32")["z_stage_ghat"] & 15 == 8 and a["status"] == B.DDA_OK
        t.set_schedule(dict(t.schedule("fp32"), z_tile=4, z_pitch=13, z_stage_ghat=0,
                            z_threads=128), "fp32")
        b = t.solve(w.kd, w.khat, w.e01, **kw)
        assert np.all(np.abs(b["Qext"] / a["Qext"] - 1) < 1e-7)
        assert np.abs(b["P"] - a["P"]).max() <= 1e-7 * np.abs(a["P"]).max()
        t.close()


def test_register_z_kernel_is_refused_where_it_has_no_plan():
    from paper_1305_6497_gb300 import binding as B
    for nz in (5, 125, 165):       # no two-factor plan, two rows beyond the box
        occ, comp = tg.rect_prism(4, 3, nz)
        t = B.Target(occ, comp, [1.5 + 0.1j], method="CM")
        x = np.ones((t.num_dipoles, 3), np.complex128)
        y = t.matvec(0.3, x, precision="fp32")
        assert np.abs(y - t.matvec(0.3, x, precision="fp64")).max() <= 4e-6 * np.abs(y).max()
        s = t.schedule("fp32")
        assert s["z_stage_ghat"] & 15 != 8
        with pytest.raises(B.DDAError):
            t.set_schedule(dict(s, z_tile=8, z_pitch=24, z_stage_ghat=8), "fp32")
        t.close()
