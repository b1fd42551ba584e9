"""Near field on boxes whose planes mostly hold no dipoles.

The forward x and y passes leave out the planes without dipoles.  The cases put
the target's planes first, last and in the middle, with rows per CTA that run
over several planes and over a component's end; the last one has no plane
without.  Compared with the oracle's direct sums over the same (arbitrary)
dipoles: a sum of N terms against an FFT convolution in FP64, to 1e-11 of the
largest value (about 50 log2(512) eps).
"""
import numpy as np
import pytest

from oracle import dda as O

pytestmark = pytest.mark.gpu

CASES = [
    (4, 1, 1, [0, 0, 0, 0, 7, 0]),
    (3, 2, 1, [0, 0, 0, 0, 0, 9]),
    (5, 7, 2, [0.4, 0.4, 0.3, 0.15, 3, 4]),
    (9, 1, 3, [0.5, 0.5, 2, 0, 1, 1]),
    (16, 9, 4, [0, 0, 1, 1, 3, 2]),
    (6, 5, 3, [0.5, 0, 0, 0.4, 0, 0]),
]


@pytest.mark.parametrize("nx,ny,nz,ext", CASES)
def test_planes_without_dipoles(nx, ny, nz, ext):
    from paper_1305_6497_gb300 import binding as B
    rng = np.random.default_rng(nx + 10 * ny + 100 * nz)
    occ = np.ones((nz, ny, nx), np.uint8)
    m, kd = 1.5 + 0.1j, 0.4
    khat, e1 = np.array([0.36, 0.48, 0.8]), np.array([0.8, -0.6, 0.0], np.complex128)
    n = nx * ny * nz
    P = rng.standard_normal((2, n, 3)) + 1j * rng.standard_normal((2, n, 3))
    t = B.Target(occ, None, [m], method="LDR")
    for _ in range(2):  # the second call finds the first one's scratch
        out = t.nearfield(kd, khat[None], e1[None], P, ext, want=("E_sca", "E_macro", "B_sca"))
    t.close()
    for r, e in enumerate(O.polarization_pair(khat, e1)):
        ref = O.nearfield(occ, occ, [m], kd, khat, e, "LDR", P[r], ext)
        for k in ("E_sca", "E_macro", "B_sca"):
            err = np.abs(out[k][r] - ref[k]).max() / np.abs(ref[k]).max()
            assert err < 1e-11, (k, r, err)
