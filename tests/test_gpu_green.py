"""The Green transform built from the octant of offsets: FP64 products against the
direct sum on boxes with one-site axes, odd grid lengths and lines longer than a tile."""
import numpy as np
import pytest

from dda_inputs import targets as tg
from dda_inputs import workloads as W
from oracle import dda as O

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("method", ["CM", "FCD"])
@pytest.mark.parametrize("shape", [(1, 1, 9), (2, 1, 3), (1, 7, 1), (13, 2, 3), (2, 41, 3),
                                   (3, 2, 130), (130, 2, 1), (4, 130, 2), (9, 10, 11)])
def test_products_match_the_direct_sum(shape, method):
    from paper_1305_6497_gb300 import binding as B
    occ, comp = tg.rect_prism(*shape)
    flat, pos = O.site_positions(occ)
    x = O.box_to_sites(W.random_polarization(occ, 17)[0], flat)
    t = B.Target(occ, comp, [1.5 + 0.1j], method=method)
    ainv = O.site_alpha_inverse(comp.reshape(-1)[flat], [1.5 + 0.1j], method, 0.4)
    for kd in (0.4, 0.7, 0.4):     # the second and third reuse the workspace
        y = t.matvec(kd, x)
        ainv = O.site_alpha_inverse(comp.reshape(-1)[flat], [1.5 + 0.1j], method, kd)
        ref = O.matvec_direct(x, pos, ainv, kd, method)
        assert np.abs(y - ref).max() <= 1e-10 * np.abs(ref).max()
        for precision, tol in (("df64", 1e-10), ("fp32", 4e-6)):
            assert np.abs(t.matvec(kd, x, precision=precision) - ref).max() <= tol * np.abs(ref).max()
    t.close()
