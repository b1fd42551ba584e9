"""Device memory that scattering directions add to a solve (the host-only estimate; CPU).

A direction may take its phase tables (16 bytes a site of each axis), its unit vector,
its sums and at most 304 blocks of partial sums (two right-hand sides of six), however
many columns the box has."""
import numpy as np
import pytest


@pytest.mark.parametrize("shape", [(1024, 1024, 8), (512, 512, 64), (600, 700, 3), (256, 256, 256)])
@pytest.mark.parametrize("ndir", [350, 65341, 1000000])
def test_directions_take_a_bounded_amount(shape, ndir):
    from paper_1305_6497_gb300 import build
    build.build()
    from paper_1305_6497_gb300 import binding as B
    nx, ny, nz = shape
    occ = np.zeros((nz, ny, nx), np.uint8)
    occ[0, 0, 0] = 1
    args = (occ, 1, "LDR", 0.3, np.array([[1.0, 0, 0]]), np.array([[0, 1.0 + 0j, 0]]))
    none = B.dda_estimate_solve_bytes(*args)
    some = B.dda_estimate_solve_bytes(*args, dirs=np.zeros((ndir, 2)))
    per_direction = 16 * (nx + ny + nz) + 24 + 96 + 12 * 304 * 8
    assert none <= some <= none + (ndir + 1) * per_direction
