"""Scattering amplitudes against the oracle's sum over the returned dipoles, for
direction counts that fill and do not fill a thread's directions, one and two
polarizations, columns fewer and more than a block, and vacant planes."""
import numpy as np
import pytest

from dda_inputs import targets as tg
from dda_inputs import workloads as W
from oracle import dda as O

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("npol", [1, 2])
@pytest.mark.parametrize("ndir", [0, 1, 2, 3, 4, 6, 8, 41])
@pytest.mark.parametrize("shape", [(3, 2, 5), (18, 17, 9), (40, 20, 1)])
def test_amplitudes_match_the_sum_over_dipoles(shape, ndir, npol):
    from paper_1305_6497_gb300 import binding as B
    occ, comp = tg.ellipsoid(*shape)
    if shape[2] == 9:
        occ[3:5] = 0        # two vacant planes
        comp[3:5] = 0
    kh, yh, e1 = W._lab_incidence([(0.4, 0.9, 1.3), (1.1, 0.2, 2.0)])
    rng = np.random.default_rng(ndir + 1)
    dirs = np.stack([rng.uniform(0, np.pi, ndir), rng.uniform(0, 2 * np.pi, ndir)], 1)
    kd = 0.3
    t = B.Target(occ, comp, [1.4 + 0.05j], method="LDR")
    o = t.solve(kd, kh, e1, yhat=yh, npol=npol, tol=1e-10, dirs=dirs)
    _, pos = O.site_positions(occ)
    for i in range(2):
        z = np.cross(kh[i], yh[i])
        for d, (th, ph) in enumerate([(0.0, 0.0)] + [tuple(v) for v in dirs]):
            n = kh[i] * np.cos(th) + (yh[i] * np.cos(ph) + z * np.sin(ph)) * np.sin(th)
            eth = -kh[i] * np.sin(th) + (yh[i] * np.cos(ph) + z * np.sin(ph)) * np.cos(th)
            eph = z * np.cos(ph) - yh[i] * np.sin(ph)
            for l in range(npol):
                F = np.exp(-1j * kd * pos @ n) @ o["P"][i * npol + l]
                big = kd ** 3 * np.abs(o["P"][i * npol + l]).sum()
                # FP64 sums of N terms
                assert abs(o["famp"][i, d, 0, l] - kd ** 3 * eth @ F) <= 1e-13 * big
                assert abs(o["famp"][i, d, 1, l] - kd ** 3 * eph @ F) <= 1e-13 * big
    t.close()


@pytest.mark.parametrize("ndir", [2093055, 2100001])
def test_phase_tables_of_more_than_int_max_entries(ndir):
    """A line of 1024 sites, whose phase tables have 1026 entries a direction: just
    below 2^31 entries in all (where a 32-bit index passes 2^31 in its last stride) and
    above, in hundreds of chunks.  The directions repeat, so every amplitude is one of
    the first 4096."""
    from paper_1305_6497_gb300 import binding as B
    occ, comp = tg.rect_prism(1024, 1, 1)
    kh, yh, e1 = W._lab_incidence([(0.4, 0.9, 1.3)])
    rng = np.random.default_rng(8)
    some = np.stack([rng.uniform(0, np.pi, 4096), rng.uniform(0, 2 * np.pi, 4096)], 1)
    dirs = np.resize(some, (ndir, 2))
    t = B.Target(occ, comp, [1.3 + 0.05j], method="CM")
    kw = dict(yhat=yh, npol=1, tol=1e-8)
    o = t.solve(0.3, kh, e1, dirs=dirs, **kw)
    f = o["famp"][0, 1:, :, 0]
    first = t.solve(0.3, kh, e1, dirs=some[:64], **kw)
    t.close()
    big = 0.3 ** 3 * np.abs(o["P"]).sum()
    assert np.abs(f[:64] - first["famp"][0, 1:, :, 0]).max() <= 1e-13 * big
    for k in range(0, ndir, 4096):
        part = f[k:k + 4096]
        np.testing.assert_array_equal(part, f[:len(part)])
