"""Schedules saved in the file that DDA_TUNE_FILE names (read once per process, so each
step is a process of its own)."""
import json
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

# autotunes a target for one right-hand side; prints the schedules and the errors of the
# products against FP64 with the default schedule
STEP = """
import json, sys
import numpy as np
from dda_inputs import targets as tg
from paper_1305_6497_gb300 import binding as B
occ, comp = tg.rect_prism(*map(int, sys.argv[1:4]))
t = B.Target(occ, comp, [1.5 + 0.1j], method="CM")
rng = np.random.default_rng(2)
x = rng.standard_normal((t.num_dipoles, 3)) + 1j * rng.standard_normal((t.num_dipoles, 3))
ref = t.matvec(0.4, x)
sched = t.autotune(0.4, 1)
err = {p: float(np.abs(t.matvec(0.4, x, precision=p) - ref).max() / np.abs(ref).max())
       for p in ("fp32", "fp64")}
print(json.dumps([sched, err]))
"""


def _step(path, shape):
    r = subprocess.run([sys.executable, "-c", STEP, *map(str, shape)], cwd=ROOT, text=True,
                       capture_output=True, env=dict(os.environ, DDA_TUNE_FILE=str(path)))
    assert r.returncode == 0, r.stderr
    return json.loads(r.stdout.strip().splitlines()[-1])


def _edit(path, change):
    """Rewrite the FP32 line's values."""
    out = []
    for line in path.read_text().splitlines():
        key, vals = line.split(" :")
        if "f32" in key:
            line = key + " : " + " ".join(map(str, change([int(v) for v in vals.split()])))
        out.append(line)
    path.write_text("\n".join(out) + "\n")


# 5 sites: a transform length of 9, which no register plan covers
@pytest.mark.parametrize("shape,kind", [((5, 16, 16), 16), ((16, 5, 16), 32), ((5, 5, 16), 48),
                                        ((16, 16, 5), 8), ((16, 16, 5), 9), ((16, 16, 16), 15)])
def test_an_entry_the_target_cannot_run_is_timed_anew(tmp_path, shape, kind):
    path = tmp_path / "tune.txt"
    first, err = _step(path, shape)
    assert max(err.values()) <= 4e-6
    _edit(path, lambda v: v[:4] + [kind] + v[5:])
    again, err = _step(path, shape)
    assert max(err.values()) <= 4e-6
    assert again["fp32"]["z_stage_ghat"] != kind
    assert again["fp64"] == first["fp64"]
    assert len(path.read_text().splitlines()) == 3


def test_an_entry_the_target_can_run_is_used(tmp_path):
    path = tmp_path / "tune.txt"
    _step(path, (13, 16, 16))
    # three lines per CTA, which the tuner never tries
    _edit(path, lambda v: [3] + v[1:4] + [v[4] & ~16] + v[5:])
    again, err = _step(path, (13, 16, 16))
    assert again["fp32"]["x_lines"] == 3 and not again["fp32"]["z_stage_ghat"] & 16
    assert max(err.values()) <= 4e-6
    assert len(path.read_text().splitlines()) == 2


def test_an_entry_of_earlier_kernels_is_timed_anew(tmp_path):
    """Lines without a version were timed before there were register passes."""
    path = tmp_path / "tune.txt"
    old = "f32 13 16 16 25 32 32 1 : 3 16 4 13 0 128 128 128\n"
    path.write_text(old)
    sched, err = _step(path, (13, 16, 16))
    assert sched["fp32"]["x_lines"] != 3
    assert max(err.values()) <= 4e-6
    assert path.read_text().startswith(old) and len(path.read_text().splitlines()) == 3
    again, _ = _step(path, (13, 16, 16))
    assert again == sched and len(path.read_text().splitlines()) == 3
