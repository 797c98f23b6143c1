"""Which tile a context runs: the small one by size alone, the default one when tuning is off, and statistics that the
tuner leaves alone."""
import json
import os
import subprocess
import sys

import numpy as np
import pytest

from paper_2004_08503_gb300 import inputs, sidp

pytestmark = pytest.mark.gpu
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def _child(code, **env):
    """The tuner's table lives as long as the process: a fresh one per case."""
    r = subprocess.run([sys.executable, "-c", code], cwd=ROOT, env={**os.environ, **env}, capture_output=True, text=True, timeout=600)
    assert r.returncode == 0, r.stderr[-2000:]
    return json.loads(r.stdout.strip().splitlines()[-1])


def test_a_stored_choice_of_the_small_tile_is_passed_over(tmp_path):
    """Index 3 in a tuning file (older builds: a large tile) does not put a mesh of 256 default tiles on the
    small one; the file's other lines hold, and the file that is written back names no 3."""
    f = tmp_path / "tune"
    f.write_text("2 3 1 3\n2 4 1 2\n")
    code = """
import json
from paper_2004_08503_gb300 import inputs, sidp
out = []
for p in (3, 4):
    sv = sidp.Solver(law="euler", p=p, nx=64, ny=64, precision="mixed", bc=("outflow",) * 4)
    sv.set_state(inputs.four_quadrant(*sv.node_coords(), 0))
    sv.set_stats(False)
    sv.step(12)
    out.append(sv.tile()[2])
print(json.dumps(out))
"""
    tiles = _child(code, SIDP_TUNE_FILE=str(f))
    assert tiles[0] != 3 and tiles[1] == 2
    assert all(line.split()[3] != "3" for line in f.read_text().splitlines())


@pytest.mark.parametrize("cfg", [dict(limiter="none"), dict(limiter="lo"), dict(limiter="subcell"), dict(limiter="elementwise"),
                                 dict(limiter="subcell", smoothness=dict(gmin=-0.5, gmax=1.6))])
def test_no_tuning_keeps_the_default_tile_in_every_mode(cfg, monkeypatch):
    for off in (True, False):
        monkeypatch.setenv("SIDP_AUTOTUNE", "0" if off else "1")
        sv = sidp.Solver(law="euler", p=3, nx=6, ny=6, bc=("outflow",) * 4, **cfg)
        sv.set_state(inputs.four_quadrant(*sv.node_coords(), 0))
        sv.step(1)
        assert sv.tile()[2] == (0 if off or cfg["limiter"] == "elementwise" else 3)
        sv.close()


def test_the_statistics_are_the_runs_own():
    """One step whose tile is chosen by timing reports what the same step reports on that tile without timing: the
    candidates' launches leave no count and no maximum behind (every degree, so that each is timed once)."""
    code = """
import json
from paper_2004_08503_gb300 import inputs, sidp
keys = ("max_bound_violation", "max_entropy_violation", "rootfind_max_iters", "rootfind_cap_hits", "bound_nudges")
out = []
for prec in ("mixed", "fp64"):
    for p, n in ((1, 200), (2, 120), (3, 80), (4, 60), (5, 50), (6, 48), (7, 48)):
        runs, tile = [], None
        for pin in (False, True):
            sv = sidp.Solver(law="euler", p=p, nx=n, ny=n, precision=prec, bc=("outflow",) * 4)
            sv.set_state(inputs.four_quadrant(*sv.node_coords(), 2))
            if pin:
                sv.set_tile(tile)
            sv.step(1)
            tile = sv.tile()[2]
            d = sv.diag()
            runs.append([d[k] for k in keys])
            sv.close()
        assert tile != 3
        out.append([prec, p, runs])
print(json.dumps(out))
"""
    for prec, p, (timed, pinned) in _child(code):
        assert timed == pinned, (prec, p, timed, pinned)


@pytest.mark.parametrize("limiter,precision,tiles,small", [
    ("none", "fp64", (9, 9), True), ("none", "fp64", (9, 10), False), ("lo", "fp64", (9, 9), True), ("lo", "fp64", (10, 9), False),
    ("subcell", "fp64", (10, 20), True), ("subcell", "fp64", (11, 19), False), ("none", "mixed", (10, 10), True),
    ("subcell", "mixed", (10, 10), True), ("subcell", "mixed", (10, 11), False)])
def test_the_size_rule_of_the_small_tile(limiter, precision, tiles, small):
    """Meshes on each side of the rule's line (p = 3: default tiles of 4 x 4 elements)."""
    nx, ny = 4 * tiles[0], 4 * tiles[1]
    sv = sidp.Solver(law="euler", p=3, nx=nx, ny=ny, domain=(0.0, 1.0, 0.0, ny / nx), bc=("outflow",) * 4, limiter=limiter,
                     precision=precision)
    sv.set_state(inputs.four_quadrant(*sv.node_coords(), 0) if limiter != "none" else
                 np.repeat(inputs._cons(np.array([1.0]), np.array([0.1]), np.array([0.0]), np.array([1.0])), sv.N, axis=1))
    sv.step(1)
    assert (sv.tile()[2] == 3) == small
    sv.close()
