"""The launches of grids whose face boxes are too large to be kept apart: one
direction after the other, FP32C z faces fused with the stage update. At a
size that divides no tile (32 x 8 faces; 83 = 10 x 8 + 3), against the oracle
and in the bounds-checked build, with the FP32C recorded step and its reverse."""
import os
import subprocess
import sys

import numpy as np
import pytest

from paper_2603_11102_gb300 import workloads as WL

from _setup import oracle_from_workload, rel_linf, smooth_workload

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
N = (101, 83, 77)
TOL = {"fp64": 1e-12, "fp32c": 1e-5, "fp64ds": 1e-12}


@pytest.fixture(scope="module")
def case():
    w = smooth_workload(N, [(3, 4), (2, 1), (0, 0)], seed=5)
    w.inflow = (1.0, 0.3, 0.0, 0.0)
    o = oracle_from_workload(w)
    o.step(1)
    return w, o.get_state()


def face_state_launches(g):
    """Face-state launches of a step: 2 with all directions together, else 6."""
    g.profile_enable(False)
    g.step(1)
    return g.profile_read()["launches"]["face_eq"]


@pytest.mark.parametrize("precision", list(TOL))
def test_ragged_large_grid(case, precision):
    from paper_2603_11102_gb300 import gks
    w, ref = case
    g = gks.Grid.from_workload(w, precision="fp32c" if precision == "fp32c" else "fp64")
    if precision == "fp64ds":
        g.set_fp64_arithmetic("ds")
    assert face_state_launches(g) == 6
    assert rel_linf(g.get_state(), ref) <= TOL[precision]
    g.close()


@pytest.mark.parametrize("precision", ["fp32c", "fp64"])
@pytest.mark.parametrize("n,launches", [((96, 80, 80), 6), ((64, 80, 80), {"fp32c": 2, "fp64": 6}), ((32, 80, 80), 2)],
                         ids=lambda v: "x".join(map(str, v)) if isinstance(v, tuple) else "")
def test_which_launches_a_size_takes(precision, n, launches):
    """The sizes that tests of equal results on both paths rely on."""
    from paper_2603_11102_gb300 import gks
    w = smooth_workload(n, [(0, 0)] * 3, seed=1)
    g = gks.Grid.from_workload(w, precision=precision)
    assert face_state_launches(g) == (launches if isinstance(launches, int) else launches[precision])
    g.close()


CHILD = r"""
import os, sys
import numpy as np
sys.path.insert(0, {root!r})
sys.path.insert(0, os.path.join({root!r}, "tests"))
import torch
from paper_2603_11102_gb300 import build, gks, workloads as WL
build.build(debug=os.environ.get("GKS_DEBUG_BOUNDS") == "1")
gks.load()
out = {{}}
for n in ({n!r}, (45, 30, 27)):
    for prec in ("fp32c", "fp64"):
        w = WL.alm_rotor(n, n_pts=10)
        w.dt_fixed = 1e-3
        w.state0 = WL.perturbed(w, 0.02, seed=6)
        g = gks.Grid.from_workload(w, precision=prec)
        g.step(1)
        if prec == "fp32c":
            tape = g.adjoint_tape()
            g.step_record(tape)
            gs = np.zeros(30)
            lam1 = np.random.default_rng(2).standard_normal(w.state0.shape)
            lam, gu = g.step_reverse(tape, g.adjoint_scratch(), torch.tensor(lam1, dtype=torch.float64, device="cuda"),
                                     0.5, gs)
            out["lam%d" % n[0]], out["gu%d" % n[0]], out["gs%d" % n[0]] = lam.cpu().numpy(), np.array([gu]), gs
        out["%s%d" % (prec, n[0])] = g.get_state()
        g.close()
np.savez({path!r}, **out)
"""


def run_child(tmp_path, debug):
    path = str(tmp_path / ("debug.npz" if debug else "plain.npz"))
    env = dict(os.environ, GKS_DEBUG_BOUNDS="1" if debug else "0")
    r = subprocess.run([sys.executable, "-c", CHILD.format(root=ROOT, path=path, n=N)], env=env, capture_output=True,
                       text=True, timeout=1500)
    assert r.returncode == 0, r.stderr[-3000:]
    return dict(np.load(path))


def test_bounds_checked_build_on_both_paths(tmp_path):
    plain, debug = run_child(tmp_path, False), run_child(tmp_path, True)
    assert set(plain) == set(debug) and len(plain) == 10
    for k in plain:
        scale = max(float(np.max(np.abs(plain[k]))), 1e-300)
        assert np.max(np.abs(plain[k] - debug[k])) <= 1e-12 * scale, k
