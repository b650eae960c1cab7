"""Which actuator points reach a cell is decided as in FP64 for rotors whose
radius is many kernel widths, where the FP32 hub-relative coordinates of the
projection's screen are coarse against the cut."""
import math

import numpy as np
import pytest

from paper_2603_11102_gb300 import workloads as WL

from _setup import oracle_from_workload, rel_linf

H = 2.0 ** -12   # cell width; eps = 2 H, radius 1: R / eps = 1024
N = (20, 40, 40)
AZIMUTH = 0.6


def tip_workload(seed):
    """The last six kernel widths of one long blade, on a grid around them
    (faces at whole multiples of H, so that the widths are equal)."""
    eps = 2.0 * H
    rng = np.random.default_rng(seed)
    r = np.sort(1.0 - 6.0 * eps * rng.random(400))
    mid = [0.3 * H, (1.0 - 3.0 * eps) * math.cos(AZIMUTH), (1.0 - 3.0 * eps) * math.sin(AZIMUTH)]
    faces = [H * (math.floor(m / H) - n // 2 + np.arange(n + 1)) for m, n in zip(mid, N)]
    # at rest relative to the blade but for the axial flow: the azimuth stays
    rot = WL.Rotor(1, r, np.full(r.size, 1e-3), np.full(r.size, 1.2), np.full(r.size, eps), (0.0, 0.0, 0.0), 1e-9,
                   AZIMUTH, 1.0, eps)
    Q = np.zeros((4, N[2], N[1], N[0]))
    Q[0], Q[1] = 1.0, 1.0
    Q[1:] += 0.01 * (2.0 * rng.random(Q[1:].shape) - 1.0)
    return WL.Workload("blade-tip", N, faces, 0.1, 1.0, 1e-6, [(3, 4), (4, 4), (4, 4)], cfl=0.5,
                       inflow=(1.0, 1.0, 0.0, 0.0), state0=Q, rotors=[rot])


def screened(w, margin):
    """Points inside the cut that an FP32 screen with this relative margin drops."""
    rot, f = w.rotors[0], np.float32
    X = np.stack([np.zeros_like(rot.r), rot.r * math.cos(AZIMUTH), rot.r * math.sin(AZIMUTH)], axis=1)
    z, y, x = np.meshgrid(*[c[0] + (np.arange(c.size - 1) + 0.5) * H for c in reversed(w.faces)], indexing="ij")
    P = np.stack([x, y, z], axis=-1).reshape(-1, 3)
    cut, n = 3.0 * rot.eps, 0
    for p in X:
        inside = np.sqrt(((P - p) ** 2).sum(1)) <= cut
        d = P.astype(f) - p.astype(f)
        s2 = d[:, 0] * d[:, 0] + d[:, 1] * d[:, 1] + d[:, 2] * d[:, 2]
        n += int((inside & (s2 > f(cut * cut) * f(1.0 + margin))).sum())
    return n


@pytest.mark.parametrize("seed", [0])
def test_fixed_margin_drops_points(seed):
    """1e-5 is too narrow here; twice the rounding bound is not."""
    w = tip_workload(seed)
    ratio = w.rotors[0].r.max() / (3.0 * w.rotors[0].eps)
    assert screened(w, 1e-5) > 0
    assert screened(w, max(1e-5, 5e-7 * (ratio + 2.0))) == 0


@pytest.mark.gpu
@pytest.mark.parametrize("arith", ["fp64", "ds"])
@pytest.mark.parametrize("seed", [0])
def test_long_blade_projection_is_decided_in_fp64(seed, arith):
    """A point just inside the cut carries exp(-9) of its force: 1e-7 of the
    state here, against the 1e-12 bar of an FP64 step."""
    from paper_2603_11102_gb300 import gks

    w = tip_workload(seed)
    o = oracle_from_workload(w)
    o.step(1)
    g = gks.Grid.from_workload(w, precision="fp64")
    g.set_fp64_arithmetic(arith)
    g.step(1)
    assert rel_linf(g.get_state(), o.get_state()) <= 1e-12
    g.close()
