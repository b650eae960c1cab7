"""The FP64 totals keep 64 bits for densities of any size."""
import numpy as np
import pytest

from _setup import smooth_workload

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("exponent", [-120, -80, -75, -74, -30, 0, 90, 120])
def test_kinetic_energy_of_small_and_large_densities(exponent):
    """24 equal cells whose density has ones in all the bits that its FP32 part
    drops: the energy's quotient to 16 roundings (a quotient from the reciprocal
    of that part alone would be off by 2^-46, 128 roundings)."""
    from paper_2603_11102_gb300 import gks
    n = (4, 3, 2)
    w = smooth_workload(n, [(0, 0)] * 3, faces=[np.arange(k + 1.0) for k in n])
    rho = float(2 ** 52 + 2 ** 29 - 1) * 2.0 ** (exponent - 52)
    w.state0 = np.empty((4, n[2], n[1], n[0]))
    w.state0[0], w.state0[1:] = rho, 0.25 * rho
    g = gks.Grid.from_workload(w, precision="fp64")
    want = 24 * 0.5 * 3 * (0.25 * rho) * 0.25
    assert abs(float(g.diagnostics()[4]) / want - 1.0) <= 16 * 2.0 ** -53
    g.close()
