"""FP32C gradients keep the rounding of the FP32 face states.

The inflow-speed gradient of a random adjoint is a sum over the inflow plane
whose terms nearly cancel. The FP32 rounding of the face values (WENO5, the
half-space series, the t1 pass) enters it through the curvature of the WENO
weights with 3e-6 to 5e-6 of its root mean square, so a change of rounding in
one of these kernels moves single gradients by far more than their 32-bit
values hold. The values below are those of the five-point window form of WENO5
and of the truncated series.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

# U_inf gradients of seeds 0..7, by grid: one that keeps the face boxes of the
# three directions apart, one that runs direction by direction
UINF = {
    (96, 48, 48): [-4.318608548e+00, -3.717045188e+01, -6.260616960e+00, 2.862408585e+01, -1.486750546e+01, 1.583661494e+01,
                   2.352703015e+01, -2.927489310e-01],
    (144, 72, 67): [-6.401728031e+01, -1.195229691e+01, -2.208451133e+01, 1.946351403e+01, -8.084702973e+01, 9.844088884e+01,
                    -6.618839858e+01, 4.258967605e+01],
}


def gradients(n):
    import torch
    from paper_2603_11102_gb300 import gks
    from paper_2603_11102_gb300 import workloads as WL

    w = WL.alm_rotor((n[0], 8, 8))
    w.n = n
    w.faces = [w.faces[0]] + [WL.uniform_faces(f[0], f[-1], k) for f, k in zip(w.faces[1:], n[1:])]
    w.state0 = None
    w.dt_fixed = 0.4 * min(float(np.min(np.diff(f))) for f in w.faces) / (1.2 * w.u_ref + w.u_ref / w.mach)
    g = gks.Grid.from_workload(w, precision="fp32c")
    g.set_adjoint_precision("fp32")
    tapes, scratch = [g.adjoint_tape() for _ in range(2)], g.adjoint_scratch()
    out = []
    for seed in range(8):
        rng = np.random.default_rng(seed)
        Q = np.zeros((4, n[2], n[1], n[0]))
        Q[0], Q[1] = 1.0, 1.0
        Q += np.array([1e-3, 0.02, 0.02, 0.02])[:, None, None, None] * rng.uniform(-1.0, 1.0, Q.shape)
        lam = torch.tensor(rng.standard_normal(Q.shape), dtype=torch.float64, device="cuda")
        g.set_state_tensor(torch.tensor(Q, dtype=torch.float64, device="cuda"))
        g.set_time(0.01 * seed)
        for tape in tapes:
            g.step_record(tape)
        gu, gs = 0.0, np.zeros(w.rotors[0].n_blades * w.rotors[0].r.size)
        for k, tape in enumerate(reversed(tapes)):
            lam, gun = g.step_reverse(tape, scratch, lam, 1.0 if k == 0 else 0.0, gs)
            gu += gun
        out.append(gu)
    g.close()
    return np.array(out)


@pytest.mark.parametrize("n", list(UINF))
def test_inflow_speed_gradient_keeps_its_rounding(n):
    """Within 2^-19 of the root mean square over the seeds: five times the 4e-7
    rms that a flux of another operation order and the FP32 reverse's own
    rounding come to, half of what another form of the face state comes to."""
    ref = np.array(UINF[n])
    got = gradients(n)
    assert np.max(np.abs(got - ref)) <= 2.0 ** -19 * np.sqrt(np.mean(ref ** 2)), (got, ref)
