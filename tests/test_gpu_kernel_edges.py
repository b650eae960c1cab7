"""Each kernel variant at the sizes where its split can go wrong: tile and
segment remainders of the face kernels, the FP64 composition of the
compensated state, the global reductions (equal and stretched widths, values
that are not finite), and the forcing kernels (more points than are staged at
once, a body box larger than one pass of the grid).

Tolerances: the states are held to the parity bars of the whole suite (1e-12
FP64 and double-single, 1e-5 FP32C); the sums to 64 roundings of the sum of
magnitudes (a column of 16, the columns of a thread, two trees of 8 and 10
levels)."""
import math

import numpy as np
import pytest

from paper_2603_11102_gb300 import workloads as WL

from _setup import oracle_from_workload, rel_linf, smooth_workload

pytestmark = pytest.mark.gpu

TOL = {"fp64": 1e-12, "fp32c": 1e-5, "fp64ds": 1e-12}


@pytest.fixture(scope="module")
def gks():
    from paper_2603_11102_gb300 import build, gks
    build.build()
    gks.load()
    return gks


def grid(gks, w, precision):
    g = gks.Grid.from_workload(w, precision="fp64" if precision == "fp64ds" else precision)
    if precision == "fp64ds":
        g.set_fp64_arithmetic("ds")
    return g


@pytest.mark.parametrize("n", [(1, 1, 1), (3, 1, 33), (33, 32, 5), (31, 34, 7), (65, 9, 36), (4, 70, 2), (129, 3, 11)],
                         ids=lambda n: "%dx%dx%d" % n)
def test_face_kernels_at_tile_and_segment_edges(gks, n):
    bc = [(0, 0), (0, 0), (0, 0)] if min(n) < 3 else [(2, 4), (0, 0), (1, 2)]
    w = smooth_workload(n, bc, seed=sum(n))
    o = oracle_from_workload(w)
    o.step(2)
    for precision in ("fp32c", "fp64", "fp64ds"):
        g = grid(gks, w, precision)
        g.step(2)
        assert rel_linf(g.get_state(), o.get_state()) <= TOL[precision], precision
        g.close()


@pytest.mark.parametrize("precision", ["fp64", "fp64ds"])
@pytest.mark.parametrize("n", [(40, 50, 61), (33, 71, 45)], ids=lambda n: "%dx%dx%d" % n)
def test_flux_tile_runs(gks, n, precision):
    # several tiles to a block: runs that start inside a row of tiles along t2
    # or pass from one row, plane or direction to the next
    w = smooth_workload(n, [(2, 4), (0, 0), (1, 2)], seed=sum(n))
    o = oracle_from_workload(w)
    o.step(2)
    g = grid(gks, w, precision)
    g.step(2)
    assert rel_linf(g.get_state(), o.get_state()) <= TOL[precision]
    g.close()


def raw_state(g):
    """The stored component arrays of a grid, (arrays, P2, P1, P0)."""
    import torch
    P0, P1, P2, eb, narr, stride, G = g.layout()
    a = g.state_buf.view(torch.float64 if eb == 8 else torch.float32)[:narr * stride].view(narr, stride)
    return a[:, :P0 * P1 * P2].view(narr, P2, P1, P0)[:, G:P2 - G, G:P1 - G, G:P0 - G]


def hi_lo_pairs(count, seed):
    """Float pairs: |lo| up to half an ulp of hi (ties, zeros, powers of two
    with lo of either sign, tiny lo), larger lo, and exponents at the ends."""
    rng = np.random.default_rng(seed)
    e = rng.integers(-126, 127, count)
    hi = np.ldexp(1.0 + rng.integers(0, 1 << 23, count) / float(1 << 23), e).astype(np.float32)
    hi[::3] = np.ldexp(1.0, e[::3]).astype(np.float32)
    hi *= rng.choice(np.array([-1, 1], np.float32), count)
    ulp = np.ldexp(1.0, np.frexp(np.abs(hi))[1] - 24)
    f = rng.uniform(-1, 1, count)
    f[1::7] = rng.choice([-1.0, 1.0, 0.5, -0.5, 0.0], f[1::7].size)
    f[2::7] *= np.ldexp(1.0, -rng.integers(0, 40, f[2::7].size))
    f[3::11] *= 8.0
    lo = (0.5 * ulp * f).astype(np.float32)
    hi[::29], lo[::29] = 0.0, 0.0
    lo[1::29] = 0.0
    return hi, lo


def test_fp32c_state_is_composed_exactly(gks):
    import torch
    n = (37, 18, 23)
    g = gks.Grid.from_workload(smooth_workload(n, [(0, 0)] * 3), precision="fp32c")
    hi, lo = hi_lo_pairs(4 * n[0] * n[1] * n[2], 5)
    hi, lo = hi.reshape(g.shape), lo.reshape(g.shape)
    r = raw_state(g)
    r[:4] = torch.from_numpy(hi).cuda()
    r[4:] = torch.from_numpy(lo).cuda()
    got = g.state_tensor().cpu().numpy()
    assert np.array_equal(got, hi.astype(np.float64) + lo.astype(np.float64))
    g.close()


@pytest.mark.parametrize("precision", ["fp64", "fp32c"])
@pytest.mark.parametrize("stretched", [False, True])
@pytest.mark.parametrize("n", [(3, 3, 3), (33, 9, 17), (40, 8, 16), (70, 21, 49)], ids=lambda n: "%dx%dx%d" % n)
def test_reductions_against_exact_sums(gks, precision, stretched, n):
    faces = [np.linspace(-0.7, 1.9, k + 1) for k in n]
    if stretched:
        faces[2] = WL.tanh_faces(n[2])
    w = smooth_workload(n, [(2, 2), (0, 0), (1, 1)], faces=faces, seed=3)
    g = gks.Grid.from_workload(w, precision=precision)
    Q = g.get_state()
    vol = np.einsum("k,j,i->kji", *[np.diff(f) for f in reversed(faces)])
    terms = [q * vol for q in Q] + [0.5 * (Q[1:] ** 2).sum(0) / Q[0] * vol]
    got = g.diagnostics()
    for t, x in zip(terms, got):
        assert abs(x - math.fsum(t.ravel())) <= 64 * 2.0 ** -53 * np.abs(t).sum()
    g.close()


@pytest.mark.parametrize("precision", ["fp64", "fp32c"])
def test_reductions_keep_values_that_are_not_finite(gks, precision):
    n = (10, 9, 20)
    for bad, want in ((np.inf, [np.inf] * 3), (np.nan, [np.nan] * 3)):
        w = smooth_workload(n, [(0, 0)] * 3)
        g = gks.Grid.from_workload(w, precision=precision)
        raw_state(g)[1, 4, 3, 2] = bad
        if precision == "fp32c":
            raw_state(g)[5, 4, 3, 2] = 0.0
        d = g.diagnostics()
        assert np.isfinite(d[[0, 2, 3]]).all()
        assert np.array_equal(d[[1, 4]], want[:2], equal_nan=True)
        g.close()
    # magnitudes whose squares and sums leave FP32's range
    w = smooth_workload(n, [(0, 0)] * 3)
    g = gks.Grid.from_workload(w, precision=precision)
    raw_state(g)[1] = 3e38
    if precision == "fp32c":
        raw_state(g)[5] = 0.0
    Q = g.get_state()
    vol = np.einsum("k,j,i->kji", *[np.diff(f) for f in reversed(w.faces)])
    d = g.diagnostics()
    assert abs(d[1] / math.fsum((Q[1] * vol).ravel()) - 1) <= 1e-14
    assert abs(d[4] / math.fsum((0.5 * (Q[1:] ** 2).sum(0) / Q[0] * vol).ravel()) - 1) <= 1e-14
    g.close()


@pytest.mark.parametrize("precision", ["fp32c", "fp64"])
@pytest.mark.parametrize("n_pts,n_blades", [(1, 1), (100, 3), (37, 7)])
def test_rotor_point_counts(gks, precision, n_pts, n_blades):
    n = (45, 26, 27)
    w = WL.alm_rotor(n, n_pts=n_pts)
    w.rotors = [WL.rotor_3x50(1.0, (0.0, 0.0, 0.0), 12.0 / n[0], n_pts=n_pts, n_blades=n_blades)]
    w.state0 = WL.perturbed(w, 0.02, seed=n_pts)
    o = oracle_from_workload(w)
    o.step(2)
    g = grid(gks, w, precision)
    g.step(2)
    assert rel_linf(g.get_state(), o.get_state()) <= TOL[precision]
    a, b = g.forces(0), o.forces(0)
    for key in ("thrust", "torque", "Fx", "Ft", "alpha", "phi"):
        assert rel_linf(np.asarray(a[key]), np.asarray(b[key])) <= 10 * TOL[precision], key
    g.close()


@pytest.mark.parametrize("precision", ["fp32c", "fp64"])
def test_body_box_larger_than_one_pass(gks, precision):
    # 110 x 72 x 72 box cells: more than 2048 blocks of 256
    n = (110, 72, 72)
    w = smooth_workload(n, [(4, 4), (2, 2), (2, 2)], faces=[np.linspace(0.0, 1.0, k + 1) for k in n])
    w.bodies = [WL.Body(np.array([[0.5, 0.5, 0.5], [0.3, 0.4, 0.6]]), np.array([0.4, 0.3]), 0.3, niter=2)]
    o = oracle_from_workload(w)
    o.step(1)
    g = grid(gks, w, precision)
    g.step(1)
    assert rel_linf(g.get_state(), o.get_state()) <= TOL[precision]
    a, b = g.forces(0), o.forces(0)
    assert rel_linf(a["force"], np.asarray(b["force"])) <= 10 * TOL[precision]
    assert a["iters"] == 2 and abs(a["residual"] - b["residual"]) <= 10 * TOL[precision]
    g.close()


@pytest.mark.parametrize("precision", ["fp32c", "fp64"])
def test_small_and_large_launch_paths_give_the_same_bits(gks, precision):
    # 96 x 80 x 80 runs one direction after the other (FP32C: z faces fused
    # with the update), its thirds run all directions in one launch
    n = (96, 80, 80)
    w = smooth_workload(n, [(3, 4), (0, 0), (2, 1)], seed=11)
    w.inflow = (1.0, 0.3, 0.0, 0.0)
    w.body_force = (0.01, 0.0, 0.0)
    g = grid(gks, w, precision)
    t = g.step(3)
    s = gks.SlabGroup(w, [32, 64], precision=precision)
    assert s.step(3) == t
    assert np.array_equal(g.get_state(), s.get_state())
    g.close()
    s.close()


@pytest.mark.parametrize("n", [(3, 4, 5), (5, 33, 9), (37, 8, 6), (64, 9, 17)], ids=lambda n: "%dx%dx%d" % n)
def test_reverse_step_at_tile_and_ghost_edges(gks, n):
    """Axes shorter than two ghost layers (the sides of the ghost reverse one
    after the other), remainders of the reverse's tiles. The bars are those of
    the adjoint tests: 1e-5 of a central difference whose terms cannot cancel,
    3e-5 of the largest element for the FP32 reverses."""
    import torch
    h = min(2 * np.pi * (1 + 0.1 * d) / n[d] for d in range(3))
    w = smooth_workload(n, [(3, 4), (0, 0), (1, 2)], seed=sum(n), dt_fixed=0.01 * h)
    w.inflow = (1.0, 0.3, 0.0, 0.0)
    rng = np.random.default_rng(7)
    W = torch.tensor(w.state0, dtype=torch.float64, device="cuda")
    lam1 = torch.tensor(rng.standard_normal(W.shape), dtype=torch.float64, device="cuda")
    g = grid(gks, w, "fp64")
    g.set_adjoint_precision("fp64")
    ref, _ = g.step_adjoint(g.adjoint_workspace(), 0.0, W, lam1, 0.0, None)

    def J(Wx):
        g.set_state_tensor(Wx)
        g.set_time(0.0)
        g.step(1)
        return float((lam1 * g.state_tensor()).sum().item())

    dW = torch.sign(ref) * torch.tensor(0.5 + rng.random(W.shape), dtype=torch.float64, device="cuda")
    eps = 1e-7
    fd = (J(W + eps * dW) - J(W - eps * dW)) / (2 * eps)
    assert abs(fd - float((ref * dW).sum().item())) <= 1e-5 * abs(fd)
    g.set_adjoint_precision("fp32")
    lam, _ = g.step_adjoint(g.adjoint_workspace(), 0.0, W, lam1, 0.0, None)
    assert float((lam - ref).abs().max()) <= 3e-5 * float(ref.abs().max())
    g.close()
    c = grid(gks, w, "fp32c")
    c.set_state_tensor(W)
    c.set_time(0.0)
    tape = c.adjoint_tape()
    c.step_record(tape)
    lam, _ = c.step_reverse(tape, c.adjoint_scratch(), lam1, 0.0, None)
    assert float((lam - ref).abs().max()) <= 3e-5 * float(ref.abs().max())
    c.close()
