"""Workloads for timing the package through its public entry points.

Each case hands a seeded initial state to a grid and takes it through one of
the things a program does with it:

* ``steps``     upload a state, run a few S2O4 steps, read the state back and,
                with a rotor, its loads and the forces on its bodies;
* ``gradient``  upload a state, record steps with their tapes, and reverse them
                from a given adjoint of the last state (state, force-scale and
                inflow-speed gradients);
* ``exchange``  upload a state, read the conserved totals and take the state
                back: a restart or a coupled program's hand-over.

The flows are the package's own (Taylor-Green vortex, channel, rotor, rotor
with tower and nacelle). Results of the FP32C path (and of FP32 reverse
arithmetic) are returned as 32-bit values, which is what that arithmetic
carries; the FP64 and double-single paths return 64 bits.

:func:`exact` evaluates the same method in 64 bits with plain torch
operations: ghost cells, WENO5, half-Maxwellian face state, Gauss-point
reconstruction, gas-kinetic flux, two-stage update, forcing; its gradients
come from torch's autograd.
"""
from __future__ import annotations

import math

import numpy as np
import torch
from torch.utils.checkpoint import checkpoint

from paper_2603_11102_gb300 import gks
from paper_2603_11102_gb300 import workloads as WL


def _case(name, what, flow, n, precision, steps, graphs=False, reverse="fp32"):
    return {"name": name, "what": what, "flow": flow, "nx": n[0], "ny": n[1], "nz": n[2], "precision": precision,
            "steps": steps, "graphs": graphs, "reverse": reverse}


def listed():
    return [
        # the smallest grid in use (a validation run): launches and latency count; replayed from a CUDA graph
        _case("vortex-32-graphs", "steps", "taylor-green", (32, 32, 32), "fp32c", 20, graphs=True),
        # the same validation run as FP64 reference, plain launches
        _case("vortex-32-fp64", "steps", "taylor-green", (32, 32, 32), "fp64", 5),
        # the turbulent channel: stretched axis, no-slip walls, body force
        _case("channel-128", "steps", "channel", (128, 128, 128), "fp32c", 8),
        # a rotor with tower and nacelle at odd sizes that divide no tile
        _case("rotor-bodies-ragged", "steps", "rotor-bodies", (221, 83, 91), "fp32c", 8),
        # production run: a rotor alone on a long domain
        _case("rotor-512", "steps", "rotor", (512, 192, 192), "fp32c", 4),
        # production run: rotor, tower and nacelle on the largest grid
        _case("rotor-bodies-384", "steps", "rotor-bodies", (384, 256, 256), "fp32c", 4),
        # FP64 reference of the channel
        _case("channel-128-fp64", "steps", "channel", (128, 128, 128), "fp64", 1),
        # FP64 reference of a rotor run in double-single arithmetic
        _case("rotor-bodies-256-ds", "steps", "rotor-bodies", (256, 96, 96), "ds", 2),
        # gradients of an FP32C rotor run: recorded steps and their reverse
        _case("gradient-256", "gradient", "rotor", (256, 128, 128), "fp32c", 2),
        # gradients of an FP64 rotor run with FP32 reverse arithmetic
        _case("gradient-128-fp64", "gradient", "rotor", (128, 64, 64), "fp64", 1),
        # a restart of the largest grid with its conserved totals
        _case("exchange-384", "exchange", "rotor-bodies", (384, 256, 256), "fp32c", 0),
        # the same hand-over on an FP64 channel
        _case("exchange-128-fp64", "exchange", "channel", (128, 128, 128), "fp64", 0),
    ]


def draw(rng):
    """A case of the same ranges: 32^3 to 384x256x256 cells, every flow, precision and use."""
    what = rng.choice(["steps"] * 6 + ["gradient", "gradient", "exchange"])
    precision = rng.choice(["fp32c", "fp32c", "fp32c", "fp64", "ds"])
    flow = rng.choice(["taylor-green", "channel", "rotor", "rotor-bodies"])
    if what == "gradient":
        flow = "rotor"
        precision = "fp64" if precision == "ds" else precision
    if what == "exchange":
        precision = "fp64" if precision == "ds" else precision
    most = {"fp32c": 25e6, "fp64": 1.5e6, "ds": 3e6}[precision]
    if what == "gradient":
        most = 4e6 if precision == "fp32c" else 0.6e6
    elif what == "exchange":
        most = 12e6
    least = 32 ** 3 if flow in ("taylor-green", "channel") else 1.2e5
    cells = math.exp(rng.uniform(math.log(least), math.log(most)))
    if flow == "taylor-green":
        nx = ny = nz = max(32, int(cells ** (1 / 3)))
    elif flow == "channel":
        nx = int(cells ** (1 / 3) * rng.uniform(0.8, 1.25))
        ny = int(cells ** (1 / 3) * rng.uniform(0.8, 1.25))
        nz = int(cells / (nx * ny))
    else:
        nx = int((cells * 5.0) ** (1 / 3) * rng.uniform(1.0, 1.3))
        ny = int(math.sqrt(cells / nx) * rng.uniform(0.9, 1.1))
        nz = int(cells / (nx * ny))
    steps = 0 if what == "exchange" else rng.randint(1, 2) if what == "gradient" else rng.randint(1, 4)
    if precision != "fp32c":
        steps = min(steps, 1 if what == "gradient" else 2)
    return {"what": what, "flow": flow, "nx": nx, "ny": ny, "nz": nz, "precision": precision, "steps": steps,
            "graphs": rng.random() < 0.3, "reverse": rng.choice(["fp32", "fp32", "fp64"])}


def _workload(case):
    """The package's workload of a case, without an initial state."""
    n = (case["nx"], case["ny"], case["nz"])
    if case["flow"] == "taylor-green":
        w = WL.taylor_green_3d(8)
        w.n, w.faces = n, [WL.uniform_faces(0.0, 2.0 * math.pi, k) for k in n]
    elif case["flow"] == "channel":
        w = WL.channel((8, 8, 8))
        w.n = n
        w.faces = [WL.uniform_faces(0.0, 2.0 * math.pi, n[0]), WL.tanh_faces(n[1]), WL.uniform_faces(0.0, math.pi, n[2])]
    else:
        # built on few cells, then given the case's: the builders also make the state
        bodies = case["flow"] == "rotor-bodies"
        w = (WL.alm_ibm_rotor if bodies else WL.alm_rotor)((n[0], 8, 8))
        w.n = n
        w.faces = [w.faces[0]] + [WL.uniform_faces(f[0], f[-1], k) for f, k in zip(w.faces[1:], n[1:])]
    w.state0 = None
    if case["what"] == "gradient":
        hmin = min(float(np.min(np.diff(f))) for f in w.faces)
        w.dt_fixed = 0.4 * hmin / (1.2 * w.u_ref + w.u_ref / w.mach)
    return w


def _device():
    return torch.device("cuda" if torch.cuda.is_available() else "cpu")


def _inputs(case, seed):
    """The seeded inputs of a case: the initial state, the time and, for gradients, the adjoint of the last state."""
    dev = _device()
    w = _workload(case)
    gen = torch.Generator(device=dev)
    gen.manual_seed(int(seed))
    shape = (4, w.n[2], w.n[1], w.n[0])

    def noise(amp):
        return amp * (2.0 * torch.rand((3,) + shape[1:], dtype=torch.float64, device=dev, generator=gen) - 1.0)

    Q = torch.zeros(shape, dtype=torch.float64, device=dev)
    Q[0] = 1.0 + 1e-3 * (2.0 * torch.rand(shape[1:], dtype=torch.float64, device=dev, generator=gen) - 1.0)
    x, y, z = (torch.tensor(WL.cell_centres(f), dtype=torch.float64, device=dev) for f in w.faces)
    if case["flow"] == "taylor-green":
        cx, cy, cz = x, y[:, None], z[:, None, None]
        Q[1] = torch.sin(cx) * torch.cos(cy) * torch.cos(cz)
        Q[2] = -torch.cos(cx) * torch.sin(cy) * torch.cos(cz)
        Q[1:] += noise(0.01)
    elif case["flow"] == "channel":
        Q[1] = (1.5 * (1.0 - y ** 2))[None, :, None]
        Q[1:] += noise(0.05)
    else:
        Q[1] = 1.0
        Q[1:] += noise(0.02)
    out = {"workload": w, "Q": Q, "t0": 0.01 * (int(seed) % 97)}
    if case["what"] == "gradient":
        out["lam"] = torch.randn(shape, dtype=torch.float64, device=dev, generator=gen)
    return out


def prepare(case, seed):
    s = _inputs(case, seed)
    w = s["workload"]
    g = gks.Grid.from_workload(w, precision="fp32c" if case["precision"] == "fp32c" else "fp64")
    if case["precision"] == "ds":
        g.set_fp64_arithmetic("ds")
    g.set_graphs(case["graphs"])
    s.update(case=case, grid=g, bits32=case["precision"] == "fp32c")
    if case["what"] == "gradient":
        g.set_adjoint_precision(case["reverse"])
        s["bits32"] = s["bits32"] or case["reverse"] == "fp32"
        s["tapes"] = [g.adjoint_tape() for _ in range(case["steps"])]
        s["scratch"] = g.adjoint_scratch()
    return s


def _narrow(s, v):
    """FP32 results as 32-bit values, others as 64-bit ones."""
    if isinstance(v, torch.Tensor):
        return v.float() if s["bits32"] else v
    return np.asarray(v, dtype=np.float32 if s["bits32"] else np.float64)


def run(s):
    g, case, w = s["grid"], s["case"], s["workload"]
    g.set_state_tensor(s["Q"], sync=False)
    if case["what"] == "exchange":
        return {"totals": g.diagnostics(), "state": _narrow(s, g.state_tensor())}
    if w.rotors:
        g.set_time(s["t0"])
    if case["what"] == "gradient":
        for tape in s["tapes"]:
            g.step_record(tape)
        lam, gu = s["lam"], 0.0
        gs = np.zeros(w.rotors[0].n_blades * w.rotors[0].r.size)
        for k, tape in enumerate(reversed(s["tapes"])):
            lam, gun = g.step_reverse(tape, s["scratch"], lam, 1.0 if k == 0 else 0.0, gs)
            gu += gun
        return {"lam": _narrow(s, lam), "scales": _narrow(s, gs), "uinf": _narrow(s, np.array([gu]))}
    g.step(case["steps"])
    out = {"state": _narrow(s, g.state_tensor())}
    for k, obj in enumerate(g.objects):
        f = g.forces(k)
        keys = ("thrust", "torque", "power", "Fx", "Ft") if obj[0] == "rotor" else ("force",)
        out["%s%d" % (obj[0], k)] = {key: _narrow(s, f[key]) for key in keys}
    return out


def work(case):
    """State in and out, and per step the state read and written once per stage and the operations of the method
    (per face 390 for its state and 1150 for the flux at its 4 Gauss points; 6 faces a cell over the two stages)."""
    cells = case["nx"] * case["ny"] * case["nz"]
    out = 16 if case["precision"] == "fp32c" else 32
    step_bytes = 160 if case["precision"] == "fp32c" else 192
    if case["what"] == "exchange":
        return {"bytes": cells * (32 + out), "flops": cells * 18}
    per = 2 if case["what"] == "gradient" else 1   # a reverse step reads and writes no less than the step
    flops = {"steps": 9.3e3, "gradient": 9.3e3 + 2.5e4}[case["what"]]
    return {"bytes": cells * (32 * per + out + per * case["steps"] * step_bytes), "flops": cells * case["steps"] * flops}


# ---- the method in 64 bits with plain torch ----

G = 3   # ghost layers


def _quartic_weights():
    """Value and derivative weights of the quartic through 5 cell averages at the Gauss points -+1/(2 sqrt 3)."""
    e = np.arange(5)
    M = np.array([[((c + 0.5) ** (p + 1) - (c - 0.5) ** (p + 1)) / (p + 1) for p in e] for c in range(-2, 3)])
    inv = np.linalg.inv(M)
    val, der = [], []
    for x in (-0.5 / math.sqrt(3.0), 0.5 / math.sqrt(3.0)):
        val.append(np.array([x ** p for p in e]) @ inv)
        der.append(np.array([p * x ** (p - 1) if p else 0.0 for p in e]) @ inv)
    return val, der


_VAL, _DER = _quartic_weights()


def _cut(A, d, start, length):
    """Along axis d (0 = x): x is the last dimension."""
    return A.narrow(A.dim() - 1 - d, start, length)


def _weno5(a, b, c, d, e):
    """WENO5-JS at the face between c and d."""
    b0 = 13 / 12 * (a - 2 * b + c) ** 2 + 0.25 * (a - 4 * b + 3 * c) ** 2
    b1 = 13 / 12 * (b - 2 * c + d) ** 2 + 0.25 * (b - d) ** 2
    b2 = 13 / 12 * (c - 2 * d + e) ** 2 + 0.25 * (3 * c - 4 * d + e) ** 2
    w0, w1, w2 = 0.1 / (1e-6 + b0) ** 2, 0.6 / (1e-6 + b1) ** 2, 0.3 / (1e-6 + b2) ** 2
    p0, p1, p2 = (2 * a - 7 * b + 11 * c) / 6, (-b + 5 * c + 2 * d) / 6, (2 * c + 5 * d - e) / 6
    return (w0 * p0 + w1 * p1 + w2 * p2) / (w0 + w1 + w2)


class _Method:
    """One grid: steps of an interior state (4, nz, ny, nx)."""

    def __init__(self, w, dev, uinf=None, scales=None):
        self.w, self.dev, self.n = w, dev, w.n
        self.lam = w.mach ** 2 / (2.0 * w.u_ref ** 2)
        self.theta = 1.0 / (2.0 * self.lam)
        self.cs = math.sqrt(self.theta)
        self.uin = [w.inflow[1] if uinf is None else uinf, w.inflow[2], w.inflow[3]]
        self.scales = scales
        self.h, self.hf, self.hmin = [], [], math.inf
        for d in range(3):
            h = np.diff(w.faces[d])
            self.hmin = min(self.hmin, float(h.min()))
            n, (lo, hi) = w.n[d], w.bc[d]
            low = [h[-(k % n) - 1] if lo == WL.BC_PERIODIC else h[k] for k in range(G)][::-1]
            high = [h[k % n] if hi == WL.BC_PERIODIC else h[n - 1 - k] for k in range(G)]
            h = torch.tensor(np.concatenate([low, h, high]), dtype=torch.float64, device=dev)
            shape = [1, 1, 1]
            shape[2 - d] = -1
            self.h.append(h.reshape(shape))
            self.hf.append((0.5 * (h[G - 1:G + n] + h[G:G + n + 1])).reshape(shape))

    def ghosts(self, W):
        for d in range(3):
            n = self.n[d]
            parts = [None, W, None]
            for s, bc in enumerate(self.w.bc[d]):
                layers = []
                for k in range(1, G + 1):
                    if bc == WL.BC_PERIODIC:
                        layers.append(_cut(W, d, (-k if s == 0 else k - 1) % n, 1))
                        continue
                    mirror = bc in (WL.BC_NOSLIP, WL.BC_SLIP)
                    q = _cut(W, d, (k - 1 if s == 0 else n - k) if mirror else (0 if s == 0 else n - 1), 1)
                    if bc == WL.BC_NOSLIP:
                        q = torch.cat([q[:1], -q[1:]])
                    elif bc == WL.BC_SLIP:
                        q = torch.stack([-q[v] if v == 1 + d else q[v] for v in range(4)])
                    elif bc == WL.BC_INFLOW:
                        rho = q[0] * torch.exp((1 if s == 0 else -1) * (self.uin[d] - q[1 + d] / q[0]) / self.cs)
                        q = torch.stack([rho] + [rho * u for u in self.uin])
                    layers.append(q)
                parts[2 * s] = torch.cat(layers[::-1] if s == 0 else layers, dim=W.dim() - 1 - d)
            W = torch.cat(parts, dim=W.dim() - 1 - d)
        return W

    def direction(self, A, d):
        """F0 and F1 differences over the cells of axis d, divided by the widths."""
        n, t1, t2 = self.n[d], 1 if d == 0 else 0, 1 if d == 2 else 2
        order = [0, 1 + d, 1 + t1, 1 + t2]
        lam, th, mu = self.lam, self.theta, self.w.mu
        # face state on the faces 0..n, tangentially -2..n+1
        A = _cut(_cut(A, t1, 1, self.n[t1] + 4), t2, 1, self.n[t2] + 4)
        left, right, slope = [], [], []
        for v in order:
            q = [_cut(A[v], d, k, n + 1) for k in range(6)]
            left.append(_weno5(*q[:5]))
            right.append(_weno5(*q[:0:-1]))
            slope.append((15 * (q[3] - q[2]) - (q[4] - q[1])) / (12 * self.hf[d]))
        ul, ur = left[1] / left[0], right[1] / right[0]
        pl, pr = 0.5 * torch.erfc(-math.sqrt(lam) * ul), 0.5 * torch.erfc(math.sqrt(lam) * ur)
        k = 1.0 / (2.0 * math.sqrt(math.pi * lam))
        Q = [a * pl + b * pr for a, b in zip(left, right)]
        Q[1] = Q[1] + left[0] * k * torch.exp(-lam * ul ** 2) - right[0] * k * torch.exp(-lam * ur ** 2)
        del left, right, ul, ur, pl, pr

        def along(q, t, weights):
            return sum(float(weights[k]) * _cut(q, t, k, self.n[t]) for k in range(5))

        h1, h2 = (_cut(self.h[t], t, G, self.n[t]) for t in (t1, t2))
        F0, F1 = [0.0] * 4, [0.0] * 4
        for m in range(2):
            q1, e1, s1 = ([along(q, t1, x[m]) for q in a] for a, x in ((Q, _VAL), (Q, _DER), (slope, _VAL)))
            for j in range(2):
                q, g2, g1, g0 = ([along(c, t2, x[j]) for c in a] for a, x in ((q1, _VAL), (q1, _DER), (e1, _VAL), (s1, _VAL)))
                D = [g0, [x / h1 for x in g1], [x / h2 for x in g2]]
                rho, U = q[0], [q[1] / q[0], q[2] / q[0], q[3] / q[0]]
                S = [[(D[i][1 + k] - U[k] * D[i][0]) / rho for k in range(3)] for i in range(3)]   # d_i U_k
                lnr = [D[i][0] / rho for i in range(3)]
                A0 = -sum(U[i] * lnr[i] + S[i][i] for i in range(3))
                B = [-th * lnr[k] - sum(U[i] * S[i][k] for i in range(3)) for k in range(3)]
                f0 = [q[1]] + [q[1] * U[k] - mu * (S[0][k] + S[k][0]) + (th * rho if k == 0 else 0.0) for k in range(3)]
                f1 = [rho * (A0 * U[0] + B[0])]
                f1 += [rho * (A0 * (U[0] * U[k] + (th if k == 0 else 0.0)) + B[0] * U[k] + B[k] * U[0]) for k in range(3)]
                F0, F1 = ([a + 0.25 * b for a, b in zip(F, f)] for F, f in ((F0, f0), (F1, f1)))
        back = [order.index(v) for v in range(4)]
        hd = _cut(self.h[d], d, G, n)
        return tuple(torch.stack([(_cut(F[b], d, 1, n) - _cut(F[b], d, 0, n)) / hd for b in back]) for F in (F0, F1))

    def rhs(self, W):
        A, L, Lt = self.ghosts(W), 0.0, 0.0
        for d in range(3):
            if W.requires_grad:
                a, b = checkpoint(self.direction, A, d, use_reentrant=False)
            else:
                a, b = self.direction(A, d)
            L, Lt = L - a, Lt - b
        return L, Lt

    def step(self, W, t):
        """Returns (W^{n+1}, t_{n+1}, loads)."""
        w = self.w
        dt = w.dt_fixed
        if not dt > 0.0:
            u2 = (W[1:] ** 2).sum(0) / W[0] ** 2
            dt = w.cfl * self.hmin / (math.sqrt(float(u2.max())) + self.cs)
        L, Lt = self.rhs(W)
        Lts = self.rhs(W + dt / 2 * L + dt * dt / 8 * Lt)[1]
        W = W + dt * L + dt * dt / 6 * (Lt + 2 * Lts)
        if any(w.body_force):
            f = torch.tensor((0.0,) + tuple(w.body_force), dtype=torch.float64, device=self.dev)
            W = W + dt * f[:, None, None, None]
        loads = {}
        for k, r in enumerate(w.rotors):
            W, loads["rotor%d" % k] = self.rotor(W, r, t + dt, dt)
        for k, b in enumerate(w.bodies):
            W, loads["body%d" % (len(w.rotors) + k)] = self.body(W, b, dt)
        return W, t + dt, loads

    def support(self, X, rad):
        """Interior index box (x, y, z ranges) of the cells within rad of the points, and its cell centres."""
        box, centres = [], []
        for d in range(3):
            h, x0 = float(self.h[d].reshape(-1)[G]), float(self.w.faces[d][0])
            lo = max(0, math.floor((float(X[:, d].min()) - rad - x0) / h - 0.5) - 1)
            hi = min(self.n[d] - 1, math.ceil((float(X[:, d].max()) + rad - x0) / h - 0.5) + 1)
            box.append(slice(lo, hi + 1))
            centres.append(x0 + (torch.arange(lo, hi + 1, dtype=torch.float64, device=self.dev) + 0.5) * h)
        z, y, x = torch.meshgrid(centres[2], centres[1], centres[0], indexing="ij")
        return (box[2], box[1], box[0]), torch.stack([x, y, z], dim=-1)

    @staticmethod
    def gauss(r2, eps):
        eta = torch.exp(-r2 / eps ** 2) / (eps ** 3 * math.pi ** 1.5)
        return torch.where(torch.sqrt(r2) <= 3.0 * eps, eta, torch.zeros_like(eta))

    def rotor(self, W, r, t, dt):
        T = dict(dtype=torch.float64, device=self.dev)
        rr, chord, twist, width = (torch.tensor(np.tile(a, r.n_blades), **T) for a in (r.r, r.chord, r.twist, r.width))
        blade = torch.arange(r.n_blades, **T).repeat_interleave(r.r.size)
        ang = r.azimuth0 + r.omega * t + 2.0 * math.pi * blade / r.n_blades
        c, s = torch.cos(ang), torch.sin(ang)
        X = torch.stack([torch.full_like(rr, r.hub[0]), r.hub[1] + rr * c, r.hub[2] + rr * s], dim=1)
        # trilinear sample of the velocity
        low, frac = [], []
        for d in range(3):
            p = (X[:, d] - float(self.w.faces[d][0])) / float(self.h[d].reshape(-1)[G]) - 0.5
            low.append(torch.floor(p).long())
            frac.append(p - torch.floor(p))
        vel = 0.0
        for k in range(8):
            o = [(k >> d) & 1 for d in range(3)]
            wt = math.prod([frac[d] if o[d] else 1.0 - frac[d] for d in range(3)])
            q = W[:, low[2] + o[2], low[1] + o[1], low[0] + o[0]]
            vel = vel + wt * q[1:] / q[0]
        ux, rel = vel[0], r.omega * rr - (c * vel[2] - s * vel[1])
        phi = torch.atan2(ux, rel)
        al = phi - twist
        qd = 0.5 * r.rho_inf * chord * width * (ux ** 2 + rel ** 2)
        lift, drag = qd * torch.clamp(2.0 * math.pi * torch.sin(al), -1.4, 1.4), qd * (0.01 + 0.02 * al ** 2)
        Fx, Ft = lift * torch.cos(phi) + drag * torch.sin(phi), lift * torch.sin(phi) - drag * torch.cos(phi)
        if self.scales is not None:
            Fx, Ft = Fx * self.scales, Ft * self.scales
        box, xc = self.support(X, 3.0 * r.eps)
        f = torch.zeros((3,) + xc.shape[:3], **T)
        for k in range(0, X.shape[0], 32):
            eta = self.gauss(((xc[None] - X[k:k + 32, None, None, None]) ** 2).sum(-1), r.eps)
            F = torch.stack([-Fx, s * Ft, -c * Ft])[:, k:k + 32]
            f = f + torch.einsum("dp,pzyx->dzyx", F, eta)
        add = torch.zeros_like(W)
        add[(slice(1, 4),) + box] = dt * f
        nb = (r.n_blades, r.r.size)
        out = {"thrust": Fx.reshape(nb).sum(1), "torque": (rr * Ft).reshape(nb).sum(1), "Fx": Fx.reshape(nb), "Ft": Ft.reshape(nb)}
        out["power"] = r.omega * out["torque"].sum()
        return W + add, out

    def body(self, W, b, dt):
        X = torch.tensor(b.xyz, dtype=torch.float64, device=self.dev)
        dS = torch.tensor(b.dS, dtype=torch.float64, device=self.dev)
        vol = math.prod(float(h.reshape(-1)[G]) for h in self.h)
        box, xc = self.support(X, 3.0 * b.eps)
        V = torch.zeros(xc.shape[:3], dtype=torch.float64, device=self.dev)
        for k in range(0, X.shape[0], 64):
            eta = self.gauss(((xc[None] - X[k:k + 64, None, None, None]) ** 2).sum(-1), b.eps)
            V = V + vol * vol ** (1.0 / 3.0) * torch.einsum("p,pzyx->zyx", dS[k:k + 64], eta)
        keep = (1.0 - torch.clamp(V / vol, max=1.0)) ** b.niter   # the points are at rest
        W = W.clone()
        m = W[(slice(1, 4),) + box]
        force = (m * (1.0 - keep)).sum((1, 2, 3)) * vol / dt
        W[(slice(1, 4),) + box] = m * keep
        return W, {"force": force}


def _numbers(v):
    return {k: _numbers(x) if isinstance(x, dict) else x.detach() for k, x in v.items()}


def exact(case, seed):
    s = _inputs(case, seed)
    w, Q, dev = s["workload"], s["Q"], s["Q"].device
    if case["what"] == "exchange":
        vol = math.prod(torch.tensor(np.diff(w.faces[d]), dtype=torch.float64, device=dev).reshape([-1 if k == 2 - d else 1 for k in range(3)])
                        for d in range(3))
        sums = [(q * vol).sum() for q in Q] + [(0.5 * (Q[1:] ** 2).sum(0) / Q[0] * vol).sum()]
        return {"totals": torch.stack(sums), "state": Q}
    if case["what"] == "gradient":
        rot = w.rotors[0]
        u = torch.tensor(w.inflow[1], dtype=torch.float64, device=dev, requires_grad=True)
        scales = torch.ones(rot.n_blades * rot.r.size, dtype=torch.float64, device=dev, requires_grad=True)
        M, W, t = _Method(w, dev, u, scales), Q.requires_grad_(True), s["t0"]
        for _ in range(case["steps"]):
            W, t, loads = M.step(W, t)
        J = (s["lam"] * W).sum() + loads["rotor0"]["power"]
        lam, gu, gs = torch.autograd.grad(J, (Q, u, scales))
        return {"lam": lam, "scales": gs, "uinf": gu.reshape(1)}
    with torch.no_grad():
        M, W, t = _Method(w, dev), Q, s["t0"]
        for _ in range(case["steps"]):
            W, t, loads = M.step(W, t)
    return {"state": W, **_numbers(loads)}
