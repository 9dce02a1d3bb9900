"""What a user of the propagator has it do, as cases that can be timed.

A case is one call (or one forward and reverse pair) through the public Python
entry points: pcprop.propagate, pcprop.propagate_groups, autodiff.propagate and
autodiff.bplane.  Plans are created as plan_from_workload and options_default
create them, with the launch tuning they come with.

Kinds of case
  batch      one batch over a common arc.  orbit "ellipse": the Sun-Venus-Earth
             study orbits (configurations 1 and 3); "flyby": starts half a day
             to a day and a half before a Venus encounter among the Sun, eight
             planets and the Moon (configuration 2).
  uneven     per-trajectory arcs, degrees and segment counts (configuration 5),
             one plan per degree.
  gradient   configuration 4: the arc to the nominal periapsis, the b-plane
             there, the rest of the arc, and the gradient of a scalar of both
             with respect to the start states.

exact() integrates the same equations of motion in 64 bits with an extrapolation
integrator of its own (Gragg's modified midpoint rule, order 16); it shares only
the workload generators' inputs with the library.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2301_03989_gb300 import autodiff
from paper_2301_03989_gb300 import pcprop as pc
from paper_2301_03989_gb300 import workloads as W

C_LIGHT = 299792.458  # km/s
DEGREES = (32, 64, 128, 256)


def _batch(name=None, **kw):
    case = dict(kind="batch", orbit="ellipse", n_ic=64, N=128, segments=8, years=0.65, backward=False,
                precision="fp64", order=1, fp32_mma=0, switch_tol=0.0, eih=False)
    case.update(kw)
    if name:
        case["name"] = name
    return case


def listed():
    return [
        # one start state through the default plan: what an interactive user or
        # an optimiser's single objective call waits for
        _batch("single_default", n_ic=1, N=64, segments=8),
        # configuration 1: a handful of dispersed states, default plan
        _batch("dispersion_64", n_ic=64, N=64, segments=8),
        # a few hundred states in mixed precision, an odd count
        _batch("mixed_301", n_ic=301, N=128, segments=13, years=1.0, precision="mixed", order=2, switch_tol=1e-6),
        # an ordinary Monte Carlo batch with the settings of the precision study
        _batch("study_mixed_4096", n_ic=4096, segments=25, years=2.0, precision="mixed", order=2, fp32_mma=1,
               switch_tol=1e-6),
        # configuration 3 in full: the headline batch
        _batch("study_mixed_65536", n_ic=65536, segments=25, years=2.0, precision="mixed", order=2, fp32_mma=1,
               switch_tol=1e-6),
        # the same study in plain FP64, second-order sweep
        _batch("study_fp64_16384", n_ic=16384, segments=25, years=2.0, order=2),
        # default plan (first-order FP64 sweep), ragged count, integrated backward
        _batch("backward_2501", n_ic=2501, segments=13, years=1.0, backward=True),
        # configuration 2: close flybys among ten bodies, mixed precision as the README creates it
        _batch("flyby_mixed_2048", orbit="flyby", n_ic=2048, segments=16, years=0.5, precision="mixed"),
        # a small flyby batch with the default plan
        _batch("flyby_fp64_129", orbit="flyby", n_ic=129, segments=16, years=0.25),
        # the paper's relativistic force on the ten-body system
        _batch("eih_1000", n_ic=1000, segments=13, years=1.0, order=2, eih=True),
        # configuration 5: uneven arcs and degrees, one plan per degree
        dict(name="uneven_6000", kind="uneven", n_ic=6000, years=10.0, precision="mixed", fp32_mma=1),
        # configuration 4: gradients of a flyby's b-plane and end state (the arc ends before these orbits meet Venus again)
        dict(name="gradient_512", kind="gradient", n_ic=512, revolutions=0.8),
    ]


def draw(rng):
    """One more case of the same ranges; sizes are log-uniform, seldom round."""
    def log_int(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(["ellipse", "ellipse", "ellipse", "ellipse", "flyby", "eih", "uneven", "gradient"])
    if kind == "uneven":
        return dict(kind="uneven", n_ic=log_int(64, 8000), years=round(rng.uniform(2.0, 10.0), 3),
                    precision=rng.choice(["mixed", "fp64"]), fp32_mma=rng.choice([0, 1]))
    if kind == "gradient":
        return dict(kind="gradient", n_ic=log_int(8, 700), revolutions=round(rng.uniform(0.3, 0.8), 3))
    precision = rng.choice(["mixed", "fp64"])
    order = rng.choice([1, 2])
    if kind == "flyby":
        return _batch(orbit="flyby", n_ic=log_int(16, 2048), segments=16, years=round(rng.uniform(0.2, 0.5), 4),
                      precision=precision, order=order)
    years = round(rng.uniform(0.4, 2.0), 4)
    N = rng.choice([48, 64, 100, 128, 128, 200])
    per_year = 16 if N < 64 else 13                       # segments per year at which these degrees converge
    n_ic = log_int(1, 2000 if kind == "eih" else 65536)
    # cost about n_ic x segments x N^2, held below the largest listed case's (FP64 sweeps cost more than mixed ones)
    budget = 65536 * 25 * 128**2 * (0.9 if precision == "mixed" and order == 2 else 0.35)
    segments = max(4, math.ceil(per_year * years))
    n_ic = max(1, min(n_ic, int(budget / (segments * N * N))))
    return _batch(n_ic=n_ic, N=N, segments=segments, years=years, backward=rng.random() < 0.3, precision=precision,
                  order=order, fp32_mma=rng.choice([0, 1]) if precision == "mixed" else 0,
                  switch_tol=rng.choice([0.0, 1e-6]) if precision == "mixed" else 0.0, eih=kind == "eih")


# --------------------------------------------------------------------------
# Workloads (inputs from the seed alone)
# --------------------------------------------------------------------------
def _workload(case, seed):
    """The force model, tables, start states and arc of a batch case."""
    if case["orbit"] == "flyby":
        return W.config2(M=case["n_ic"], seed=seed, years=case["years"])
    w = W.config3(M=case["n_ic"], seed=seed)
    if case["eih"]:  # the ten-body system's tables over the same span
        s = W.config2(M=1, seed=seed, years=2.0)
        w.body_names, w.mu, w.t_begin, w.granule, w.coef = s.body_names, s.mu, s.t_begin, s.granule, s.coef
    w.N, w.segments = case["N"], case["segments"]
    span = case["years"] * W.YEAR
    w.t0, w.tf = (span, 0.0) if case["backward"] else (0.0, span)
    return w


def _gradient_parts(case, seed):
    w = W.config4(M=case["n_ic"], seed=seed)
    w.tf = case["revolutions"] * w.tf
    g = np.random.default_rng(seed + 1)
    return w, g.standard_normal((6, case["n_ic"])), g.standard_normal((2, case["n_ic"]))


def _dev(a, dtype=torch.float64):
    return torch.as_tensor(np.ascontiguousarray(a), dtype=dtype, device="cuda")


def _precision(case):
    return pc.PC_PREC_MIXED if case["precision"] == "mixed" else pc.PC_PREC_FP64


def prepare(case, seed):
    if case["kind"] == "uneven":
        uw = W.config5(M=case["n_ic"], seed=seed, years_max=case["years"])
        perm, degrees, counts = uw.groups()
        b = uw.base
        plans = []
        for d in degrees:
            o = pc.options_default(tol=b.tol, max_iters=b.max_iters, max_depth=b.max_depth, seg_mode=0,
                                   precision=_precision(case), fp32_mma=case["fp32_mma"])
            plans.append(pc.plan_create(int(d), 4, b.mu_central, b.mu, b.t_begin, b.granule, b.coef, b.indirect, o))
        x0 = _dev(W.to_planar(uw.x0[perm]))
        return dict(kind="uneven", plans=plans, counts=counts, x0=x0, t0=_dev(uw.t0[perm]), tf=_dev(uw.tf[perm]),
                    segments=_dev(uw.S[perm], torch.int32), xf=torch.zeros_like(x0),
                    status=torch.zeros(uw.n_ic, dtype=torch.int32, device="cuda"))
    if case["kind"] == "gradient":
        w, c_state, c_plane = _gradient_parts(case, seed)
        M = w.n_ic
        return dict(kind="gradient", plan=pc.plan_from_workload(w), x0=_dev(W.to_planar(w.x0)),
                    t0=torch.full((M,), w.t0, dtype=torch.float64, device="cuda"), t_ca=_dev(w.meta["t_ca"]),
                    tf=torch.full((M,), w.tf, dtype=torch.float64, device="cuda"), body=w.meta["body"],
                    mu_body=w.meta["mu_body"], c_state=_dev(c_state), c_plane=_dev(c_plane))
    w = _workload(case, seed)
    opts = dict(precision=_precision(case), order=case["order"], fp32_mma=case["fp32_mma"],
                switch_tol=case["switch_tol"])
    plan = pc.plan_from_workload(w, c_light=C_LIGHT if case["eih"] else 0.0, **opts)
    x0 = _dev(W.to_planar(w.x0))
    return dict(kind="batch", plan=plan, x0=x0, t0=w.t0, tf=w.tf, xf=torch.zeros_like(x0),
                status=torch.zeros(w.n_ic, dtype=torch.int32, device="cuda"))


def run(state):
    s = state
    if s["kind"] == "batch":
        pc.propagate(s["plan"], s["x0"], s["t0"], s["tf"], s["xf"], status=s["status"])
        return {"xf": s["xf"], "status": s["status"]}
    if s["kind"] == "uneven":
        pc.propagate_groups(s["plans"], s["counts"], s["x0"], s["t0"], s["tf"], s["xf"], segments=s["segments"],
                            status=s["status"])
        return {"xf": s["xf"], "status": s["status"]}
    x0 = s["x0"].detach().requires_grad_(True)
    x_ca, _, _ = autodiff.propagate(x0, s["plan"], s["t0"], s["t_ca"])
    plane = autodiff.bplane(x_ca, s["plan"], s["body"], s["mu_body"], s["t_ca"])
    xf, _, _ = autodiff.propagate(x_ca, s["plan"], s["t_ca"], s["tf"])
    # end state in units of the orbit's size and speed, b-plane in planet radii
    unit = torch.tensor([1e8] * 3 + [30.0] * 3, dtype=torch.float64, device=xf.device)[:, None]
    loss = (s["c_state"] * xf / unit).sum() + (s["c_plane"] * plane / 6052.0).sum()
    (grad,) = torch.autograd.grad(loss, x0)
    return {"xf": xf.detach(), "plane": plane.detach(), "grad_r": grad[:3], "grad_v": grad[3:]}


# --------------------------------------------------------------------------
# Work of one pass
# --------------------------------------------------------------------------
def _pass_flops(N, B, segments, sweeps, reverse=0):
    """FP64-equivalent operations of `sweeps` sweeps of every segment of one
    trajectory: the (N+1) x N x 6 operator product and the force at N+1 nodes."""
    return segments * (sweeps + reverse) * (2.0 * 6 * N * (N + 1) + (N + 1) * (25.0 + 25.0 * B))


def work(case):
    M = case["n_ic"]
    if case["kind"] == "uneven":
        flops = 0.0
        for d in DEGREES:
            length = 0.65 / W.SEGMENTS_PER_REV[d]        # years per segment (0.65 yr a revolution)
            flops += M / 4 * _pass_flops(d, 2, max(4.0, 0.5 * case["years"] / length), 12)
        return dict(bytes=M * (2 * 48 + 20.0), flops=flops)
    if case["kind"] == "gradient":
        segs = 4 + 30.0 * case["revolutions"]
        tape = M * segs * (2 + 6 * 129) * 8.0
        return dict(bytes=M * 4 * 48 + 2 * tape, flops=M * _pass_flops(128, 2, segs, 12, reverse=14))
    B = 9 if case["orbit"] == "flyby" or case["eih"] else 2
    segs = case["segments"] * (1.7 * case["years"] + 0.5) if case["orbit"] == "flyby" else case["segments"]
    sweeps = 7 if case["order"] == 2 else 12
    table = B * (case["years"] * 365.25 / 32.0 + 3) * 3 * 14 * 8.0
    return dict(bytes=M * (2 * 48 + 4.0) + table, flops=M * _pass_flops(case["N"], B, segs, sweeps))


# --------------------------------------------------------------------------
# The same in 64 bits, without the library
# --------------------------------------------------------------------------
class _Sky:
    """Body positions and velocities from the Chebyshev tables, by plain
    polynomial evaluation at times t [M] (or [1], shared by a batch)."""

    def __init__(self, w):
        self.mu_c, self.tb, self.L = float(w.mu_central), float(w.t_begin), float(w.granule)
        self.c = torch.as_tensor(np.ascontiguousarray(np.transpose(w.coef, (1, 3, 0, 2))), device="cuda")  # [G][k][B][3]
        K = self.c.shape[1]
        rows = [np.pad(k * _second_kind(k - 1), (0, K - k)) if k else np.zeros(K) for k in range(K)]
        self.d = torch.as_tensor(np.array(rows) * 2.0 / self.L, device="cuda")  # dT_k/dt = sum_i d[k][i] T_i
        self.m = torch.as_tensor(np.asarray(w.mu, dtype=np.float64), device="cuda")
        self.all_mu = torch.cat([torch.full_like(self.m[:1], self.mu_c), self.m])
        self.eye = torch.eye(len(self.all_mu), dtype=torch.float64, device="cuda")

    def at(self, t, velocity=False):
        g = torch.floor((t - self.tb) / self.L).long().clamp(0, self.c.shape[0] - 1)
        s = 2.0 * (t - (self.tb + g * self.L)) / self.L - 1.0
        cols = [torch.ones_like(s), s]
        for _ in range(2, self.c.shape[1]):
            cols.append(2.0 * s * cols[-1] - cols[-2])
        T, c = torch.stack(cols, 1), self.c[g]
        r = (T[:, :, None, None] * c).sum(1)
        if not velocity:
            return r
        dT = (T[:, None, :] * self.d[None]).sum(2)
        return r, (dT[:, :, None, None] * c).sum(1)

    def accel(self, t, r):
        """Newtonian heliocentric acceleration with the indirect term; r [M][3]."""
        rb = self.at(t)
        d = r[:, None, :] - rb
        k = self.m[None, :, None]
        a = -self.mu_c * r / r.norm(dim=1, keepdim=True) ** 3
        return a - (k * (d / d.norm(dim=2, keepdim=True) ** 3 + rb / rb.norm(dim=2, keepdim=True) ** 3)).sum(1)

    def accel_eih(self, t, r, v):
        """The same plus the 1/c^2 terms of the Einstein-Infeld-Hoffmann equations."""
        rb, vb = self.at(t, velocity=True)
        zero, mu = torch.zeros_like(rb[:, :1]), self.all_mu
        P, V = torch.cat([zero, rb], 1), torch.cat([zero, vb], 1)              # [1][B+1][3]
        V = V - (mu[:, None] * V).sum(1, keepdim=True) / mu.sum()
        D = P[:, None, :] - P[:, :, None]                                      # to body k (axis 2) from body j (axis 1)
        n = D.norm(dim=3) + self.eye
        off = (1.0 - self.eye) * mu
        A = ((off / n**3)[..., None] * D).sum(2)
        Phi = (off / n).sum(2)
        Wv = v + V[:, 0]                                                       # barycentric velocity
        d = P - r[:, None, :]
        q = d.norm(dim=2)
        phi = (mu / q).sum(1)
        br = (-4.0 * phi[:, None] - Phi + (Wv * Wv).sum(1)[:, None] + 2.0 * (V * V).sum(2)
              - 4.0 * (Wv[:, None] * V).sum(2) - 1.5 * ((d * V).sum(2) / q)**2 + 0.5 * (d * A).sum(2))
        s = (-d * (4.0 * Wv[:, None] - 3.0 * V)).sum(2)
        k3 = (mu / q**3)[:, :, None]
        rel = k3 * d * br[:, :, None] + k3 * s[:, :, None] * (Wv[:, None] - V) + 3.5 * (mu / q)[:, :, None] * A
        return self.accel(t, r) + rel.sum(1) / C_LIGHT**2


def _second_kind(k):
    """Chebyshev coefficients (first kind) of U_k."""
    c = np.zeros(k + 1)
    c[k::-2] = 2.0
    if k % 2 == 0:
        c[0] = 1.0
    return c


_ORDER = tuple(range(2, 18, 2))


class _Stepper:
    """Extrapolated steps (order 16) of y' = f(t, y), the whole step replayed
    as one CUDA graph; t and h are tensors [M] or [1]."""

    def __init__(self, f, t, y):
        self.t, self.h, self.y = t.clone(), torch.ones_like(t), y.clone()
        side = torch.cuda.Stream()
        side.wait_stream(torch.cuda.current_stream())
        with torch.cuda.stream(side):
            f(self.t, self.y)
        torch.cuda.current_stream().wait_stream(side)
        self.graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(self.graph):
            self.out = self._step(f, self.t, self.y, self.h)

    @staticmethod
    def _step(f, t, y, h):
        f0 = f(t, y)
        hy, rows = h[:, None], []
        for j, n in enumerate(_ORDER):
            s = hy / n
            a, b = y, y + s * f0
            for i in range(1, n):
                a, b = b, a + 2.0 * s * f(t + (i / n) * h, b)
            new = [0.5 * (a + b + s * f(t + h, b))]
            for k in range(1, j + 1):
                ratio = (_ORDER[j] / _ORDER[j - k]) ** 2 - 1.0
                new.append(new[-1] + (new[-1] - rows[k - 1]) / ratio)
            rows = new
        return rows[-1]

    def step(self, h):
        self.h.copy_(h) if torch.is_tensor(h) else self.h.fill_(h)
        self.graph.replay()
        self.y.copy_(self.out)
        self.t.add_(self.h)
        return self.y


def _integrate(sky, x, t0, tf, rhs=None):
    """x [M][6] from t0 to tf (floats); steps from the shortest time scale of
    the batch, the distance to each body against speed and free fall."""
    f = rhs or (lambda t, y: torch.cat([y[:, 3:6], sky.accel(t, y[:, :3])], 1))
    st = _Stepper(f, torch.full((1,), float(t0), dtype=torch.float64, device="cuda"), x)
    t, sign = float(t0), 1.0 if tf >= t0 else -1.0
    while (tf - t) * sign > 0:
        r, v = st.y[:, :3], st.y[:, 3:6]
        scale = (r.norm(dim=1) ** 3 / sky.mu_c).sqrt().min() * 0.4
        d = (r[:, None] - sky.at(st.t)).norm(dim=2)
        near = torch.minimum((d**3 / sky.m).sqrt(), 2.0 * d / (v.norm(dim=1, keepdim=True) + 10.0)).min() * 0.4
        h = min(float(torch.minimum(scale, near)), abs(tf - t), 8.0 * 86400.0)
        # steps end on the tables' granule boundaries, where the series change
        k = (t - sky.tb) / sky.L
        edge = sky.tb + sky.L * ((math.floor(k + 1e-9) + 1) if sign > 0 else (math.ceil(k - 1e-9) - 1))
        h = min(h, abs(edge - t))
        st.step(sign * h)
        t += sign * h
        if abs(tf - t) < 1e-6:
            break
        st.t.fill_(t)
    return st.y


def _exact_uneven(case, seed):
    uw = W.config5(M=case["n_ic"], seed=seed, years_max=case["years"])
    perm, _, _ = uw.groups()
    sky = _Sky(uw.base)
    span = _dev(uw.tf[perm] - uw.t0[perm])
    x = _dev(uw.x0[perm])
    steps = int(math.ceil(case["years"] * 365.25 / 7.0))
    f = lambda t, y: torch.cat([y[:, 3:6], sky.accel(t, y[:, :3])], 1)  # noqa: E731
    st = _Stepper(f, _dev(uw.t0[perm]), x)
    h = span / steps
    for _ in range(steps):
        st.step(h)
    return st.y


def _exact_gradient(case, seed):
    w, c_state, c_plane = _gradient_parts(case, seed)
    sky, M = _Sky(w), w.n_ic
    t_ca = _dev(w.meta["t_ca"])

    def rhs(t, y):
        x, Phi = y[:, :6], y[:, 6:].reshape(-1, 6, 6)
        r = x[:, :3]
        eye = torch.eye(3, dtype=torch.float64, device="cuda")
        n = r.norm(dim=1)[:, None, None]
        A = -sky.mu_c * (eye / n**3 - 3.0 * r[:, :, None] * r[:, None, :] / n**5)
        d = r[:, None] - sky.at(t)
        q = d.norm(dim=2)[:, :, None, None]
        A = A - (sky.m[None, :, None, None] * (eye / q**3 - 3.0 * d[..., :, None] * d[..., None, :] / q**5)).sum(1)
        dPhi = torch.cat([Phi[:, 3:], A @ Phi[:, :3]], 1)
        return torch.cat([x[:, 3:], sky.accel(t, r), dPhi.reshape(-1, 36)], 1)

    eye6 = torch.eye(6, dtype=torch.float64, device="cuda").reshape(1, 36).expand(M, 36)
    st = _Stepper(rhs, torch.full_like(t_ca, w.t0), torch.cat([_dev(w.x0), eye6], 1))
    # to the periapsis and away from it: steps of a tenth of the time from it,
    # 100 s within 1000 s of it, at most four days
    left = t_ca - w.t0
    while float(left.max()) > 0:
        h = torch.minimum(left, (0.1 * left).clamp(100.0, 345600.0))
        st.step(h)
        left = left - h
    y = st.y.clone()
    Phi1 = y[:, 6:].reshape(-1, 6, 6)
    x_ca = y[:, :6].clone().requires_grad_(True)
    # b-plane of the Venus-relative hyperbola
    t_np = w.meta["t_ca"]
    g = np.clip(np.floor((t_np - w.t_begin) / w.granule).astype(int), 0, w.coef.shape[1] - 1)
    sig = 2.0 * (t_np - (w.t_begin + g * w.granule)) / w.granule - 1.0
    body = np.zeros((M, 6))
    for m in range(M):
        c = w.coef[w.meta["body"], g[m]].T
        body[m, :3] = np.polynomial.chebyshev.chebval(sig[m], c)
        body[m, 3:] = np.polynomial.chebyshev.chebval(sig[m], np.polynomial.chebyshev.chebder(c)) * 2.0 / w.granule
    rel = x_ca - _dev(body)
    mu = w.meta["mu_body"]
    r, v = rel[:, :3], rel[:, 3:]
    hv = torch.linalg.cross(r, v)
    rn = r.norm(dim=1, keepdim=True)
    v2 = (v * v).sum(1, keepdim=True)
    ev = ((v2 - mu / rn) * r - (r * v).sum(1, keepdim=True) * v) / mu
    e = ev.norm(dim=1, keepdim=True)
    p = ev / e
    q = torch.linalg.cross(hv / hv.norm(dim=1, keepdim=True), p)
    s = p / e + torch.sqrt(e**2 - 1.0) / e * q
    z = torch.tensor([0.0, 0.0, 1.0], dtype=torch.float64, device="cuda").expand_as(s)
    tt = torch.linalg.cross(s, z)
    tt = tt / tt.norm(dim=1, keepdim=True)
    bv = torch.linalg.cross(s, hv) / torch.sqrt(v2 - 2.0 * mu / rn)
    plane = torch.stack([(bv * tt).sum(1), (bv * torch.linalg.cross(s, tt)).sum(1)])
    (g_plane,) = torch.autograd.grad((_dev(c_plane) * plane / 6052.0).sum(), x_ca)
    st.t.copy_(t_ca)
    st.y.copy_(torch.cat([x_ca.detach(), eye6], 1))
    gone, span = torch.zeros_like(t_ca), w.tf - t_ca
    while float((span - gone).max()) > 0:
        h = torch.minimum(span - gone, (0.1 * gone).clamp(100.0, 345600.0))
        st.step(h)
        gone = gone + h
    y = st.y
    xf, Phi2 = y[:, :6], y[:, 6:].reshape(-1, 6, 6)
    unit = torch.tensor([1e8] * 3 + [30.0] * 3, dtype=torch.float64, device="cuda")
    g_ca = torch.einsum("mij,mi->mj", Phi2, _dev(c_state).T / unit) + g_plane
    grad = torch.einsum("mij,mi->mj", Phi1, g_ca).T.contiguous()
    return {"xf": xf.T.contiguous(), "plane": plane.detach(), "grad_r": grad[:3], "grad_v": grad[3:]}


def exact(case, seed):
    if case["kind"] == "gradient":
        return _exact_gradient(case, seed)
    if case["kind"] == "uneven":
        return {"xf": _exact_uneven(case, seed).T.contiguous(), "status": None}
    w = _workload(case, seed)
    sky = _Sky(w)
    rhs = None
    if case["eih"]:
        rhs = lambda t, y: torch.cat([y[:, 3:6], sky.accel_eih(t, y[:, :3], y[:, 3:6])], 1)  # noqa: E731
    x = _integrate(sky, _dev(w.x0), w.t0, w.tf, rhs)
    return {"xf": x.T.contiguous(), "status": None}
