"""The solves whose speed this framework is judged by.

One pass of a case is a whole solve through the public entry points, as a
user's program makes it: sample the walkers, propagate them with their output
times, read the observables (`qcl.Run`, `qcl.SpawnRun`), or submit a batch of
requests to the request server and wait for them (`qcl.Server`).  The models
are those of `workloads.py`.  `exact` states the same solve in plain torch in
64 bits (the same Philox streams, the method's own equations), without the
library.
"""
import ctypes
import math

import numpy as np
import torch

from paper_2608_14544_gb300 import qcl
from paper_2608_14544_gb300 import workloads as wl


# ---------------------------------------------------------------- the cases --
def _solve(name, model, modes, walkers, steps, stride, dt, beta=0.0, repr="adiabatic",
           precision="fp32"):
    # (beta = 0: the ground state)
    return {"name": name, "call": "solve", "model": model, "modes": modes, "walkers": walkers,
            "steps": steps, "stride": stride, "dt": dt, "beta": beta, "repr": repr,
            "precision": precision}


def listed():
    return [
        # the one-mode spin-boson model at its stated size and precision: a small
        # reference run, bound by launches and by one step's latency
        _solve("sb1_fp64_small", "spin_boson", 1, 10_000, 1000, 10, 0.01, precision="fp64"),
        # the same run in bulk precision: the smallest solve a user makes
        _solve("sb1_fp32_small", "spin_boson", 1, 10_000, 1000, 10, 0.01),
        # the headline model at its walker count, over the time its estimator resolves
        _solve("sb3_fp32_large", "spin_boson", 3, 10_000_000, 200, 10, 0.01, beta=5.0),
        # the same model in the diabatic representation, an ordinary ragged size
        _solve("sb3_dia_fp32", "spin_boson", 3, 1_000_003, 200, 10, 0.01, beta=5.0,
               repr="diabatic"),
        # the vibronic model with a conical intersection (general two-state form)
        _solve("vib3_fp32", "vibronic", 3, 4_000_037, 200, 20, 0.05),
        # the 100-mode spin-boson bath
        _solve("sb100_fp32", "spin_boson", 100, 1_000_000, 100, 20, 0.005, beta=1.0),
        # the four-state model of the served mix
        _solve("lvc4_fp32", "lvc4", 6, 1_000_000, 50, 10, 0.01),
        # a four-state model with many modes
        _solve("lvc4_64mode_fp32", "lvc4", 64, 262_147, 30, 10, 0.01),
        # double precision at an ordinary size: two states, and four
        _solve("sb3_fp64", "spin_boson", 3, 1_000_000, 20, 10, 0.01, beta=5.0, precision="fp64"),
        _solve("lvc4_fp64", "lvc4", 6, 20_001, 20, 10, 0.01, precision="fp64"),
        # trajectory spawning: the benchmark's case (the walker count grows about
        # fifteenfold during the solve)
        {"name": "sb1_spawn_fp32", "call": "spawn", "model": "spin_boson", "modes": 1,
         "walkers": 100_000, "slots": 64, "steps": 400, "stride": 10, "dt": 0.01, "beta": 0.0,
         "repr": "adiabatic", "precision": "fp32"},
        # a batch of mixed small requests at the server
        {"name": "served_mix", "call": "serve", "requests": 16, "mix": 12345,
         "walkers_low": 10_000, "walkers_high": 200_000, "steps_low": 100, "steps_high": 300,
         "quantum": 400},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["spin_boson"] * 4 + ["vibronic", "lvc2", "lvc4", "lvc4", "fp64", "spawn",
                                            "serve"])
    if kind == "serve":
        lo = _log(rng, 1_000, 50_000)
        return {"call": "serve", "requests": rng.randint(2, 16), "mix": rng.randint(1, 10**6),
                "walkers_low": lo, "walkers_high": 4 * lo, "steps_low": 50, "steps_high": rng.randint(60, 300),
                "quantum": rng.choice([100, 200, 400])}
    stride = rng.choice([5, 10, 12, 20, 25])
    if kind == "spawn":
        prec = rng.choice(["fp32", "fp32", "fp64"])
        steps = stride * rng.randint(2, 200 // stride)
        return {"call": "spawn", "model": rng.choice(["spin_boson", "lvc2"]),
                "modes": rng.randint(1, 6), "walkers": _log(rng, 1_000, 60_000), "slots": 64,
                "steps": steps if prec == "fp32" else max(stride, steps // 2 // stride * stride),
                "stride": stride, "dt": 0.01, "beta": 0.0,
                "repr": rng.choice(["adiabatic", "diabatic"]), "precision": prec}
    if kind == "fp64":
        model = rng.choice(["spin_boson", "spin_boson", "vibronic", "lvc2", "lvc4"])
        modes = 3 if model == "vibronic" else _log(rng, 1, 12)
        most = 20_000_000 if model != "lvc4" else 400_000
        walkers = _log(rng, 2_000, most / 5 / stride / modes)
        steps = stride * max(1, min(40, int(most / walkers / stride / max(1, modes // 3))))
        dt = 0.05 if model == "vibronic" else 0.01
        return _drop_name(_solve("", model, modes, walkers, steps, stride, dt,
                                 repr=rng.choice(["adiabatic", "diabatic"]), precision="fp64"))
    rep = rng.choice(["adiabatic", "adiabatic", "diabatic"])
    if kind == "lvc4":
        modes, most, dt = _log(rng, 2, 64), 40_000_000, 0.01
        cost = 1.0 if modes <= 8 else modes / 8.0
    elif kind == "lvc2":
        modes, most, dt = _log(rng, 1, 100), 1_000_000_000, 0.01
        cost = max(1.0, modes / 4.0) * (3.0 if modes > 8 else 1.0)
    elif kind == "vibronic":
        modes, most, dt, cost = 3, 1_000_000_000, 0.05, 1.0
    else:
        modes, most, dt = _log(rng, 1, 100), 1_600_000_000, rng.choice([0.005, 0.01])
        cost = max(1.0, modes / 4.0) * (2.0 if modes > 8 else 1.0)
    most /= cost
    walkers = _log(rng, 5_000, most / 2 / stride)
    steps = stride * max(2, min(600 // stride, int(most / walkers / stride)))
    beta = rng.choice([0.0, 1.0, 5.0])
    return _drop_name(_solve("", kind, modes, walkers, steps, stride, dt, beta=beta, repr=rep))


def _drop_name(case):
    return {k: v for k, v in case.items() if k != "name"}


# ------------------------------------------------------------------ a solve --
def _model_init(case, seed):
    kind, n = case["model"], case["modes"]
    beta = case["beta"] or math.inf
    if kind == "spin_boson":
        if n == 1:
            m = wl.spin_boson(0.0, 0.5, [1.0], [1.0])
        elif n > 8:
            m = wl.spin_boson(1.0, 1.0, *wl.ohmic_modes(n, 0.25, 5.0))
        else:
            m = wl.spin_boson(0.5, 0.5, *wl.ohmic_modes(n, 0.5, 2.5))
        init = wl.sb_init(m, beta=beta)
    elif kind == "vibronic":
        m = wl.vibronic_ci()
        init = wl.vibronic_init(m)
    elif kind == "lvc2":
        m = wl.random_lvc2(n, seed % 1000)
        init = wl.sb_init(m, beta=beta)
    else:
        m = wl.random_lvc4(seed % 1000, n)
        init = wl.sb_init(m, beta=beta)
    m["repr"] = case["repr"]
    return m, init


def _requests(case, seed):
    # (the mix of models and sizes is the case's, the walkers' streams the seed's)
    reqs = wl.served_mix(case["requests"], seed=case["mix"],
                         traj_range=(case["walkers_low"], case["walkers_high"]),
                         steps_range=(case["steps_low"], case["steps_high"]))
    for r in reqs:
        r["seed"] = seed * 1000 + r["seed"]
    return reqs


def _precision(case):
    return qcl.PREC_FP64 if case["precision"] == "fp64" else qcl.PREC_FP32_BULK


def _arrays(buf, off, n, walkers, fp64):
    """The walker arrays inside an ensemble buffer (views)."""
    ft, w = (torch.float64, 8) if fp64 else (torch.float32, 4)

    def at(o, count, dtype, width):
        return buf[o:o + count * width].view(dtype)

    s = {"R": at(off[0], n * walkers, ft, w).view(n, walkers),
         "P": at(off[1], n * walkers, ft, w).view(n, walkers),
         "m": at(off[2], walkers, ft, w), "phi": at(off[4], walkers, ft, w),
         "pair": at(off[6], walkers, torch.int16, 2)}
    if not fp64:
        s["m_exp"] = at(off[8], walkers, torch.int32, 4)
    return s


def _spawn_arrays(r, which, n, fp64):
    """The walker slots of set `which` of a spawning ensemble (views)."""
    off = (ctypes.c_size_t * 12)()
    if qcl.load().qcl_spawn_layout(r.model.handle, ctypes.byref(r.ens), r.capacity, which, off):
        raise RuntimeError(qcl.last_error())
    ft, w, cap = (torch.float64, 8, r.capacity) if fp64 else (torch.float32, 4, r.capacity)

    def at(o, count, dtype, width):
        return r.buf[o:o + count * width].view(dtype)

    s = {"R": at(off[0], n * cap, ft, w).view(n, cap), "P": at(off[1], n * cap, ft, w).view(n, cap),
         "m": at(off[2], cap, ft, w), "phi": at(off[3], cap, ft, w),
         "pair": at(off[4], cap, torch.int16, 2), "id": at(off[5], cap, torch.int64, 8),
         "family": at(off[6], cap, torch.int32, 4)}
    if not fp64:
        s["m_exp"] = at(off[9], cap, torch.int32, 4)
    return s


def prepare(case, seed):
    if case["call"] == "serve":
        return {"case": case, "requests": _requests(case, seed),
                "server": qcl.Server(2 << 30, max_active=64, quantum_steps=case["quantum"])}
    m, init = _model_init(case, seed)
    model = qcl.Model(m)
    n_out = case["steps"] // case["stride"] + 1
    s = {"case": case, "model": model, "init": init}
    if case["call"] == "spawn":
        s["run"] = qcl.SpawnRun(model, case["walkers"], case["slots"] * case["walkers"], seed,
                                n_out, precision=_precision(case))
        s["state"] = _spawn_arrays(s["run"], case["steps"] & 1, case["modes"],
                                   case["precision"] == "fp64")
        s["run"].buf.zero_()  # (slots that no walker takes stay zero)
    else:
        s["run"] = qcl.Run(model, case["walkers"], seed, _precision(case), n_out)
        s["state"] = _arrays(s["run"].ens_buf, qcl.ensemble_layout(model, s["run"].ens),
                             case["modes"], case["walkers"], case["precision"] == "fp64")
    return s


def _rows(rows, ns):
    """The rows of qcl_reduce_observables by what their columns are."""
    q = 4 * ns * ns
    return {"mean": rows[:, :q], "error": rows[:, q:2 * q], "trace": rows[:, 2 * q:2 * q + 2],
            "walkers": rows[:, 2 * q + 2]}


def run(state):
    case = state["case"]
    if case["call"] == "serve":
        ids = [state["server"].submit(r) for r in state["requests"]]
        out = []
        for i, r in zip(ids, state["requests"]):
            st, rows = state["server"].wait(i)
            if st != qcl.REQ_DONE:
                raise RuntimeError("request failed: " + qcl.last_error())
            out.append(_rows(rows, r["model"]["n_states"]))
        return {"mean": np.concatenate([o["mean"].ravel() for o in out]),
                "error": np.concatenate([o["error"].ravel() for o in out]),
                "trace": np.concatenate([o["trace"].ravel() for o in out])}
    r = state["run"]
    r.sample(state["init"])
    r.propagate(case["steps"], case["dt"], case["stride"])
    out = _rows(r.observables(), state["model"].ns)
    if case["call"] == "spawn":
        out["n_live"] = r.n_live()
    out.update(state["state"])
    return out


# --------------------------------------------------------------------- work --
def _flops(ns, n, general):
    """Algorithmic operations of a walker's step: two states 10 a mode and 26
    (12 in the general form); more states 25 N_s^2 for the decomposition and
    the events and, a mode, the force, W and the coupling sum over K_j."""
    if ns == 2:
        return (12 if general else 10) * n + 26
    return 25 * ns * ns + n * (3 * ns * (ns + 1) + 10)


def work(case):
    if case["call"] == "serve":
        w = {"bytes": 0, "flops": 0}
        for r in _requests(case, 1):
            ns, n = r["model"]["n_states"], r["model"]["n_modes"]
            w["flops"] += r["n_traj"] * r["n_steps"] * _flops(ns, n, r["kind"] == 2)
            w["bytes"] += (r["n_steps"] // r["out_stride"] + 1) * (8 * ns * ns + 3) * 8
        return w
    ns = 4 if case["model"] == "lvc4" else 2
    n, rows = case["modes"], case["steps"] // case["stride"] + 1
    w = 8 if case["precision"] == "fp64" else 4
    state = 2 * n * w + (18 if w == 8 else 22) + (ns * ns * w + ns * 4 if ns > 2 else 0)
    f = _flops(ns, n, case["model"] != "spin_boson")
    out = rows * (8 * ns * ns + 3) * 8
    if case["call"] == "spawn":
        # every step starts from at least the initial walkers
        return {"bytes": case["walkers"] * (state + 12) + out,
                "flops": case["walkers"] * case["steps"] * f}
    return {"bytes": case["walkers"] * state + out, "flops": case["walkers"] * case["steps"] * f}


# ------------------------------------------------ the same solve in 64 bits --
_M32 = 0xFFFFFFFF
_P24 = 16777216.0


def _philox(c0, c1, c2, c3, seed):
    """Philox4x32-10 of counters (c0, c1, c2, c3) (int64 tensors or numbers,
    32-bit values): its four words."""
    k0, k1 = seed & _M32, (seed >> 32) & _M32
    c0, c1, c2, c3 = torch.broadcast_tensors(*[torch.as_tensor(c, dtype=torch.int64,
                                                               device="cuda")
                                               for c in (c0, c1, c2, c3)])
    for _ in range(10):
        p0, p1 = c0 * 0xD2511F53, c2 * 0xCD9E8D57
        c0, c1, c2, c3 = ((p1 >> 32) & _M32) ^ c1 ^ k0, p1 & _M32, \
            ((p0 >> 32) & _M32) ^ c3 ^ k1, p0 & _M32
        k0, k1 = (k0 + 0x9E3779B9) & _M32, (k1 + 0xBB67AE85) & _M32
    return c0, c1, c2, c3


def _turn(U, W):
    """U^T W U of [ns, ns, N] arrays."""
    ns = range(U.shape[0])
    X = sum(W[:, k, None] * U[None, k] for k in ns)
    return sum(U[k, :, None] * X[None, k] for k in ns)


class _Walkers:
    """N_s-state walkers of the method, one tensor entry each: R, P [n, N],
    eigenvalues e [ns, N] and eigenvectors U [ns, ns, N] (adiabatic), weight m,
    phase phi, pair (a, b), quarter turns q, random-stream id (lo, hi)."""

    def __init__(self, m, init, n_traj, seed, dt):
        f = dict(dtype=torch.float64, device="cuda")
        t = lambda x: torch.as_tensor(np.asarray(x, dtype=np.float64), **f)  # noqa: E731
        self.ns, self.n, self.hbar, self.dt, self.seed = (m["n_states"], m["n_modes"], m["hbar"],
                                                          dt, seed)
        self.kappa, self.pmax = m["hop_scale"], m["p_max"]
        self.dia = m.get("repr") == "diabatic"
        mass, omega = np.asarray(m["mass"]), np.asarray(m["omega"])
        self.E, self.K = t(m["E"]), t(m["K"])
        self.mass, self.k = t(mass)[:, None], t(mass * omega**2)[:, None]
        self.Kflat = self.K.reshape(self.n, -1)
        self.lo = torch.arange(n_traj, dtype=torch.int64, device="cuda")
        self.hi = torch.zeros_like(self.lo)
        ns, n = self.ns, self.n
        beta = init["beta"]
        cth = np.ones(n) if math.isinf(beta) else 1 / np.tanh(0.5 * beta * m["hbar"] * omega)
        sR = np.sqrt(m["hbar"] / (2 * mass * omega) * cth)
        sP = np.sqrt(0.5 * m["hbar"] * mass * omega * cth)
        self.R, self.P = torch.empty(n, n_traj, **f), torch.empty(n, n_traj, **f)
        for j in range(n):
            x, y, _, _ = _philox(j, self.lo, self.hi, 1, seed)
            rad = torch.sqrt(-2 * torch.log((x.double() + 0.5) * 2.0**-32))
            ang = 2 * math.pi * ((y.double() + 0.5) * 2.0**-32)
            self.R[j] = init["R0"][j] + sR[j] * rad * torch.cos(ang)
            self.P[j] = init["P0"][j] + sP[j] * rad * torch.sin(ang)
        W = self.elec()
        self.W = W
        self.e, self.U = self.decompose(W, None)
        rho = t(init["rho_el0"])
        rho = rho[:, :, None].expand(ns, ns, n_traj) if self.dia else \
            _turn(self.U, rho[:, :, None])
        rho = rho.reshape(ns * ns, n_traj)
        T = torch.floor(rho.abs() / rho.abs().sum(0) * _P24).long()
        last = torch.where(rho != 0, torch.arange(ns * ns, device="cuda")[:, None], -1).amax(0)
        T.scatter_add_(0, last[None], (16777216 - T.sum(0))[None])
        y = _philox(n, self.lo, self.hi, 1, seed)[0] >> 8
        pick = torch.minimum((y[None] >= T.cumsum(0)).sum(0), last)
        self.m = rho.gather(0, pick[None])[0] / (T.gather(0, pick[None])[0].double() / _P24)
        self.a, self.b = pick // ns, pick % ns
        self.phi, self.q = torch.zeros(n_traj, **f), torch.zeros_like(self.a)

    def elec(self):
        return self.E[:, :, None] + (self.Kflat.T @ self.R).reshape(self.ns, self.ns, -1)

    def decompose(self, W, ref):
        """Ascending eigenvalues and eigenvectors; signs follow `ref`, or make
        each vector's largest component positive."""
        ns = self.ns
        if ns == 2:  # the closed form, theta = atan2(b, a) / 2
            s, a, b = 0.5 * (W[0, 0] + W[1, 1]), 0.5 * (W[0, 0] - W[1, 1]), W[0, 1]
            r, th = torch.hypot(a, b), 0.5 * torch.atan2(b, a)
            c, sn = torch.cos(th), torch.sin(th)
            return torch.stack([s - r, s + r]), torch.stack([torch.stack([-sn, c]),
                                                             torch.stack([c, sn])])
        if ref is None:
            A, V, sweeps = W.clone(), torch.zeros_like(W), 8
            for i in range(ns):
                V[i, i] = 1.0
        else:
            A, V, sweeps = _turn(ref, W), ref.clone(), 4
        for _ in range(sweeps):  # cyclic Jacobi
            for p in range(ns):
                for q in range(p + 1, ns):
                    apq = A[p, q].clone()
                    zero = apq == 0
                    tau = (A[q, q] - A[p, p]) / (2 * torch.where(zero, 1.0, apq))
                    t = torch.where(tau >= 0, 1.0, -1.0) / (tau.abs() + torch.sqrt(1 + tau * tau))
                    t = torch.where(zero, 0.0, t)
                    c = 1 / torch.sqrt(1 + t * t)
                    s = t * c
                    A[:, p], A[:, q] = c * A[:, p] - s * A[:, q], s * A[:, p] + c * A[:, q]
                    A[p], A[q] = c * A[p] - s * A[q], s * A[p] + c * A[q]
                    V[:, p], V[:, q] = c * V[:, p] - s * V[:, q], s * V[:, p] + c * V[:, q]
        d = torch.diagonal(A, dim1=0, dim2=1).T
        rank = torch.stack([sum(((d[j] < d[i]) | ((d[j] == d[i]) if j < i else False)).long()
                                for j in range(ns) if j != i) for i in range(ns)])
        e = torch.empty_like(d).scatter_(0, rank, d)
        U = torch.empty_like(V).scatter_(1, rank[None].expand(ns, ns, -1), V)
        lead = (U * ref).sum(0) if ref is not None else \
            U.gather(0, U.abs().argmax(0)[None])[0]
        return e, U * torch.where(lead < 0, -1.0, 1.0)

    def col(self, U, a):
        return U.gather(1, a[None, None].expand(self.ns, 1, -1))[:, 0]

    def force(self):
        if self.dia:
            d = torch.diagonal(self.K, dim1=1, dim2=2)  # [n, ns]
            g = 0.5 * (d[:, self.a] + d[:, self.b])
        else:
            ua, ub = self.col(self.U, self.a), self.col(self.U, self.b)
            Q = 0.5 * (ua[:, None] * ua[None] + ub[:, None] * ub[None])
            g = self.Kflat @ Q.reshape(self.ns**2, -1)
        return -self.k * self.R - g

    def gap(self):
        e = torch.diagonal(self.W, dim1=0, dim2=1).T if self.dia else self.e
        return (e.gather(0, self.a[None])[0] - e.gather(0, self.b[None])[0]) / self.hbar

    def step(self, n):
        """Everything of step n but the event's outcome; returns the event
        drawn (-1: none), its amplitude and probability, and all events'."""
        ns, dt = self.ns, self.dt
        w0 = self.gap()
        self.P = self.P + 0.5 * dt * self.force()
        self.R = self.R + dt * self.P / self.mass
        self.W = self.elec()
        if not self.dia:
            self.e, self.U = self.decompose(self.W, self.U)
        self.P = self.P + 0.5 * dt * self.force()
        self.phi = self.phi + 0.5 * dt * (w0 + self.gap())
        nu = torch.arange(ns, device="cuda")[:, None]
        other = torch.cat([nu != self.a, nu != self.b])
        if self.dia:
            c = self.W * dt / self.hbar
            A = torch.cat([self.col(c, self.a), self.col(c, self.b)])
        else:
            v = self.P / self.mass
            G = (self.Kflat.T @ v).reshape(ns, ns, -1)
            D = _turn(self.U, G)
            ea, eb = self.e.gather(0, self.a[None]), self.e.gather(0, self.b[None])
            gap = torch.cat([ea - self.e, self.e - eb])
            ok = other & (gap.abs() >= 1e-12)
            sign = torch.cat([torch.full((ns, 1), -dt, device="cuda", dtype=torch.float64),
                              torch.full((ns, 1), dt, device="cuda", dtype=torch.float64)])
            A = sign * torch.cat([self.col(D, self.a), self.col(D, self.b)]) \
                / torch.where(ok, gap, 1.0) * ok
        T = torch.floor(torch.clamp(self.kappa * A.abs(), max=self.pmax) * _P24).long() * other
        Tmax, tot = int(math.floor(self.pmax * _P24)), T.sum(0)
        T = torch.where(tot > Tmax, T * Tmax // torch.clamp(tot, min=1), T)
        if n & 3 == 0 or self.words is None:
            self.words = _philox(n >> 2, self.lo, self.hi, 2, self.seed)
        y = self.words[n & 3] >> 8
        hit = (y[None] >= T.cumsum(0)).sum(0)
        hop = hit < 2 * ns
        at = torch.clamp(hit, max=2 * ns - 1)[None]
        return (torch.where(hop, hit, -1), A.gather(0, at)[0],
                T.gather(0, at)[0].double() / _P24, T.sum(0).double() / _P24)

    words = None

    def moved(self, hit):
        """(a, b, q) after event `hit` (where it is one)."""
        first, second = (hit >= 0) & (hit < self.ns), hit >= self.ns
        q = (self.q + torch.where(first, 3, torch.where(second, 1, 0))) & 3 if self.dia else self.q
        return torch.where(first, hit, self.a), torch.where(second, hit - self.ns, self.b), q

    def hop(self, n):
        hit, A, p, tot = self.step(n)
        go = hit >= 0
        self.m = self.m * torch.where(go, A / torch.where(go, p, 1.0), 1 / (1 - tot))
        self.a, self.b, self.q = self.moved(hit)

    def spawn(self, n):
        """A fired event leaves its walker and adds a child after it."""
        hit, A, p, _ = self.step(n)
        go = hit >= 0
        mc = self.m * torch.where(go, A / torch.where(go, p, 1.0), 0.0)
        ca, cb, cq = self.moved(hit)
        w0, w1, _, _ = _philox(n, self.lo, self.hi, 3, self.seed)
        idx = torch.repeat_interleave(torch.arange(go.numel(), device="cuda"), 1 + go.long())
        child = torch.zeros_like(idx, dtype=torch.bool)
        child[1:] = idx[1:] == idx[:-1]
        pickc = lambda old, new: torch.where(child, new[idx], old[idx])  # noqa: E731
        self.m, self.a, self.b, self.q = (pickc(self.m, mc), pickc(self.a, ca), pickc(self.b, cb),
                                          pickc(self.q, cq))
        self.lo, self.hi = pickc(self.lo, w0), pickc(self.hi, w1 | 0x80000000)
        self.R, self.P, self.phi = self.R[:, idx], self.P[:, idx], self.phi[idx]
        self.W, self.family = self.W[:, :, idx], self.family[idx]
        self.e, self.U = self.e[:, idx], self.U[:, :, idx]
        self.words = None

    def observe(self, families=None):
        ns = self.ns
        z = torch.polar(self.m, -self.phi) * torch.tensor([1, 1j, -1, -1j], device="cuda",
                                                          dtype=torch.complex128)[self.q]
        own = torch.zeros(ns * ns, z.numel(), dtype=z.dtype, device="cuda")
        own.scatter_(0, (self.a * ns + self.b)[None], z[None])
        if self.dia:
            _, U = self.decompose(self.W, None)
            U = U.transpose(0, 1)
        else:
            U = self.U
        o = (self.col(U, self.a)[:, None] * self.col(U, self.b)[None] * z).reshape(ns * ns, -1)
        x = torch.cat([own, o] if self.dia else [o, own])
        x = torch.view_as_real(x).transpose(1, 2).reshape(4 * ns * ns, -1)
        N = x.shape[1]
        if families is not None:
            N = families
            x = torch.zeros(x.shape[0], N, dtype=x.dtype, device="cuda").index_add_(
                1, self.family, x)
        S, S2 = x.sum(1), (x * x).sum(1)
        se = torch.sqrt(torch.clamp(S2 - S * S / N, min=0) / max(N - 1, 1) / N)
        tr = sum(S[2 * (i * ns + i):2 * (i * ns + i) + 2] for i in range(ns)) / N
        return torch.cat([S / N, se, tr, torch.tensor([float(N)], device="cuda",
                                                      dtype=torch.float64)])


def _exact_rows(m, init, walkers, seed, dt, steps, stride, spawn=False):
    w = _Walkers(m, init, walkers, seed, dt)
    fam = walkers if spawn else None
    if spawn:
        w.family = w.lo.clone()
    rows = [w.observe(fam)]
    for n in range(steps):
        w.spawn(n) if spawn else w.hop(n)
        if (n + 1) % stride == 0:
            rows.append(w.observe(fam))
    return torch.stack(rows).cpu().numpy(), w


def exact(case, seed):
    if case["call"] == "serve":
        if case["requests"] * case["steps_high"] > 5000:
            return None  # (past about 20 seconds)
        out = [_rows(_exact_rows(r["model"], r["init"], r["n_traj"], r["seed"], r["dt"],
                                 r["n_steps"], r["out_stride"])[0], r["model"]["n_states"])
               for r in _requests(case, seed)]
        return {k: np.concatenate([o[k].ravel() for o in out]) for k in ("mean", "error", "trace")}
    m, init = _model_init(case, seed)
    rows, w = _exact_rows(m, init, case["walkers"], seed, case["dt"], case["steps"],
                          case["stride"], case["call"] == "spawn")
    out = _rows(rows, m["n_states"])
    if case["call"] == "spawn":
        return out
    out.update({"R": w.R, "P": w.P, "pair": None})
    if case["precision"] == "fp64":
        out.update({"m": w.m, "phi": w.phi})
    else:  # the weight's mantissa and exponent, and the reduced phase, are the code's own form
        out.update({"m": None, "m_exp": None, "phi": None})
    return out
