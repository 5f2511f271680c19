"""Cases by which the speed of this library is measured: the calls a user's program makes, through the public
entry points of paper_2011_07978_gb300.dlbchem, over the sizes this repository's configurations, tests and
benchmark use.

A case is a dict of plain values with an "op":

* integrate: dlbchem.Context.integrate (device arrays) or integrate_host (host arrays) of a field over one flow
  step: the operator-split chemistry step. Attempted steps are the queue's cost key: the call reads the counts of
  the call before and writes its own, as a flow solver's time loop does. They are not among the outputs: a count
  may move by one where an error norm lies within rounding of 1 (tests/test_oracle_rounding.py).
* batch: dlbchem.Batch, meshes over two mechanisms in one captured graph.
* rhs: dlbchem.Context.rhs, f(y) of every cell.
* forward, train: dlbchem.MLP, inference of the learned predictor and one training step.

States. "uniform": T U[300, 2500] K, Dirichlet(0.5) mass fractions (synth.states.uniform_states). "flame": the
burnt and the flame-front cells of synth.states.bimodal_states, 90 % near-equilibrium (stored bases with a relative
noise of 1e-6) and 10 % front (T U[900, 1600] K, Dirichlet(0.5)), in random order. The flow steps are 2e-7 s (the
paper's spray) to 1e-6 s. The bimodal field's cold ambient cells and steps of 1e-5 s are left out, and the 10-species
mechanism runs at rtol 1e-8, atol 1e-12: there the equations amplify a last-bit change of the input to more than 1e-9
in the result of some cells, so that two correct programs cannot be compared (tests/test_oracle_rounding.py).
"""
from __future__ import annotations

import math
import os

import numpy as np
import torch

from paper_2011_07978_gb300 import dlbchem

DATA = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "synth", "data")
DEV = "cuda"
F64 = torch.float64
MECH = {10: (10, 20, 0), 53: (53, 325, 0), 100: (100, 1000, 1)}   # species: (species, reactions, seed)
HIDDEN = 256


def _integrate(name, nsp, n, dt, states="uniform", p=101325.0, rtol=1e-6, atol=1e-10, queue=True, mapping=0,
               precision=0, host=False):
    return {"name": name, "op": "integrate", "nsp": nsp, "n": n, "dt": dt, "states": states, "p": p, "rtol": rtol,
            "atol": atol, "queue": queue, "mapping": mapping, "precision": precision, "host": host}


def listed():
    return [
        # one right-hand side: a solver that probes a single cell (launch latency)
        {"name": "rhs_53sp_1", "op": "rhs", "nsp": 53, "n": 1},
        # f(y) of the benchmark's field size, as the residual surrogate's training targets need it
        {"name": "rhs_53sp_262144", "op": "rhs", "nsp": 53, "n": 262144},
        # a CPU flow solver's small patch, host buffers, default schedule
        _integrate("host_10sp_64", 10, 64, 1e-6, rtol=1e-8, atol=1e-12, queue=False, host=True),
        # the 10-species configuration with the work queue
        _integrate("queue_10sp_4096", 10, 4096, 1e-6, rtol=1e-8, atol=1e-12),
        # the 53-species mesh of the batched configuration, a ragged number of cells
        _integrate("queue_53sp_4001", 53, 4001, 1e-6),
        # the benchmark's form: queue and one reference per state bucket on a partly burnt field at 20 bar
        _integrate("flame_53sp_32768", 53, 32768, 2e-7, states="flame", p=20e5, rtol=1e-5, atol=1e-8, mapping=2),
        # a field that is burnt out almost everywhere: classification, mapping and ordering of many cheap cells
        _integrate("burnt_53sp_262144", 53, 262144, 2e-7, states="burnt", p=20e5, rtol=1e-5, atol=1e-8, mapping=2),
        # the caller's choice of an FP32 factorisation
        _integrate("mixed_53sp_1500", 53, 1500, 1e-6, precision=1),
        # the large mechanism, one cell per team in index order
        _integrate("plain_100sp_400", 100, 400, 1e-6, queue=False),
        # uneven meshes over two mechanisms in one graph (the batched configuration's mix of sizes and steps, scaled down)
        {"name": "batch_53sp_100sp", "op": "batch", "n0": 256, "n1": 100, "n2": 1000, "dt": 2e-7},
        # inference of the predictor on the benchmark's field size
        {"name": "forward_10sp_262144", "op": "forward", "nsp": 10, "n": 262144},
        # one step of the training loop with its default batch
        {"name": "train_10sp_4096", "op": "train", "nsp": 10, "n": 4096},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _dt(rng, lo, hi):
    return float("%.3g" % math.exp(rng.uniform(math.log(lo), math.log(hi))))


def draw(rng):
    op = rng.choice(["rhs", "forward", "train", "train", "i10", "i53", "i53", "flame", "flame", "burnt", "mixed", "i100",
                     "batch"])
    if op == "rhs":
        return {"op": "rhs", "nsp": rng.choice([10, 53, 53, 100]), "n": _log(rng, 1, 100000)}
    if op in ("forward", "train"):
        return {"op": op, "nsp": rng.choice([10, 53]), "n": _log(rng, 64, 262144 if op == "forward" else 16384)}
    if op == "i10":
        c = _integrate("", 10, _log(rng, 16, 4096), _dt(rng, 2e-7, 1e-6), rtol=1e-8, atol=1e-12,
                       queue=rng.random() < 0.5, host=rng.random() < 0.3)
    elif op == "i53":
        c = _integrate("", 53, _log(rng, 16, 4001), _dt(rng, 2e-7, 1e-6), queue=rng.random() < 0.7,
                       host=rng.random() < 0.3)
    elif op == "flame":
        c = _integrate("", 53, _log(rng, 1000, 32768), 2e-7, states="flame", p=20e5, rtol=1e-5, atol=1e-8,
                       mapping=rng.choice([0, 2, 2]))
    elif op == "burnt":
        c = _integrate("", 53, _log(rng, 10000, 262144), 2e-7, states="burnt", p=20e5, rtol=1e-5, atol=1e-8, mapping=2)
    elif op == "mixed":
        c = _integrate("", 53, _log(rng, 16, 1500), _dt(rng, 2e-7, 1e-6), precision=1)
    elif op == "i100":
        c = _integrate("", 100, _log(rng, 16, 400), _dt(rng, 2e-7, 1e-6), queue=rng.random() < 0.5)
    else:
        return {"op": "batch", "n0": _log(rng, 16, 256), "n1": _log(rng, 16, 100), "n2": _log(rng, 64, 1000),
                "dt": _dt(rng, 2e-7, 1e-6)}
    del c["name"]
    return c


def mech_path(nsp):
    return os.path.join(DATA, "mech_%d_%d_s%d.bin" % MECH[nsp])


# ---- inputs -------------------------------------------------------------------------------------------------

def _gen(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed))
    return g


def _uniform(g, n, lo, hi):
    return torch.rand(n, generator=g, device=DEV, dtype=F64) * (hi - lo) + lo


def _dirichlet(g, nsp, n):
    """Dirichlet(0.5) columns: normalised chi-square(1) variates."""
    z = torch.randn(nsp, n, generator=g, device=DEV, dtype=F64).square_()
    return z / z.sum(0, keepdim=True)


def _states(kind, nsp, n, p, seed):
    g = _gen(seed)
    T, Y = _uniform(g, n, 300.0, 2500.0), _dirichlet(g, nsp, n)
    if kind in ("flame", "burnt"):
        base = np.load(os.path.join(DATA, "burnt_base_%d_%d_s%d.npz" % MECH[nsp]))
        Tb, Yb = torch.tensor(base["T"], device=DEV), torch.tensor(base["Y"], device=DEV)
        which = torch.randint(Tb.numel(), (n,), generator=g, device=DEV)
        noise = lambda *s: 1.0 + (torch.rand(*s, generator=g, device=DEV, dtype=F64) * 2.0 - 1.0) * 1e-6
        Tw, Yw = Tb[which] * noise(n), Yb[:, which] * noise(nsp, n)
        # 10 % front cells; the burnt-out field keeps one in 2,000
        front = torch.rand(n, generator=g, device=DEV, dtype=F64) < (0.1 if kind == "flame" else 5e-4)
        T = torch.where(front, _uniform(g, n, 900.0, 1600.0), Tw)
        Y = torch.where(front, Y, Yw / Yw.sum(0, keepdim=True))
    return T, torch.full((n,), float(p), device=DEV, dtype=F64), Y.contiguous()


def _meshes(c):
    return [(53, c["n0"], 1e-6), (100, c["n1"], 1e-6), (53, c["n2"], c["dt"])]


def _net_io(c, seed):
    """Parameters (He-normal weights, zero biases), normalised inputs and targets."""
    n_in, n_out = c["nsp"] + 3, c["nsp"] + 2
    g = _gen(seed)
    rn = lambda *s: torch.randn(*s, generator=g, device=DEV)
    dims = [n_in, HIDDEN, HIDDEN, HIDDEN, n_out]
    parts = []
    for a, b in zip(dims[:-1], dims[1:]):
        parts += [(rn(a, b) * math.sqrt(2.0 / a)).reshape(-1), torch.zeros(b, device=DEV)]
    return dims, torch.cat(parts), rn(c["n"], n_in), rn(c["n"], n_out)


def prepare(case, seed):
    c = case
    if c["op"] in ("forward", "train"):
        dims, params, X, Y = _net_io(c, seed)
        net = dlbchem.MLP(dims[0], HIDDEN, dims[-1])
        net.set_params(params)
        s = {"op": c["op"], "net": net, "X": X}
        if c["op"] == "forward":
            s["out"] = torch.empty(c["n"], dims[-1], device=DEV)
        else:
            s.update(Y=Y, grad=torch.empty(net.nparams, device=DEV), loss=torch.zeros(1, device=DEV))
        return s
    if c["op"] == "batch":
        b = dlbchem.Batch(rtol=1e-6, atol=1e-10)
        out = []
        for i, (nsp, n, dt) in enumerate(_meshes(c)):
            T, p, Y = _states("uniform", nsp, n, 101325.0, 10 * seed + i)
            To, Yo = torch.empty_like(T), torch.empty_like(Y)
            st, ss = (torch.zeros(n, dtype=torch.int32, device=DEV) for _ in range(2))
            b.add(mech_path(nsp), T, p, Y, dt, To, Yo, steps=st, status=ss)
            out += [To, Yo, ss]
        stream = torch.cuda.Stream()
        torch.cuda.synchronize()
        b.capture(stream)
        return {"op": "batch", "batch": b, "stream": stream, "out": out}
    if c["op"] == "rhs":
        T, p, Y = _states("uniform", c["nsp"], c["n"], 101325.0, seed)
        return {"op": "rhs", "ctx": dlbchem.Context(mech_path(c["nsp"])), "in": (T, p, Y),
                "out": (torch.empty_like(T), torch.empty_like(Y))}
    T, p, Y = _states(c["states"], c["nsp"], c["n"], c["p"], seed)
    ctx = dlbchem.Context(mech_path(c["nsp"]), rtol=c["rtol"], atol=c["atol"], mapping=c["mapping"],
                          schedule=dlbchem.SCHED_QUEUE if c["queue"] else dlbchem.SCHED_PLAIN,
                          precision=c["precision"])
    st, ss = (torch.zeros(c["n"], dtype=torch.int32, device=DEV) for _ in range(2))
    s = {"op": "integrate", "ctx": ctx, "dt": c["dt"], "host": c["host"], "in": (T, p, Y),
         "out": (torch.empty_like(T), torch.empty_like(Y)), "steps": st, "status": ss}
    if c["host"]:
        s["in"], s["out"] = (tuple(t.cpu().pin_memory() for t in s[k]) for k in ("in", "out"))
        s["steps"], s["status"] = st.cpu(), ss.cpu()
    return s


def run(state):
    s = state
    if s["op"] == "integrate":
        f = s["ctx"].integrate_host if s["host"] else s["ctx"].integrate
        f(*s["in"], s["dt"], T_out=s["out"][0], Y_out=s["out"][1], steps=s["steps"], status=s["status"])
        return [s["out"][0], s["out"][1], s["status"]]
    if s["op"] == "rhs":
        return list(s["ctx"].rhs(*s["in"], fT=s["out"][0], fY=s["out"][1]))
    if s["op"] == "batch":
        s["stream"].wait_stream(torch.cuda.current_stream())
        s["batch"].launch(s["stream"])
        torch.cuda.current_stream().wait_stream(s["stream"])
        return s["out"]
    if s["op"] == "forward":
        return [s["net"].forward(s["X"], s["out"])]
    s["net"].grad(s["X"], s["Y"], grad=s["grad"], loss=s["loss"])
    s["net"].adam(1e-3, grad=s["grad"])
    return [s["grad"], s["loss"]]


# ---- work ---------------------------------------------------------------------------------------------------

def _step_flops(nsp):
    """Flops of one attempted step (bench.py, flops_per_step)."""
    R, N = MECH[nsp][1], nsp + 1
    return (2.0 / 3.0) * N**3 + 8.0 * N**2 + 3 * (25 * R + 15 * nsp) + 90 * R + 3 * N**2


def _steps(nsp, dt, states="uniform"):
    """Attempted steps of a cell, as the integrator counts them on average on these states."""
    if states == "flame":
        return 0.1 * 208
    if states == "burnt":
        return 5e-4 * 208
    at, slope = {10: (2350, 0.13), 53: (390, 0.14), 100: (520, 0.14)}[nsp]
    return at * (dt / 1e-6) ** slope


def work(case):
    c = case
    n = c.get("n", 0)
    if c["op"] in ("forward", "train"):
        n_in, n_out = c["nsp"] + 3, c["nsp"] + 2
        mul = n_in * HIDDEN + 2 * HIDDEN * HIDDEN + HIDDEN * n_out
        par = 4 * (mul + 3 * HIDDEN + n_out)
        if c["op"] == "forward":
            return {"bytes": 4 * n * (n_in + n_out) + par, "flops": 2.0 * n * mul}
        # forward, weight gradients and input gradients (none for the first layer); Adam reads the parameters, the
        # gradient and two moments and writes all but the gradient, which the backward pass writes
        return {"bytes": 4 * n * (n_in + n_out) + 8 * par, "flops": 2.0 * n * (3 * mul - n_in * HIDDEN)}
    if c["op"] == "batch":
        m = _meshes(c)
        return {"bytes": sum(8 * k * (2 * nsp + 3) + 12 * k for nsp, k, _ in m),
                "flops": sum(k * _steps(nsp, dt) * _step_flops(nsp) for nsp, k, dt in m)}
    nsp = c["nsp"]
    if c["op"] == "rhs":
        return {"bytes": 8 * n * (2 * nsp + 3), "flops": float(n) * (25 * MECH[nsp][1] + 15 * nsp)}
    return {"bytes": 8 * n * (2 * nsp + 3) + 12 * n,
            "flops": n * _steps(nsp, c["dt"], c["states"]) * _step_flops(nsp)}


# ---- the same results in 64 bits, by torch alone ------------------------------------------------------------

R_GAS, RC, T0 = 8.314462618, 82.05736, 298.15


class _Mech:
    """A DLBMECH1 file without optional sections: linear cp, Arrhenius, unit third-body efficiencies."""

    def __init__(self, nsp):
        b = open(mech_path(nsp), "rb").read()
        _, R, nelem, neff = np.frombuffer(b, np.int32, 4, 8)
        assert neff == 0
        d = lambda a: torch.tensor(np.ascontiguousarray(a), device=DEV)
        self.W, self.a, self.b, self.hf, self.s0 = (d(v) for v in np.frombuffer(b, np.float64, 5 * nsp, 24).reshape(5, nsp))
        rec = np.frombuffer(b, np.dtype([("k", "<f8", 3), ("i", "<i4", 16)]), R, 24 + 40 * nsp + 4 * nsp * nelem)
        self.lnA, self.beta, self.Ea = (d(v) for v in rec["k"].T)
        v = rec["i"]
        self.rev, self.tb = d(v[:, 2].astype(float)), d(v[:, 3].astype(float))
        slots, nu = np.full((R, 6), nsp), np.zeros((R, nsp))
        for r in range(R):
            for side, (cnt, i0, m0) in enumerate(((v[r, 0], 4, 7), (v[r, 1], 10, 13))):
                s = [k for i in range(cnt) for k in [v[r, i0 + i]] * v[r, m0 + i]]
                slots[r, 3 * side:3 * side + len(s)] = s
                for k in s:
                    nu[r, k] += 2 * side - 1
        self.slots, self.nu, self.dnu, self.nsp = d(slots), d(nu), d(nu.sum(1)), nsp
        # entries of dwdot/dc: (reaction, slot) -> (species, slot's species)
        ent = [(r * 6 + s, k * nsp + slots[r, s], nu[r, k]) for r in range(R) for s in range(6) if slots[r, s] < nsp
               for k in np.flatnonzero(nu[r])]
        self.e_src, self.e_dst = d([e[0] for e in ent]), d([e[1] for e in ent])
        self.e_nu = d([e[2] for e in ent])

    def thermo(self, T):
        h = self.hf + self.a * (T - T0) + 0.5 * self.b * (T * T - T0 * T0)
        return h, self.s0 + self.a * torch.log(T / T0) + self.b * (T - T0), self.a + self.b * T

    def f(self, y, p, jac=False):
        """f(y) of [B, 1 + nsp] states, and its Jacobian."""
        B, nsp, T, Yv = y.shape[0], self.nsp, y[:, :1], y[:, 1:]
        P1 = 1e-6 * p[:, None] / R_GAS
        S = (Yv / self.W).sum(1, keepdim=True)
        rho = P1 / (T * S)
        c = rho * Yv / self.W
        h, s, cpk = self.thermo(T)
        kf = torch.exp(self.lnA + self.beta * torch.log(T) - self.Ea / (R_GAS * T))
        dg = (h / (R_GAS * T) - s / R_GAS) @ self.nu.T
        kr = self.rev * kf * torch.exp(dg + self.dnu * torch.log(RC * T))
        x = torch.cat([c, torch.ones_like(T)], 1)[:, self.slots]
        M = 1.0 + self.tb * (c.sum(1, keepdim=True) - 1.0)
        pf, pr = kf * x[:, :, :3].prod(2), kr * x[:, :, 3:].prod(2)
        q = M * (pf - pr)
        wd = q @ self.nu
        cp = (Yv * cpk / self.W).sum(1, keepdim=True)
        Q = (h * wd).sum(1, keepdim=True)
        f = torch.cat([-Q / (rho * cp), self.W * wd / rho], 1)
        if not jac:
            return f
        oth = torch.stack([x[:, :, i] * x[:, :, j] for i, j in ((1, 2), (0, 2), (0, 1), (4, 5), (3, 5), (3, 4))], 2)
        D = oth * torch.stack([M * kf] * 3 + [-M * kr] * 3, 2)
        A = torch.zeros(B, nsp * nsp, device=DEV, dtype=F64)
        A.index_add_(1, self.e_dst, D.reshape(B, -1)[:, self.e_src] * self.e_nu)
        A = A.view(B, nsp, nsp) + ((self.tb * (pf - pr)) @ self.nu)[:, :, None]
        Ac = (A @ c[:, :, None])[:, :, 0]
        dlf = self.beta / T + self.Ea / (R_GAS * T * T)
        dlr = dlf - ((h @ self.nu.T) / (R_GAS * T * T) - self.dnu / T)
        wT = (M * (pf * dlf - pr * dlr)) @ self.nu - Ac / T
        iSW = 1.0 / (S * self.W)
        wY = A * (rho / self.W)[:, None, :] - Ac[:, :, None] * iSW[:, None, :]
        J = torch.empty(B, nsp + 1, nsp + 1, device=DEV, dtype=F64)
        J[:, 1:, 1:] = (self.W / rho)[:, :, None] * (wY + wd[:, :, None] * iSW[:, None, :])
        J[:, 1:, 0] = self.W / rho * (wT + wd / T)
        rc = rho * cp
        J[:, 0, 1:] = -(h[:, None, :] @ wY)[:, 0] / rc - Q / rc * iSW + Q / (rc * cp) * cpk / self.W
        dQ = (cpk * wd + h * wT).sum(1, keepdim=True)
        J[:, 0, :1] = -dQ / rc - Q / rc / T + Q / (rc * cp) * (Yv * self.b / self.W).sum(1, keepdim=True)
        return f, J


GAMMA = 0.57282
A2, A3 = (2.0,), (1.867943637803922, 0.2344449711399156)
C2, C3 = (-7.137615036412310,), (2.580708087951457, 0.6515950076447975)
C4 = (-2.137148994382534, -0.3214669691237626, -0.6949742501781779)
MU = (2.255570073418735, 0.2870493262186792, 0.4353179431840180, 1.093502252409163)
ER = (-0.2815431932141155, -0.07276199124938920, -0.1082196201495311, -1.093502252409163)


def _integrate64(m, T, p, Y, dt, rtol, atol):
    """The same Rosenbrock method (Hairer and Wanner, Solving ODEs II, Sec. IV.7) over all cells at once."""
    y = torch.cat([T[:, None], Y.T], 1)
    N = y.shape[1]
    norm = lambda v, sc: ((v / sc).square().sum(1) / N).sqrt()
    f0 = m.f(y, p)
    sc = atol + rtol * y.abs()
    d0, d1 = norm(y, sc), norm(f0, sc)
    h0 = torch.where((d0 < 1e-5) | (d1 < 1e-5), torch.full_like(d0, 1e-6 * dt), 0.01 * d0 / d1).clamp(max=dt)
    d2 = norm(m.f(y + h0[:, None] * f0, p) - f0, sc) / h0
    dm = torch.maximum(d1, d2)
    h1 = torch.where(dm <= 1e-15, (h0 * 1e-3).clamp(min=1e-6 * dt), (0.01 / dm) ** 0.25)
    h = torch.where(torch.isfinite(d2), torch.minimum(100.0 * h0, h1).clamp(max=dt), h0)
    done, idx = torch.empty_like(y), torch.arange(y.shape[0], device=DEV)
    t, rej = torch.zeros_like(h), torch.zeros_like(h, dtype=torch.bool)
    eye = torch.eye(N, device=DEV, dtype=F64)
    comb = lambda co, us: sum(a * u for a, u in zip(co, us))
    it = 0
    while idx.numel():
        live = t < dt
        h = torch.where(live, torch.where((dt - t) - h <= 1e-12 * dt, dt - t, h), torch.full_like(h, dt))
        f0, J = m.f(y, p, jac=True)
        LU = torch.linalg.lu_factor_ex(eye / (GAMMA * h)[:, None, None] - J)
        solve = lambda b: torch.linalg.lu_solve(LU.LU, LU.pivots, b[:, :, None])[:, :, 0]
        ih = 1.0 / h[:, None]
        u = [solve(f0)]
        u.append(solve(m.f(y + comb(A2, u), p) + ih * comb(C2, u)))
        f3 = m.f(y + comb(A3, u), p)
        u.append(solve(f3 + ih * comb(C3, u)))
        u.append(solve(f3 + ih * comb(C4, u)))
        yn = y + comb(MU, u)
        err = norm(comb(ER, u), atol + rtol * torch.maximum(y.abs(), yn.abs()))
        ok = (err <= 1.0) & live   # finished cells wait for the next compaction
        fac = torch.where(torch.isfinite(err), 0.9 * err.clamp(min=1e-300) ** -0.25, torch.full_like(err, 0.2))
        fac = fac.clamp(0.2, 5.0)
        fac = torch.where(~ok | rej, fac.clamp(max=1.0), fac)
        t = torch.where(ok, torch.where(t + h >= dt, torch.full_like(t, dt), t + h), t)
        y, rej, h = torch.where(ok[:, None], yn, y), ~ok, h * fac
        it += 1
        if it % 8 == 0:
            end = t >= dt
            done[idx[end]] = y[end]
            idx, y, p, h, t, rej = (v[~end] for v in (idx, y, p, h, t, rej))
    return done[:, 0], done[:, 1:].T.contiguous()


def _buckets(T, Y, tol=1e-4):
    """Each cell's reference (itself, if it is integrated) with one reference per state bucket."""
    n = T.numel()
    shift = 51 + math.frexp(tol)[1]
    key = torch.cat([(T.view(torch.int64) >> shift)[None], torch.floor(Y * (1.0 / tol)).to(torch.int64)])
    g = _gen(1)
    mul = torch.randint(-2**62, 2**62, (key.shape[0], 1), generator=g, device=DEV) | 1
    _, inv = torch.unique((key * mul).sum(0), return_inverse=True)
    i = torch.arange(n, device=DEV)
    ref = torch.full((n,), n, device=DEV).scatter_reduce(0, inv, i, "amin")[inv]
    near = ((Y - Y[:, ref]).abs().max(0).values < tol) & ((T - T[ref]).abs() < tol * T[ref])
    return torch.where(near, ref, i)


def _exact_integrate(nsp, T, p, Y, dt, rtol, atol, mapping):
    n = T.numel()
    ref = _buckets(T, Y) if mapping else torch.arange(n, device=DEV)
    own = torch.nonzero(ref == torch.arange(n, device=DEV))[:, 0]
    To, Yo = T.clone(), Y.clone()
    To[own], Yo[:, own] = _integrate64(_Mech(nsp), T[own], p[own], Y[:, own].contiguous(), dt, rtol, atol)
    return [To[ref] + (T - T[ref]), Yo[:, ref] + (Y - Y[:, ref])]


def _exact_net(c, seed):
    dims, params, X, Y = _net_io(c, seed)
    w = params.double().requires_grad_(c["op"] == "train")
    x, o = X.double(), 0
    for i, (a, b) in enumerate(zip(dims[:-1], dims[1:])):
        x = x @ w[o:o + a * b].view(a, b) + w[o + a * b:o + a * b + b]
        o += a * b + b
        if i < 3:
            x = torch.nn.functional.silu(x)
    if c["op"] == "forward":
        return [x]
    loss = (x - Y.double()).square().mean()
    return [torch.autograd.grad(loss, w)[0], loss.detach().reshape(1)]


def exact(case, seed):
    c = case
    if c["op"] in ("forward", "train"):
        return _exact_net(c, seed)
    if c["op"] == "rhs":
        m, out = _Mech(c["nsp"]), []
        T, p, Y = _states("uniform", c["nsp"], c["n"], 101325.0, seed)
        for i in range(0, c["n"], 16384):
            s = slice(i, i + 16384)
            out.append(m.f(torch.cat([T[s, None], Y[:, s].T], 1), p[s]))
        f = torch.cat(out)
        return [f[:, 0].contiguous(), f[:, 1:].T.contiguous()]
    if c["op"] == "batch":
        out = []
        for i, (nsp, n, dt) in enumerate(_meshes(c)):
            T, p, Y = _states("uniform", nsp, n, 101325.0, 10 * seed + i)
            out += _exact_integrate(nsp, T, p, Y, dt, 1e-6, 1e-10, 0) + [None]
        return out
    if c["nsp"] == 10:   # thousands of sequential steps: over 20 seconds
        return None
    T, p, Y = _states(c["states"], c["nsp"], c["n"], c["p"], seed)
    return _exact_integrate(c["nsp"], T, p, Y, c["dt"], c["rtol"], c["atol"], c["mapping"]) + [None]
