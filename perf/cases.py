"""The work that a planner's program has this framework do, as cases that can be timed.

A case is one call sequence of the public API (``paper_2410_13055_gb300.gx`` and
``.autograd``) on seeded synthetic inputs (``paper_2410_13055_gb300.synth``):

* ``step``       one implicit-gradient step: dispatch, adjoint, projected plan step; from a
                 cold start, or (``warm = "prev"``) from the checkpointed solution of a base
                 plan, as an interactive planner evaluates a candidate one gradient step away
* ``dispatch``   the dispatch of every scenario alone (evaluating a plan)
* ``objective``  the torch.autograd wrapper, forward and backward, with the envelope gradient
* ``predict``, ``train``  the learned warm start: a prediction, one training step

Iterations are capped at ``cap`` per loop, so that a pass is bounded on any draw of the
inputs; most loops stop at their residual tolerance before it.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2410_13055_gb300 import gx, synth
from paper_2410_13055_gb300.autograd import planner_objective

DEV = "cuda"

# What a case says when it does not say otherwise.
BASE = dict(call="step", nets="one", buses=100, lines=150, gens=300, bats=50, hours=24, scenarios=1, batch=0,
            warm="cold", kappa=50.0, rho=0.3, inner=2, adj_inner=0, tol=1e-3, cap=4000, ramps=0.0, hvdc=0, scaling=0.0)


def _case(name, **kw):
    c = dict(BASE, **kw)
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # the smallest call: the 5-bus, 24-hour network, one plan step from a cold start
        _case("tiny step", nets="tiny", buses=5, lines=7, gens=6, bats=2),
        # stochastic planning on the 100-bus network: 4 of 16 daily scenarios, continued from
        # the previous plan (the planner studies' loop, with their carbon weight)
        _case("sgd step 100x24", scenarios=16, batch=4, warm="prev", kappa=200.0),
        # the paper's network size (500 buses, 8 daily scenarios), continued from the previous plan
        _case("day step 500x24", buses=500, lines=1191, gens=1799, bats=576, scenarios=8, warm="prev", rho=0.2,
              adj_inner=1),
        # single hours on a large network, no coupling in time: a screening of operating points
        _case("hour dispatch 400x1", call="dispatch", buses=400, lines=600, gens=1200, bats=40, hours=1, scenarios=24),
        # a ragged horizon with ramp limits, HVDC links and capacity-dependent susceptances
        _case("extended step 100x45", hours=45, scenarios=3, ramps=1.0, hvdc=3, scaling=0.3, rho=0.2),
        # envelope gradient of a cost-only objective through torch.autograd, one week at a time
        _case("objective 100x168", call="objective", hours=168, scenarios=2, kappa=0.0),
        # the headline workload: 16 weeks of the 100-bus network, the planner's next step
        _case("medium step 100x168", hours=168, scenarios=16, warm="prev", rho=0.2, adj_inner=1),
        # the same weeks, the plan evaluated from nothing
        _case("medium dispatch 100x168", call="dispatch", hours=168, scenarios=16, rho=0.2),
        # 64 scenarios on their own networks of 50 to 500 buses over 24, 72 or 168 hours
        _case("uneven step x64", nets="uneven", buses=0, lines=0, gens=0, bats=0, hours=0, scenarios=64, warm="prev",
              rho=0.2, adj_inner=1),
        # the largest: a quarter of a year in weeks on the 2000-bus network
        _case("scale step 2000x168", buses=2000, lines=3000, gens=8000, bats=500, hours=168, scenarios=13, warm="prev",
              rho=0.2, adj_inner=1),
        # the learned warm start on the headline workload's 268,800 bus-hours
        _case("predict 100x168", call="predict", hours=168, scenarios=16),
        _case("train 100x168", call="train", hours=168, scenarios=16),
    ]


def _loguniform(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    call = rng.choice(["step", "step", "step", "step", "dispatch", "dispatch", "objective", "predict", "train"])
    buses = _loguniform(rng, 4, 600)
    hours = rng.choice([1, 24, 72, 168, rng.randint(2, 40), rng.randint(41, 256)])
    per_bus = rng.uniform(1.2, 2.5), rng.uniform(1.5, 4.0), rng.uniform(0.1, 1.1)
    lines = max(buses - 1, min(int(per_bus[0] * buses), buses * (buses - 1) // 2))
    gens, bats = max(1, int(per_bus[1] * buses)), max(1, int(per_bus[2] * buses))
    # at most 3 million device-hours, and at least one scenario
    scenarios = _loguniform(rng, 1, max(1, min(32, int(3e6 / ((buses + lines + gens + bats) * hours)))))
    c = _case(None, call=call, buses=buses, lines=lines, gens=gens, bats=bats, hours=hours, scenarios=scenarios,
              rho=rng.choice([0.2, 0.3]), inner=rng.choice([1, 2, 2, 2]), adj_inner=rng.choice([0, 1]), cap=2000)
    if call == "step":
        c["warm"] = rng.choice(["cold", "prev", "prev"])
        c["kappa"] = rng.choice([0.0, 50.0, 200.0])
        if rng.random() < 0.3:
            c.update(ramps=rng.choice([0.0, 0.5, 1.0]), hvdc=rng.randint(0, 3) if buses > 8 else 0,
                     scaling=rng.choice([0.0, 0.3]))
        if scenarios > 2 and rng.random() < 0.3:
            c["batch"] = rng.randint(1, scenarios - 1)
    elif call == "objective":
        c["kappa"] = 0.0
    return c


# ------------------------------------------------------------------------------ inputs
def _uneven(case):
    """Buses, lines, generators, batteries and hours of each network (any seed's inputs have these sizes)."""
    rng = np.random.default_rng(2)
    out = []
    for _ in range(case["scenarios"]):
        n, T = int(rng.integers(50, 501)), int(rng.choice([24, 72, 168]))
        out.append((n, int(round(1.5 * n)), 3 * n, max(1, int(round(0.3 * n))), T))
    return out


def _networks(case, seed):
    if case["nets"] == "tiny":
        return synth.tiny(seed)
    if case["nets"] == "uneven":
        parts = [synth.custom(n, l, g, b, T, seed=64 * seed + k, net_index=k) for k, (n, l, g, b, T) in enumerate(_uneven(case))]
        scens = [dict(s[0], weight=1.0 / len(parts)) for _, s in parts]
        return [n for n, _ in parts], scens
    net, scens = synth.custom(case["buses"], case["lines"], case["gens"], case["bats"], case["hours"],
                              S=case["scenarios"], seed=seed)
    if case["hvdc"]:
        net = synth.add_hvdc(net, case["hvdc"], seed=seed + 1)
    if case["ramps"]:
        net = synth.add_ramps(net, share=case["ramps"], seed=seed + 2)
    if case["scaling"]:
        net = synth.add_scaling(net, share=case["scaling"], seed=seed + 3)
    return [net], scens


def _base_plan(nets, seed):
    """A plan between the existing and the largest capacities."""
    rng = np.random.default_rng(seed)
    lo, hi = (np.concatenate([n[k] for n in nets]) for k in ("eta_min", "eta_max"))
    return lo + 0.1 * rng.random(lo.size) * (hi - lo)


def _batch(case):
    return list(range(1, 1 + case["batch"])) if case["batch"] else None


def _options(case):
    return dict(kappa=case["kappa"], rho=case["rho"], inner_iters=case["inner"], adj_inner_iters=case["adj_inner"],
                tol=case["tol"], adj_tol=case["tol"], max_iter=case["cap"], adj_max_iter=case["cap"], check_every=20,
                grad_envelope=int(case["call"] == "objective"))


def _alpha(gamma, grad, lo):
    """The planner's fixed step: 1 % of the median capacity at the largest entry."""
    return 1e-2 * float(lo.median()) / max(float((gamma + grad).abs().max()), 1e-30)


class State:
    pass


def prepare(case, seed):
    s = State()
    nets, scens = _networks(case, seed)
    s.case = case
    s.net = gx.Network(nets, scens, **_options(case))
    cat = lambda k: torch.tensor(np.concatenate([n[k] for n in nets]), dtype=torch.float32, device=DEV)
    s.lo, s.hi, s.gamma = cat("eta_min"), cat("eta_max"), cat("gamma")
    s.eta = torch.tensor(_base_plan(nets, seed), dtype=torch.float32, device=DEV)
    s.batch = _batch(case)
    s.grad = torch.zeros_like(s.eta)
    s.plan = torch.empty_like(s.eta)
    s.alpha = 1e-3
    if case["call"] in ("predict", "train"):
        s.gnn = gx.WarmStartGNN(s.net)
        s.gnn.set_params(_weights(seed))
        s.out = torch.empty(2 * s.gnn.M, dtype=torch.float32, device=DEV)
        s.target = torch.tensor(_targets(s.gnn.M, seed), device=DEV)
    elif case["call"] == "objective":
        s.eta.requires_grad_(True)
    elif case["call"] == "step" and case["warm"] == "prev":
        # the base plan's solution and the candidate one gradient step away
        s.net.solve(s.eta, batch=s.batch, warm="cold")
        s.net.grad(s.eta, out=s.grad, warm="cold")
        s.alpha = _alpha(s.gamma, s.grad, s.lo)
        s.net.plan_step(s.eta, s.grad, s.gamma, s.lo, s.hi, s.alpha)
        s.saved = s.net.state(False).clone(), s.net.state(True).clone()
    return s


def _weights(seed):
    """The learned start's parameters: input layer 16 x 64 (10 features used), three layers of
    128 x 64, head 64 x 2, each followed by its bias."""
    rng = np.random.default_rng(seed + 6)
    w_in = rng.normal(0.0, math.sqrt(0.2), (16, 64)) * (np.arange(16) < 10)[:, None]
    parts = [w_in, rng.normal(0.0, 0.05, 64)]
    for _ in range(3):
        parts += [rng.normal(0.0, math.sqrt(1 / 128), (128, 64)), rng.normal(0.0, 0.05, 64)]
    parts += [rng.normal(0.0, 0.125, (64, 2)), rng.normal(0.0, 0.05, 2)]
    return np.concatenate([p.reshape(-1) for p in parts]).astype(np.float32)


def _targets(M, seed):
    rng = np.random.default_rng(seed + 5)
    return np.concatenate([np.clip(rng.normal(40.0, 20.0, M), 0.0, 200.0), rng.normal(0.0, 0.1, M)]).astype(np.float32)


def run(s):
    call, warm = s.case["call"], s.case["warm"]
    if call == "predict":
        return {"start": s.gnn.predict(s.eta, out=s.out)}
    if call == "train":
        s.gnn.train_step(s.eta, s.target, lr=1e-3, w_theta=10.0)
        return {"gradients": s.gnn.params(1), "weights": s.gnn.params(0)}
    if call == "objective":
        J = planner_objective(s.eta, s.net)
        (g,) = torch.autograd.grad(J, s.eta)
        return {"objective": J.detach(), "gradient": g, "price": s.net.array("price"), "output": s.net.array("p")}
    if warm == "prev":
        s.net.state(False).copy_(s.saved[0])
        s.net.state(True).copy_(s.saved[1])
    s.net.solve(s.eta, batch=s.batch, warm=warm)
    if call == "dispatch":
        return {"price": s.net.array("price"), "output": s.net.array("p")}
    s.net.grad(s.eta, out=s.grad, warm=warm)
    s.plan.copy_(s.eta)
    s.net.plan_step(s.plan, s.grad, s.gamma, s.lo, s.hi, s.alpha)
    return {"plan": s.plan, "gradient": s.grad, "price": s.net.array("price"), "output": s.net.array("p")}


# ------------------------------------------------------------------------------ work
def _sizes(case):
    """Sums over the scenarios of a pass: bus-, generator-, line- and battery-hours; plan length."""
    if case["nets"] == "uneven":
        rows = _uneven(case)
        tot = lambda k: sum(r[k] * r[4] for r in rows)
        return tot(0), tot(2), tot(1), tot(3), sum(r[1] + r[2] + r[3] for r in rows)
    S = case["batch"] or case["scenarios"]
    h = S * case["hours"]
    return (h * case["buses"], h * case["gens"], h * (case["lines"] + case["hvdc"]), h * case["bats"],
            case["gens"] + case["lines"] + case["hvdc"] + case["bats"])


def work(case):
    """One pass's inputs read once and outputs written once, and the arithmetic of its fewest
    iterations (a solve runs at least one residual check of 20 iterations)."""
    bus, gen, line, bat, K = _sizes(case)
    if case["call"] in ("predict", "train"):
        layer = 2 * 64 * 128
        fwd = bus * (2 * 10 * 64 + 3 * layer + 2 * 64 * 2 + 3 * 64 * 2 * line / bus)
        n_par = 16 * 64 + 64 + 3 * (128 * 64 + 64) + 130
        if case["call"] == "predict":
            return {"bytes": 4 * (bus + gen + K + n_par + 2 * bus), "flops": fwd}
        return {"bytes": 4 * (bus + gen + K + 2 * bus + 6 * n_par), "flops": 3 * fwd}
    # one iteration: clip and sums of a generator or load 14, a line 40, a battery hour 60 a sweep pair, a bus 20
    it = 14 * (gen + bus) + 40 * line + 60 * case["inner"] * bat + 20 * bus
    loops = 2 if case["call"] == "step" else 1
    # inputs: load, capacity factor, the plan; outputs: dispatch and prices, the gradient
    nbytes = 4 * (bus + gen + K) + 4 * (gen + bus + line + 3 * bat + bus) + 4 * K
    if case["warm"] == "prev":  # the previous plan's forward and adjoint state, read and written
        nbytes += 2 * 2 * 4 * (gen + 4 * bus + 4 * line + 7 * bat)
    return {"bytes": nbytes, "flops": 20 * loops * it}


# ------------------------------------------------------------------------------ 64 bits
class _Proximal:
    """The message passing in plain torch FP64, over [scenario, device, hour]."""

    def __init__(self, case, net, scens):
        T = lambda a: torch.tensor(np.asarray(a, np.float64), dtype=torch.float64, device=DEV)
        I = lambda a: torch.tensor(np.asarray(a, np.int64), device=DEV)
        self.c = case
        self.load, self.cf = T(np.stack([s["load"] for s in scens])), T(np.stack([s["cf"] for s in scens]))
        self.wt = np.array([s["weight"] for s in scens])
        self.gb, self.gc, self.ge = I(net["gen_bus"]), T(net["gen_cost"])[None, :, None], T(net["gen_emis"])[None, :, None]
        self.fr, self.to = I(net["line_from"]), I(net["line_to"])
        self.bb, self.dur = I(net["bat_bus"]), T(net["bat_dur"])[None, :, None]
        self.N, self.G, self.L, self.B = net["n_bus"], self.gb.numel(), self.fr.numel(), self.bb.numel()
        self.S, _, self.T = self.load.shape
        self.dc = torch.zeros(self.L, dtype=torch.bool, device=DEV)
        if "line_dc" in net:
            self.dc = I(net["line_dc"]) != 0
        beta = T(net["line_beta"])
        self.beta = torch.where(self.dc, torch.ones_like(beta), beta)[None, :, None]
        self.dth = torch.where(self.dc, torch.full_like(beta, 3e38), T(net["line_dtheta"]))[None, :, None]
        b2 = beta[~self.dc] ** 2
        w = torch.where(self.dc, torch.zeros_like(beta), torch.full_like(beta, float(b2.mean()) if b2.numel() else 1.0))
        self.w = w[None, :, None]
        one = lambda ix: torch.bincount(ix, minlength=self.N).double()
        self.cnt = (1 + one(self.gb) + one(self.bb) + one(self.fr) + one(self.to))[None, :, None]
        ws = torch.zeros(self.N, dtype=torch.float64, device=DEV).index_add_(0, self.fr, w).index_add_(0, self.to, w)
        self.iw = torch.where(ws > 0, 1 / ws.clamp_min(1e-300), torch.zeros_like(ws))[None, :, None]
        d = (w / self.beta[0, :, 0]) ** 2
        self.dres = torch.zeros(self.N, dtype=torch.float64, device=DEV).index_add_(0, self.fr, d).index_add_(0, self.to, d)
        self.norm = self.load.square().sum((1, 2)).sqrt().clamp_min(1e-30)
        self.a, self.k = float(net["bat_eff_c"][0]), 1.0 / float(net["bat_eff_d"][0])
        self.tol_act = 1e-5 * max(1.0, float(np.abs(net["gen_cost"]).max()))
        self.eps, self.voll = 1e-3, 1000.0

    def plan(self, eta):
        G, L = self.G, self.L
        e = eta.clamp_min(0)
        self.cap = self.cf * e[:G][None, :, None]
        self.capl = e[G:G + L][None, :, None] / self.beta
        self.P = e[G + L:][None, :, None]

    def zero(self):
        z = lambda n: torch.zeros(self.S, n, self.T, dtype=torch.float64, device=DEV)
        st = {k: z(self.L) for k in ("dl", "sg", "qf", "qt")}
        st.update({k: z(self.B) for k in ("xb", "zc", "zd", "zs", "yc", "yd", "ys")})
        st.update({k: z(self.N) for k in ("xl", "u", "pb", "th")})
        st["xg"] = z(self.G)
        return st

    def to_bus(self, n, parts):
        out = torch.zeros(n, self.N, self.T, dtype=torch.float64, device=DEV)
        for ix, v in parts:
            out.index_add_(1, ix, v)
        return out

    def start(self, st):
        """The bus averages of the given device state."""
        n = st["xg"].shape[0]
        f = self.beta * st["dl"]
        s = st["xl"] + self.to_bus(n, [(self.gb, st["xg"]), (self.bb, st["xb"]), (self.fr, -f), (self.to, f)])
        st["pb"] = s / self.cnt
        st["th"] = self.to_bus(n, [(self.fr, self.w * st["qf"]), (self.to, self.w * st["qt"])]) * self.iw

    def pivots(self, rho, ri):
        A = self.eps + ri + rho
        det = A * A - rho * rho
        gc, gd = (A * self.a - rho * self.k) / det, (rho * self.a - A * self.k) / det
        g = self.a * gc - self.k * gd
        T = self.T
        M = torch.diag(torch.full((T,), 2 + g * ri, dtype=torch.float64))
        M[0, 0] = 1 + g * ri
        i = torch.arange(T - 1)
        M[i, i + 1] = M[i + 1, i] = -1
        return A, det, gc, gd, torch.linalg.inv(M).to(DEV)

    def line_target(self, st, rho, rth, lin):
        fr, to, b, d = self.fr, self.to, self.beta, st["dl"]
        zf, zt = st["th"][:, fr], st["th"][:, to]
        vf, vt = st["qf"] - zf, st["qt"] - zt
        wf, wt = zf - vf, zt - vt
        tf = -b * d - st["pb"][:, fr] - st["u"][:, fr]
        tt = b * d - st["pb"][:, to] - st["u"][:, to]
        den = 2 * rho * b * b + 0.5 * rth * self.w + self.dc[None, :, None] * self.eps
        dun = (rho * b * (tt - tf) + 0.5 * rth * self.w * (wf - wt) + lin) / den
        return dun, den, zf, zt, vf, vt, wf, wt, tf, tt

    def loop(self, st, adj, act=None, batch=None):
        """Iterate every scenario of `batch` to its tolerance; `st` is updated."""
        c, eps = self.c, self.eps
        rho = 0.002 if adj else c["rho"]
        ri, rth, inner = rho, rho * 0.1, (c["adj_inner"] or c["inner"]) if adj else c["inner"]
        A, det, gc, gd, Minv = self.pivots(rho, ri)
        idx = torch.tensor(list(range(self.S)) if batch is None else batch, device=DEV)
        cur = {k: v[idx] for k, v in st.items()}
        sub = lambda v: v[idx] if v.shape[0] == self.S else v
        it = 0
        while idx.numel() and it < c["cap"]:
            load, cap = sub(self.load), sub(self.cap)
            if adj:
                m = {k: v[idx] for k, v in act.items()}
                lin = self.dc[None, :, None] * eps * m["fl"]
                fixg, fixl = m["g"] != 0, m["l"] != 0
                box = [m[k] != 0 for k in ("bc", "bd", "bs")]
                qc, qd = -eps * m["zc"], -eps * m["zd"]
                scale = (((m["ag"] / (rho + eps)) ** 2 * ~fixg).sum((1, 2)) + ((m["al"] / (rho + eps)) ** 2 * ~fixl).sum((1, 2))).sqrt().clamp_min(1e-30)
            else:
                lin = qc = qd = 0.0
                scale = self.norm[idx]
            n = idx.numel()
            for j in range(min(20, c["cap"] - it)):
                s = cur
                pb, u, th = s["pb"], s["u"], s["th"]
                dun, _, zf, zt, vf, vt, wf, wt, _, _ = self.line_target(s, rho, rth, lin)
                ef, et = 0.5 * (s["sg"] + s["dl"]) - zf, 0.5 * (s["sg"] - s["dl"]) - zt
                if adj:
                    dn = torch.where(m["ln"] != 0, 0.0, dun)
                else:
                    lc = torch.minimum(self.capl, self.dth)
                    dn = torch.minimum(torch.maximum(dun, -lc), lc)
                gn = wf + wt
                v = s["xb"] - pb[:, self.bb] - u[:, self.bb]
                z, y = [s["zc"], s["zd"], s["zs"]], [s["yc"], s["yd"], s["ys"]]
                for _ in range(inner):
                    r = [zz - yy / ri for zz, yy in zip(z, y)]
                    b1, b2 = ri * r[0] - rho * v - qc, ri * r[1] + rho * v - qd
                    c0, d0 = (A * b1 + rho * b2) / det, (rho * b1 + A * b2) / det
                    prev = torch.nn.functional.pad(r[2], (1, 0))[..., :-1]
                    mu = (ri * (r[2] - prev - (self.a * c0 - self.k * d0))) @ Minv
                    x = [c0 + mu * gc, d0 + mu * gd, r[2] - (mu - torch.nn.functional.pad(mu, (0, 1))[..., 1:]) / ri]
                    t = [xx + yy / ri for xx, yy in zip(x, y)]
                    if adj:
                        z = [torch.where(f, 0.0, tt) for f, tt in zip(box, t)]
                    else:
                        hi = [self.P, self.P, self.dur * self.P]
                        z = [torch.minimum(tt.clamp_min(0), h) for tt, h in zip(t, hi)]
                    y = [yy + ri * (xx - zz) for yy, xx, zz in zip(y, x, z)]
                xb = x[1] - x[0]
                vg = s["xg"] - pb[:, self.gb] - u[:, self.gb]
                vl = s["xl"] - pb - u
                if adj:
                    xg = torch.where(fixg, 0.0, (rho * vg + m["ag"]) / (rho + eps))
                    xl = torch.where(fixl, 0.0, (rho * vl + m["al"]) / (rho + eps))
                else:
                    xg = torch.minimum(((rho * vg - self.gc) / (rho + eps)).clamp_min(0), cap)
                    xl = torch.minimum(((rho * (vl + load) - self.voll) / (rho + eps)).clamp_min(0), load) - load
                new = dict(dl=dn, sg=gn, qf=0.5 * (gn + dn) + vf, qt=0.5 * (gn - dn) + vt, xb=xb, zc=z[0], zd=z[1], zs=z[2],
                           yc=y[0], yd=y[1], ys=y[2], xg=xg, xl=xl, u=u)
                self.start(new)
                new["u"] = u + new["pb"]
                old, cur = s, new
            it += min(20, c["cap"] - it)
            sq = lambda v: v.square().sum((1, 2))
            th2 = ((self.beta ** 2) * (~self.dc)[None, :, None] * (ef * ef + et * et)).sum((1, 2))
            dx = sq(cur["xg"] - old["xg"]) + sq(cur["xl"] - old["xl"]) + sq(cur["xb"] - old["xb"]) + 2 * sq(self.beta * (cur["dl"] - old["dl"]))
            dz = (dx - (self.cnt * (cur["pb"] - old["pb"]) ** 2).sum((1, 2))).clamp_min(0)
            a3 = (self.dres[None, :, None] * (cur["th"] - old["th"]) ** 2).sum((1, 2))
            rp = ((self.cnt * cur["pb"] ** 2).sum((1, 2)) + th2).sqrt() / scale
            rd = (rho * rho * dz + rth * rth * a3).sqrt() / (self.cnt * (rho * cur["u"]) ** 2).sum((1, 2)).sqrt().clamp_min(1e-30)
            done = (rp <= c["tol"]) & (rd <= c["tol"])
            if it >= c["cap"]:
                done = torch.ones_like(done)
            if bool(done.any()):
                for k in st:
                    st[k][idx[done]] = cur[k][done]
                idx = idx[~done]
                cur = {k: v[~done] for k, v in cur.items()}

    def active(self, st):
        """The active set of the solved dispatch and the adjoint's linear terms."""
        c, eps, rho, tol = self.c, self.eps, self.c["rho"], self.tol_act
        pb, u = st["pb"], st["u"]
        code = lambda up, lo: up.double() - lo.double()
        pun = (rho * (st["xg"] - pb[:, self.gb] - u[:, self.gb]) - self.gc) / (rho + eps)
        g = code((rho + eps) * (pun - self.cap) > tol, -(rho + eps) * pun > tol)
        sun = (rho * (st["xl"] - pb - u + self.load) - self.voll) / (rho + eps)
        l = code((rho + eps) * (sun - self.load) > tol, -(rho + eps) * sun > tol)
        dun, den = self.line_target(st, rho, rho * 0.1, 0.0)[:2]
        over = den * (dun.abs() - torch.minimum(self.capl, self.dth)) / self.beta > tol
        ln = torch.sign(dun) * over.double() * torch.where(self.capl <= self.dth, 1.0, 2.0)
        bat = {k: code(st[y] > tol, st[y] < -tol) for k, y in (("bc", "yc"), ("bd", "yd"), ("bs", "ys"))}
        return dict(bat, g=g, l=l, ln=ln, ag=self.gc + eps * st["xg"] + c["kappa"] * self.ge,
                    al=self.voll + eps * (st["xl"] + self.load), fl=st["dl"], zc=st["zc"], zd=st["zd"])

    def adjoint_start(self, st):
        ratio = self.c["rho"] / 0.002
        a = self.zero()
        a["u"] = -ratio * st["u"]
        a["qf"] = -ratio * (st["qf"] - st["th"][:, self.fr])
        a["qt"] = -ratio * (st["qt"] - st["th"][:, self.to])
        for y in ("yc", "yd", "ys"):
            a[y] = -st[y]
        return a

    def gradient(self, act, st, ad, batch):
        """sum_s w'_s dh_s/d eta; `ad` is None for the envelope gradient."""
        c, eps = self.c, self.eps
        env = ad is None
        s, rho = (st, c["rho"]) if env else (ad, 0.002)
        v = s["xg"] - s["pb"][:, self.gb] - s["u"][:, self.gb]
        xi = -(rho * (v - s["xg"]) - self.gc - eps * s["xg"]) if env else act["ag"] + rho * v
        gg = ((act["g"] > 0) * xi * self.cf).sum(2)
        _, _, _, _, _, _, wf, wt, tf, tt = self.line_target(s, rho, rho * 0.1, 0.0)
        d = s["dl"] if env else 0.0 * s["dl"]
        F = rho * self.beta * (2 * self.beta * d + tf - tt) + 0.5 * rho * 0.1 * self.w * (d - (wf - wt))
        F = F + self.dc[None, :, None] * eps * (d if env else -act["fl"])
        sign = torch.where(act["ln"].abs() == 1, act["ln"], torch.zeros_like(act["ln"])) * (1.0 if env else -1.0)
        gl = (sign * F / self.beta).sum(2)
        pm = -1.0 if env else 1.0
        gb = pm * sum(((act[k] > 0) * s[y] * f).sum(2) for k, y, f in (("bc", "yc", 1.0), ("bd", "yd", 1.0), ("bs", "ys", self.dur)))
        wt_ = self.wt if batch is None else np.array([self.wt[i] if i in batch else 0.0 for i in range(self.S)])
        wt_ = torch.tensor(wt_ * self.wt.sum() / wt_.sum(), device=DEV)
        return (wt_[:, None] * torch.cat([gg, gl, gb], 1)).sum(0)

    def value(self, st):
        p, sh, f = st["xg"], st["xl"] + self.load, st["dl"] * self.dc[None, :, None]
        cost = (self.gc * p + 0.5 * self.eps * p * p).sum((1, 2)) + (self.voll * sh + 0.5 * self.eps * sh * sh).sum((1, 2))
        cost = cost + 0.5 * self.eps * ((st["zc"] ** 2).sum((1, 2)) + (st["zd"] ** 2).sum((1, 2)) + (f * f).sum((1, 2)))
        h = cost + self.c["kappa"] * (self.ge * p).sum((1, 2))
        return (torch.tensor(self.wt, device=DEV) * h).sum()


def _rows(v):
    """[S, device, T] as the workspace holds it: rows padded to a multiple of 4 hours."""
    return torch.nn.functional.pad(v, (0, -v.shape[2] % 4)).reshape(-1)


def _exact_network(case, seed):
    """The learned start's graph network: its prediction, or a step's gradients (the weights
    after the step follow the sign of gradients near zero, and have no value here)."""
    nets, scens = _networks(case, seed)
    net = nets[0]
    par = torch.tensor(_weights(seed).astype(np.float64), device=DEV)
    N, G, T, S, L = net["n_bus"], net["gen_bus"].size, case["hours"], len(scens), net["line_from"].size
    D = lambda a: torch.tensor(np.asarray(a, np.float64), dtype=torch.float64, device=DEV)
    eta = D(_base_plan(nets, seed)).float().double()
    load, cf = D(np.stack([s["load"] for s in scens])), D(np.stack([s["cf"] for s in scens]))
    gb, fr, to, bb = (torch.tensor(np.asarray(net[k], np.int64), device=DEV) for k in ("gen_bus", "line_from", "line_to", "bat_bus"))
    bus = lambda ix, v: torch.zeros(S, N, T, dtype=torch.float64, device=DEV).index_add_(1, ix, v)
    cost = D(net["gen_cost"])[None, :, None]
    cap = cf * eta[:G][None, :, None]
    row = lambda ix, v: bus(ix, v[None, :, None].expand(S, -1, T))
    dear, free = bus(gb, cap * (cost != 0)), bus(gb, cap * (cost == 0))
    hour = (torch.arange(T, device=DEV).double() % 24).expand(S, N, T) * (2 * math.pi / 24)
    costw = torch.where(dear > 0, bus(gb, cap * cost) / dear.clamp_min(1e-300), torch.zeros_like(dear))
    lin = row(fr, eta[G:G + L]) + row(to, eta[G:G + L])
    f = [load, bus(gb, cap), costw, free, row(bb, eta[G + L:]), lin]
    x = torch.stack([0.01 * v for v in f] + [hour.sin(), hour.cos(), 0.01 * (load - free), torch.ones_like(load)], -1)
    Tp = T + -T % 4
    x = torch.nn.functional.pad(x, (0, 6, 0, Tp - T))  # 16 input columns, rows padded in hours
    deg = (torch.bincount(fr, minlength=N) + torch.bincount(to, minlength=N)).double().clamp_min(1)[None, :, None, None]
    mean = lambda h: torch.zeros_like(h).index_add_(1, fr, h[:, to]).index_add_(1, to, h[:, fr]) / deg
    par.requires_grad_(case["call"] == "train")
    at = 0

    def take(*shape):
        nonlocal at
        n = math.prod(shape)
        at += n
        return par[at - n:at].view(*shape)

    h = torch.relu(x @ take(16, 64) + take(64))
    for _ in range(3):
        W, b = take(128, 64), take(64)
        h = h + torch.relu(torch.cat([h, mean(h)], -1) @ W + b)
    y = h @ take(64, 2) + take(2)
    price, angle = 100 * y[..., 0].reshape(-1), y[..., 1].reshape(-1)
    if case["call"] == "predict":
        return {"start": torch.cat([price, angle])}
    tgt = D(_targets(price.numel(), seed))
    on = (torch.arange(Tp, device=DEV) < T).expand(S, N, Tp).reshape(-1).double()
    loss = (on * ((price - tgt[:price.numel()]) / 100) ** 2 + 10.0 * on * (angle - tgt[price.numel():]) ** 2).sum() / on.sum()
    (g,) = torch.autograd.grad(loss, par)
    return {"gradients": g, "weights": None}


def exact(case, seed):
    # None: ramps and scaling susceptances follow another iteration, 64 networks or 2000
    # buses take minutes in plain torch
    if case["nets"] == "uneven" or case["ramps"] or case["scaling"] or case["buses"] > 1000:
        return None
    if case["call"] in ("predict", "train"):
        return _exact_network(case, seed)
    nets, scens = _networks(case, seed)
    E = _Proximal(case, nets[0], scens)
    lo, hi, gamma = (torch.tensor(nets[0][k], dtype=torch.float64, device=DEV) for k in ("eta_min", "eta_max", "gamma"))
    eta = torch.tensor(_base_plan(nets, seed), dtype=torch.float64, device=DEV)
    batch, st, ad, alpha = _batch(case), E.zero(), None, 1e-3
    st["xl"] = -E.load

    def solve():
        E.plan(eta)
        E.loop(st, False, batch=batch)

    def grad(cold):
        nonlocal ad
        act = E.active(st)
        if cold:
            ad = E.adjoint_start(st)
        E.start(ad)
        E.loop(ad, True, act, batch)
        return E.gradient(act, st, ad, batch)

    step = lambda e, g: torch.minimum(torch.maximum(e - alpha * (gamma + g), lo), hi)
    E.plan(eta)
    E.start(st)
    solve()
    rows = {"price": _rows(-case["rho"] * st["u"]), "output": _rows(st["xg"])}
    if case["call"] == "dispatch":
        return rows
    if case["call"] == "objective":
        return dict(rows, objective=E.value(st), gradient=E.gradient(E.active(st), st, None, batch))
    g = grad(True)
    if case["warm"] == "prev":
        alpha = _alpha(gamma, g, lo)
        eta = step(eta, g)
        solve()
        g = grad(False)
    out = {"plan": step(eta, g), "gradient": g}
    if batch is None:
        return dict(out, price=_rows(-case["rho"] * st["u"]), output=_rows(st["xg"]))
    return dict(out, price=None, output=None)  # scenarios outside the batch hold what was there
