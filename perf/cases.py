"""What is measured: the work that a user of the time step has it do, through its public entry points.

A case is one of three kinds of pass:
  * ``run``: advance the tubes of one handle by some steps and read the macroscopic fields and the state. Handles
    of small tubes start each pass from the same checkpoint (rlb_set_state), so that a pass is a whole run; the
    large ones go on from where the last pass left them, as a long simulation does;
  * ``fit``: one gradient of the inverse problem through the torch.autograd wrapper: the fields after a run, the
    loss of its energy and particle density against targets, the gradient in log(tau) and in the initial P, n, v;
  * ``sweepback``: the same through the adjoint entry points themselves on a handle that is kept.

States are given by a start: ``sod`` (Riemann data, the membrane just removed), ``shock`` (a tube part-way through
its run: a moving rarefaction, plateau and shock, most of the gas in motion), ``waves`` (smooth periodic waves) and
``bumps`` (Gaussian pressure bumps at rest, the inverse problem's).

``exact`` evaluates the method in plain torch in 64 bits, from the method's formulas, and shares no code with the
library; the gradients are torch's own, through that evaluation.
"""
from __future__ import annotations

import math

import numpy as np
import torch
from torch.utils.checkpoint import checkpoint

import paper_1608_03004_gb300 as rlb
from paper_1608_03004_gb300.adjoint import run_fields

DEV = "cuda"
STORE = {"f64": torch.float64, "f32": torch.float32, "bf16": torch.bfloat16}
TAUS = (1e-4, 1e-3, 1e-2, 1e-1, 1.0, 10.0, math.inf)  # the relaxation-time sweep
SWEEP_QXI = (8, 32, 128, 200)


def listed():
    one = {"kind": "run", "storage": "f64", "tubes": "one", "Qp": 3, "Np": 2, "Nv": 5, "bc": "open", "graph": 0}
    return [
        # the paper's small Sod tube, one step and its fields: a program that looks at every step; launches and
        # latency are all there is
        dict(one, name="sod_step", Nx=400, Qxi=8, tau=1e-3, start="shock", steps=1, restart=True),
        # the same tube from the membrane to t = 0.3 in one call
        dict(one, name="sod_run", Nx=400, Qxi=8, tau=1e-3, start="sod", steps=320, restart=True),
        # a tube of the inverse problem's size with all its gas in motion, forward only, replayed as CUDA graphs
        dict(one, name="waves_graph", Nx=2048, Qxi=32, tau=5e-2, bc="periodic", start="waves", steps=50, restart=True,
             graph=10),
        # the relaxation-time sweep: 28 tubes, tau = 1e-4 .. inf, Qxi = 8 .. 200, in one handle
        dict(one, name="sweep_f64", tubes="sweep", Nx=4096, Qxi=0, tau=0.0, start="shock", steps=3, restart=True),
        # uneven tubes with odd sizes, odd orders, ballistic and periodic ones among them
        dict(one, name="ragged_f64", tubes="ragged", Nx=3000, Qxi=0, tau=0.0, start="shock", steps=6, restart=True,
             count=13),
        # the largest FP64 tube: 2^20 cells x 384 velocities
        dict(one, name="stress_f64", Nx=1 << 20, Qxi=128, tau=1e-2, start="shock", steps=2, restart=False),
        # the same tube with FP32 and with BF16 storage
        dict(one, name="stress_f32", storage="f32", Nx=1 << 20, Qxi=128, tau=1e-2, start="shock", steps=12,
             restart=False),
        dict(one, name="stress_bf16", storage="bf16", Nx=1 << 20, Qxi=128, tau=1e-2, start="shock", steps=12,
             restart=False),
        # a batch of uneven shock tubes in FP32, warps taking tiles from a counter, replayed as CUDA graphs
        dict(one, name="batch_f32", storage="f32", tubes="batch", Nx=8192, Qxi=0, tau=0.0, start="shock", steps=6,
             restart=False, count=128, graph=3),
        # a checkpoint read back into an FP32 tube of odd size and odd order, a few steps, the next checkpoint
        dict(one, name="restart_f32", storage="f32", Nx=50021, Qxi=33, tau=3e-2, start="shock", steps=4,
             restart=True),
        # one gradient of the inverse problem through autograd, checkpoints along the run
        {"name": "fit", "kind": "fit", "tubes": 1, "Nx": 2048, "Qxi": 32, "tau": 8e-2, "start": "bumps", "steps": 100,
         "every": 25},
        # reverse sweeps over a batch of tubes on a kept handle, every stage input kept
        {"name": "sweepback", "kind": "sweepback", "tubes": 16, "Nx": 1537, "Qxi": 24, "tau": 5e-2, "start": "waves",
         "steps": 8, "every": 8},
    ]


def draw(rng):
    def logint(a, b):
        return int(round(math.exp(rng.uniform(math.log(a), math.log(b)))))

    tau = 10.0 ** rng.uniform(-4, 1)
    if rng.random() < 0.25:
        tubes, Nx, Qxi = rng.choice([1, 1, 3, 8]), logint(48, 4000), logint(4, 64)
        steps = max(2, min(100, int(1.6e7 / (tubes * Nx * 3 * Qxi))))
        return {"kind": rng.choice(["fit", "sweepback"]), "tubes": tubes, "Nx": Nx, "Qxi": Qxi, "tau": max(tau, 1e-3),
                "start": rng.choice(["bumps", "waves"]), "steps": steps, "every": rng.randint(2, steps)}
    storage = rng.choice(["f64", "f64", "f32", "f32", "bf16"])
    c = {"kind": "run", "storage": storage, "tubes": rng.choice(["one", "one", "ragged"]), "bc": "open", "graph": 0,
         "Qp": 3, "Np": 2, "Nv": 5, "Qxi": logint(4, 200), "tau": tau if rng.random() < 0.9 else math.inf,
         "start": rng.choice(["sod", "shock", "waves"]), "restart": True}
    most = 1.5e8 if storage == "f64" else 3e8
    if c["tubes"] == "ragged":
        c.update(count=rng.randint(2, 24), Nx=logint(100, 20000))
        nodes = c["count"] * c["Nx"] * 3 * 40
    else:
        if c["start"] == "waves":
            c["bc"] = "periodic"
        if rng.random() < 0.15:
            c.update(Qp=4, Np=3, Nv=8, Qxi=max(6, c["Qxi"]))
        c["Nx"] = logint(64, min(1 << 18, int(most / (c["Qp"] * c["Qxi"]))))
        nodes = c["Nx"] * c["Qp"] * c["Qxi"]
    if rng.random() < 0.3:
        c["graph"] = rng.randint(1, 4)
    c["steps"] = max(1, min(64, int(3 * most / nodes), logint(1, 64)))
    return c


# ---------------------------------------------------------------------------------------------------------------
# Inputs
# ---------------------------------------------------------------------------------------------------------------

def _dt(dx, tau):
    return min(0.5 * dx, 0.45 * tau)  # CFL 0.5 and the stiffness rule of strong shocks


def _tubes(case):
    """Tube descriptions of a case (plain dicts)."""
    base = {k: case.get(k, d) for k, d in (("Qp", 3), ("Np", 2), ("Nv", 5), ("bc", "open"))}
    if case["kind"] != "run":
        bc = "periodic" if case["start"] == "waves" else "open"
        many = case["tubes"]
        # a batch of tubes of uneven length around the case's
        out = [dict(base, Nx=case["Nx"] + (37 * k) % 101 if many > 1 else case["Nx"], Qxi=case["Qxi"], tau=case["tau"],
                    bc=bc) for k in range(many)]
    elif case["tubes"] == "sweep":
        out = [dict(base, Nx=case["Nx"], Qxi=q, tau=t) for t in TAUS for q in SWEEP_QXI]
    elif case["tubes"] == "ragged":
        rng = np.random.default_rng(case["Nx"] + case["count"])  # sizes belong to the case, not to the seed
        out = []
        for k in range(case["count"]):
            t = dict(base, Nx=max(16, int(case["Nx"] * rng.uniform(0.2, 1.8))), Qxi=int(rng.integers(4, 72)),
                     tau=float(10.0 ** rng.uniform(-3, 1)), bc="periodic" if k % 4 == 3 else "open")
            if k % 5 == 2:
                t["tau"] = math.inf
            if k % 6 == 4:
                t.update(Qp=4, Np=3, Nv=8, Qxi=max(6, t["Qxi"]))
            out.append(t)
    elif case["tubes"] == "batch":
        rng = np.random.default_rng(160803004)
        out = [dict(base, Nx=int(rng.integers(case["Nx"] // 8, 2 * case["Nx"])), Qxi=int(rng.choice([8, 16, 32, 64])),
                    tau=float(10.0 ** rng.uniform(-4, 1))) for _ in range(case["count"])]
    else:
        out = [dict(base, Nx=case["Nx"], Qxi=case["Qxi"], tau=case["tau"])]
    for t in out:
        t["dx"] = 1.0 / t["Nx"]
        t["dt"] = _dt(t["dx"], t["tau"])
    return out


def _start(case, t, rng):
    """(P, n, v) of one tube on the GPU, from the seed's generator."""
    Nx = t["Nx"]
    x = -0.5 + (torch.arange(Nx, dtype=torch.float64, device=DEV) + 0.5) * t["dx"]
    u = lambda a, b: float(rng.uniform(a, b))  # noqa: E731
    start = "waves" if t["bc"] == "periodic" else case["start"]
    if start == "sod":
        PL = u(0.8, 1.2)
        PR = PL * u(0.1, 0.3)
        right = x > 0
        P = torch.where(right, PR, PL).to(torch.float64)
        n = torch.where(right, PR / 0.8, PL).to(torch.float64)
        return P, n, torch.zeros_like(x)
    if start == "shock":
        PL = u(0.8, 1.2)
        PR = PL * u(0.1, 0.3)
        Pm, vm = math.sqrt(PL * PR), u(0.2, 0.45)
        head, tail, contact, shock = u(-0.4, -0.3), u(-0.15, -0.05), u(0.05, 0.15), u(0.25, 0.35)
        fan = torch.clamp((x - head) / (tail - head), 0.0, 1.0)  # rarefaction fan

        def edge(at):  # a front some cells wide
            return 0.5 * (1.0 + torch.tanh((x - at) / (4.0 * t["dx"])))

        P = PL + (Pm - PL) * fan + (PR - Pm) * edge(shock)
        v = vm * fan * (1.0 - edge(shock))
        T = 1.0 - 0.15 * fan + 0.2 * edge(contact) - 0.25 * edge(shock)
        return P, P / T, v
    if start == "bumps":
        P = torch.ones_like(x)
        for _ in range(5):
            P = P + 0.05 * u(0.5, 1.0) * torch.exp(-0.5 * ((x - u(-0.3, 0.3)) / u(0.02, 0.08)) ** 2)
        return P, P.clone(), torch.zeros_like(x)

    def wave(amp):
        f = sum(u(-1, 1) / k * torch.sin(2 * math.pi * k * x + u(0, 6)) for k in (1, 2, 3))
        return amp * f / torch.clamp(f.abs().max(), min=1e-9)

    return 1.0 + wave(0.4), 1.0 + wave(0.3), wave(0.45)


def _inputs(case, seed):
    rng = np.random.default_rng([int(seed) & 0x7FFFFFFF, 1608])
    tubes = _tubes(case)
    parts = [_start(case, t, rng) for t in tubes]
    P, n, v = (torch.cat([p[k] for p in parts]) for k in range(3))
    return tubes, P, n, v


def _handle_tubes(tubes, storage="f64"):
    return [rlb.Tube(t["Qp"], t["Qxi"], t["Np"], t["Nv"], t["Nx"], t["dx"], t["dt"], t["tau"],
                     rlb.BC_PERIODIC if t["bc"] == "periodic" else rlb.BC_OPEN, rlb.STORAGE[storage]) for t in tubes]


def _weights(case, nx, seed):
    """The loss's target densities, energy and particles (fit), or the fields' adjoint (sweepback)."""
    g = torch.Generator(device="cpu").manual_seed(int(seed) + 77)
    x = torch.linspace(0, 1, nx, dtype=torch.float64, device=DEV)
    a = torch.rand(16, generator=g, dtype=torch.float64).tolist()
    if case["kind"] == "fit":
        f = 1.0 + 0.05 * torch.sin(12 * math.pi * x + 6 * a[0]) + 0.03 * torch.cos(40 * math.pi * x + 6 * a[1])
        return torch.stack([3.0 * f, f * f])
    return torch.stack([torch.sin((3 + k) * math.pi * x + 6 * a[2 * k]) * (0.5 + a[2 * k + 1]) for k in range(8)])


# ---------------------------------------------------------------------------------------------------------------
# Passes
# ---------------------------------------------------------------------------------------------------------------

def prepare(case, seed):
    tubes, P, n, v = _inputs(case, seed)
    s = {"case": case, "P": P, "n": n, "v": v}
    if case["kind"] == "fit":
        s["tubes"] = _handle_tubes(tubes)
        s["log_tau"] = torch.log(torch.tensor([t["tau"] for t in tubes], dtype=torch.float64))
        s["target"] = _weights(case, P.numel(), seed)
        return s
    h = rlb.rlb_init(_handle_tubes(tubes, case.get("storage", "f64")), P, n, v)
    s["h"] = h
    if case["kind"] == "sweepback":
        s["gf"] = _weights(case, P.numel(), seed).contiguous()
        s["F0"] = rlb.rlb_get_state(h, torch.empty(h.state_size, dtype=torch.float64, device=DEV))
        return s
    if case["graph"]:
        rlb.rlb_set_launch(h, {"schedule": rlb.SCHED_COUNTER if case["tubes"] == "batch" else rlb.SCHED_TILE,
                               "ctas_per_sm": 0, "graph_steps": case["graph"], "order": rlb.ORDER_COST, "split": 0})
    s["fields"] = torch.empty((rlb.NFIELDS, h.nx_total), dtype=torch.float64, device=DEV)
    s["state"] = torch.empty(h.state_size, dtype=torch.float64, device=DEV)
    if case["restart"]:
        s["F0"] = rlb.rlb_get_state(h, torch.empty_like(s["state"]))
    return s


def run(s):
    case = s["case"]
    if case["kind"] == "fit":
        leaves = [s["log_tau"].detach().requires_grad_(True)] + [s[k].detach().requires_grad_(True) for k in ("P", "n", "v")]
        fields = run_fields(*leaves, s["tubes"], case["steps"], case["every"])
        loss = 0.5 * ((fields[[rlb.F_E, rlb.F_N]] - s["target"]) ** 2).sum()
        grads = torch.autograd.grad(loss, leaves)
        return {"fields": fields.detach(), "log_tau": grads[0], "P": grads[1], "n": grads[2], "v": grads[3]}
    h = s["h"]
    if case["kind"] == "sweepback":
        rlb.rlb_set_state(h, s["F0"])
        rlb.rlb_record(h, case["steps"], case["every"])
        seed = rlb.rlb_fields_vjp(h, s["gf"], torch.empty_like(s["F0"]))
        gF, glt = rlb.rlb_backward(h, seed, torch.empty_like(s["F0"]))
        g = [torch.empty_like(s["P"]) for _ in range(3)]
        rlb.rlb_init_vjp(h, s["P"], s["n"], s["v"], gF, *g)
        return {"state": gF, "log_tau": glt, "P": g[0], "n": g[1], "v": g[2]}
    if case["restart"]:
        rlb.rlb_set_state(h, s["F0"])
    rlb.rlb_step(h, case["steps"])
    fields = rlb.rlb_moments(h, s["fields"])
    state = rlb.rlb_get_state(h, s["state"])
    # the checkpoint a program keeps has the handle's storage type
    return {"fields": fields, "state": state.to(STORE[case["storage"]])}


def work(case):
    """The start read once, the result written once (a reverse sweep: the adjoint of each); the method's arithmetic
    per velocity, cell and stage: 84 operations forward, 201 reverse, plus the run before it."""
    tubes = _tubes(case)
    nodes = sum(t["Nx"] * t["Qp"] * t["Qxi"] for t in tubes)
    cells = sum(t["Nx"] for t in tubes)
    if case["kind"] != "run":
        extra = 8 * nodes * 2 if case["kind"] == "sweepback" else 0
        return {"bytes": 8 * cells * (3 + 3 + 8 + 1) + extra, "flops": 3 * case["steps"] * nodes * (84 + 201)}
    size = {"f64": 8, "f32": 4, "bf16": 2}[case["storage"]]
    return {"bytes": 2 * size * nodes + 8 * 8 * cells, "flops": 3 * case["steps"] * nodes * 84}


# ---------------------------------------------------------------------------------------------------------------
# The method in 64 bits
# ---------------------------------------------------------------------------------------------------------------

def _legendre_rule(n):
    L = np.longdouble
    x = np.polynomial.legendre.leggauss(n)[0].astype(L)
    for _ in range(3):  # Newton steps in extended precision
        p0, p1 = np.ones_like(x), x.copy()
        for k in range(2, n + 1):
            p0, p1 = p1, ((2 * k - 1) * x * p1 - (k - 1) * p0) / L(k)
        d = n * (x * p1 - p0) / (x * x - 1)
        x = x - p1 / d
    x = (x - x[::-1]) / 2
    return x, 2 / ((1 - x * x) * d * d)


def _laguerre(l, x):  # L^(1)_l
    p0, p1 = np.ones_like(x), 2 - x
    if l == 0:
        return p0
    for k in range(2, l + 1):
        p0, p1 = p1, ((2 * k - x) * p1 - k * p0) / np.longdouble(k)
    return p1


def _laguerre_rule(n):
    k = np.arange(n)
    x = np.linalg.eigvalsh(np.diag(2.0 * k + 2) + np.diag(np.sqrt(k[1:] * (k[1:] + 1.0)), 1)
                           + np.diag(np.sqrt(k[1:] * (k[1:] + 1.0)), -1)).astype(np.longdouble)
    for _ in range(3):
        d = (n * _laguerre(n, x) - (n + 1) * _laguerre(n - 1, x)) / x
        x = x - _laguerre(n, x) / d
    return x, x / ((n + 1) * _laguerre(n + 1, x) ** 2)


class _Method:
    """One tube's step in plain torch, F as [Qp, Qxi, Nx]."""

    def __init__(self, t):
        self.t = t
        p, wp = _laguerre_rule(t["Qp"])
        xi, wxi = _legendre_rule(t["Qxi"])
        ten = lambda a: torch.tensor(np.asarray(a, dtype=np.float64), device=DEV)  # noqa: E731
        self.p, self.xi = ten(p), ten(xi)
        self.xi_host = [float(a) for a in xi]
        self.ws = ten(0.5 * wp[:, None] * wxi[None, :])
        Np, Nv = t["Np"], t["Nv"]
        K = np.zeros((t["Qp"], Np + 1), dtype=np.longdouble)
        for q in range(Np + 1):
            for l in range(q, Np + 1):
                K[:, q] += (-1) ** q * math.comb(l, q) * _laguerre(l, p)
        self.K = ten(wp[:, None] * K)  # [Qp, Np + 1]

        def pol(x):
            P = [np.ones_like(x), x.copy()]
            for k in range(2, Nv + 1):
                P.append(((2 * k - 1) * x * P[-1] - (k - 1) * P[-2]) / np.longdouble(k))
            return np.stack(P[:Nv + 1])

        self.PW = ten(wxi * pol(xi))  # [Nv + 1, Qxi]
        y, wy = _legendre_rule(64)  # a rule of its own for the projection of (1 - beta xi)^-m
        self.y = ten(y)
        self.Y = ten((wy * pol(y) * (np.arange(Nv + 1)[:, None] + np.longdouble(0.5))).T)  # [64, Nv + 1]

    def equilibrium(self, n, T, beta):
        g = torch.sqrt(1.0 - beta * beta)
        base = 1.0 / (1.0 - beta[:, None] * self.y)
        h, B = base * base, 0.0
        for q in range(self.t["Np"] + 1):
            H = h @ self.Y  # [Nx, Nv + 1]
            B = B + self.K[:, q, None, None] * ((T * g) ** (q + 2))[:, None] * H
            h = h * base
        B = B * (n / (4.0 * T ** 3))[:, None]  # [Qp, Nx, Nv + 1]
        return torch.matmul(B, self.PW).transpose(1, 2)  # [Qp, Qxi, Nx]

    def moments(self, F):
        a, b = torch.einsum("ijx,i->jx", F, self.p), torch.einsum("ijx,i->jx", F, self.p ** 2)
        N0, Nx, T00 = a.sum(0), self.xi @ a, b.sum(0)
        return N0, Nx, T00, self.xi @ b, (self.xi ** 2) @ b

    def landau(self, m):
        A = m[2] + m[4]
        e = 0.5 * ((m[2] - m[4]) + torch.sqrt(A * A - 4.0 * m[3] * m[3]))
        beta = m[3] / (m[4] + e)
        n = (m[0] - beta * m[1]) / torch.sqrt(1.0 - beta * beta)
        return e, beta, n, e / (3.0 * n)

    def fields(self, F):
        m = self.moments(F)
        e, beta, n, _ = self.landau(m)
        return torch.stack(list(m) + [e, beta, n])

    def _difference(self, g):
        """Phi(x + 1/2) - Phi(x - 1/2) for a wind toward increasing x, rows of g."""
        N = g.shape[-1]
        if self.t["bc"] == "periodic":
            q = torch.cat([g[..., -3:], g, g[..., :3]], -1)
        else:
            q = torch.cat([g[..., :1]] * 3 + [g] + [g[..., -1:]] * 3, -1)
        a, b, c, d, e = (q[..., k:k + N + 1] for k in range(5))
        s0 = 13.0 / 12.0 * (a - 2 * b + c) ** 2 + 0.25 * (a - 4 * b + 3 * c) ** 2
        s1 = 13.0 / 12.0 * (b - 2 * c + d) ** 2 + 0.25 * (b - d) ** 2
        s2 = 13.0 / 12.0 * (c - 2 * d + e) ** 2 + 0.25 * (3 * c - 4 * d + e) ** 2
        w0, w1, w2 = 0.1 / (1e-6 + s0) ** 2, 0.6 / (1e-6 + s1) ** 2, 0.3 / (1e-6 + s2) ** 2
        # the candidates relative to the upwind cell, whose own difference is taken exactly
        r = w0 * (2 * (a - c) - 7 * (b - c)) + w1 * (-(b - c) + 2 * (d - c)) + w2 * (5 * (d - c) - (e - c))
        r = r / (6.0 * (w0 + w1 + w2))
        return (c[..., 1:] - c[..., :-1]) + (r[..., 1:] - r[..., :-1])

    def rhs(self, F, itau):
        t = self.t
        rate = feq = None
        if itau is not None:
            _, beta, n, T = self.landau(self.moments(F))
            g = 1.0 / torch.sqrt(1.0 - beta * beta)
            feq = self.equilibrium(n, T, beta)
            rate = (g * itau, g * beta * itau)
        step = max(1, int(3e7 / t["Nx"]))
        out = []
        for i in range(t["Qp"]):
            rows = []
            for j0 in range(0, t["Qxi"], step):
                js = list(range(j0, min(t["Qxi"], j0 + step)))
                while js:  # runs of one wind direction
                    sign = [(self.xi_host[j] > 0) - (self.xi_host[j] < 0) for j in js]
                    k = next((q for q, sg in enumerate(sign) if sg != sign[0]), len(js))
                    sl = slice(js[0], js[0] + k)
                    f, ws, xi = F[i, sl], self.ws[i, sl, None], self.xi[sl, None]
                    if sign[0] > 0:
                        d = self._difference(f / ws) * ws
                    elif sign[0] < 0:
                        d = -(self._difference((f / ws).flip(-1)) * ws).flip(-1)
                    else:
                        d = torch.zeros_like(f)
                    r = -xi / t["dx"] * d
                    if feq is not None:
                        r = r + (rate[0] - rate[1] * xi) * (feq[i, sl] - f)
                    rows.append(r)
                    js = js[k:]
            out.append(torch.cat(rows))
        return torch.stack(out)

    def step(self, F, itau):
        """One SSP-RK3 step; itau: 1/tau, None without collisions."""
        dt = self.t["dt"]
        F1 = F + dt * self.rhs(F, itau)
        F2 = 0.75 * F + 0.25 * (F1 + dt * self.rhs(F1, itau))
        return F / 3.0 + 2.0 / 3.0 * (F2 + dt * self.rhs(F2, itau))


def exact(case, seed):
    tubes, P, n, v = _inputs(case, seed)
    nx = P.numel()
    W = None if case["kind"] == "run" else _weights(case, nx, seed)
    states, fields, grads, at = [], [], [], 0
    for t in tubes:
        cells = slice(at, at + t["Nx"])
        at += t["Nx"]
        if case["kind"] == "run":
            with torch.no_grad():
                m = _Method(t)
                F = m.equilibrium(n[cells], P[cells] / n[cells], v[cells])
                itau = 1.0 / t["tau"] if math.isfinite(t["tau"]) else None
                for _ in range(case["steps"]):
                    F = m.step(F, itau)
                fields.append(m.fields(F))
                states.append(F.reshape(-1))
            continue
        lt = torch.log(torch.tensor(t["tau"], dtype=torch.float64, device=DEV)).requires_grad_(True)
        leaf = [lt] + [a[cells].detach().requires_grad_(True) for a in (P, n, v)]
        m = _Method(t)
        F0 = m.equilibrium(leaf[2], leaf[1] / leaf[2], leaf[3])
        F, itau = F0, torch.exp(-lt)
        for _ in range(case["steps"]):  # each step is evaluated again on the way back
            F = checkpoint(m.step, F, itau, use_reentrant=False)
        f = m.fields(F)
        if case["kind"] == "fit":
            loss = 0.5 * ((f[[5, 7]] - W[:, cells]) ** 2).sum()
        else:
            loss = (W[:, cells] * f).sum()
        grads.append(torch.autograd.grad(loss, leaf + [F0]))
        fields.append(f.detach())
    if case["kind"] == "run":
        return {"fields": torch.cat(fields, 1), "state": torch.cat(states)}
    cat = [torch.cat([g[k].reshape(-1) for g in grads]) for k in range(5)]
    out = {"log_tau": cat[0], "P": cat[1], "n": cat[2], "v": cat[3]}
    return dict(out, fields=torch.cat(fields, 1)) if case["kind"] == "fit" else dict(out, state=cat[4])
