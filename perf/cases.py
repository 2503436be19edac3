"""The work that users of this library have it do, as cases that can be timed and checked.

Every case goes through the package's public calls (Simulation, Batch, TumorRollout, the C
binding's static solve).  Inputs are made on the GPU from a seed: a brain-shaped phantom with a
developed tumor (hypoxic core, edema, a displacement from the initial solve and a velocity in
the direction it grows), so that no field is trivial.  `exact` restates the operator-split step
in plain torch, every solve to 1e-12, without the package.

A pass of a stepping case starts from a kept checkpoint (the way a gradient's recompute, a
parameter study or a restarted run does): restore the fields, forget the step history, step.
"""
import math

import numpy as np
import torch

from paper_1810_05370_gb300 import Simulation, _tg
from paper_1810_05370_gb300.batch import Batch
from paper_1810_05370_gb300 import rollout

TWO_PI = 2.0 * math.pi
DT = 0.01
FIELDS = ("p", "i", "n", "g", "w", "f", "o", "l", "ux", "uy", "uz", "vx", "vy", "vz")
U = ("ux", "uy", "uz")
V = ("vx", "vy", "vz")
GROWTH = 5.0          # v = GROWTH u at the checkpoint: the displacement grows with the tumor


def _params(case):
    return {
        "k_g": 0.01, "k_w": 0.1, "k_f": 0.0, "k_scale": case.get("k_scale", 1.0),
        "rho_g": case.get("rho", 10.0), "rho_w": case.get("rho", 10.0), "rho_i_frac": 0.1,
        "alpha0": 0.15, "beta0": 0.02, "gamma": 1.0, "sigma_b": 0.9,
        "o_hyp": 0.65, "o_inv": 0.7, "o_heal": 1.0, "delta_s": 55.0, "delta_p": 8.0,
        "eps_H": 0.01, "E": [2100.0, 2100.0, 2100.0, 100.0, 15000.0], "nu": [0.45] * 5,
        "eta": [0.0, 1.0e4, 1.0e4, 1.0e4, 1.0e6], "E_scale": 1.0, "zeta": 14000.0,
        "delta_e": 40.0, "delta_half": 0.01, "delta_l": 80.0,
        "rtol_diff": 1.0e-8, "rtol_elas": 1.0e-8, "maxit_diff": 1000, "maxit_elas": 10000,
        "precond_elas": case.get("precond", 0), "model": case.get("model", 0),
    }


def _case(name, kind, n, **more):
    return dict({"name": name, "kind": kind, "nx": n[0], "ny": n[1], "nz": n[2]}, **more)


def listed():
    return [
        # the smallest call: the workspace-free solve a host program makes in a latency-critical
        # loop (Jacobi-PCG, grids of at most 32^3 voxels)
        _case("static solve 16", "static", (16, 16, 16)),
        # an elasticity solve of its own, caller's right-hand side, a ragged anisotropic grid
        _case("solve fp64 96x80x72", "solve", (96, 80, 72), precision="fp64"),
        # the small forward workload: 32^3, FP64, Jacobi
        _case("step fp64 32", "step", (32, 32, 32), precision="fp64", steps=2),
        # the plain forward workload's grid with the benchmark's preconditioner, FP64
        _case("step fp64 128", "step", (128, 128, 128), precision="fp64", precond=2, steps=1),
        # one point of a mass-effect study: new parameters, two steps, diagnostics with fields
        _case("study mixed 64", "study", (64, 64, 64), precision="mixed", precond=1, steps=2),
        # the mixed-precision forward run at the batch's and at the headline's largest grid
        _case("step mixed 128", "step", (128, 128, 128), precision="mixed", precond=2, steps=2),
        _case("step mixed 256", "step", (256, 256, 256), precision="mixed", precond=2, steps=2),
        # a cropped scan: no axis a power of two, so Jacobi
        _case("step mixed 100x84x60", "step", (100, 84, 60), precision="mixed", steps=1),
        # the single-species model
        _case("single mixed 128", "step", (128, 128, 128), precision="mixed", precond=2, steps=1,
              model=1),
        # parameter estimation: forward and discrete adjoint through torch.autograd
        _case("gradient fp64 48x40x36", "gradient", (48, 40, 36), steps=3, every=2),
        # many patients at once, each on its own stream
        _case("batch mixed 64 96 64 128", "batch", (128, 128, 128), precision="mixed",
              sizes="64 96 64 128"),
        # a caller whose state lives in (pinned) host memory
        _case("host mixed 128", "host", (128, 128, 128), precision="mixed", precond=2),
    ]


def draw(rng):
    def log_int(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    def ragged(most):
        while True:
            n = tuple(log_int(12, 144) for _ in range(3))
            if n[0] * n[1] * n[2] <= most:
                return n

    def pow2(most):
        while True:
            n = tuple(1 << rng.randint(4, 8) for _ in range(3))
            if n[0] * n[1] * n[2] <= most:
                return n

    more = {"rho": round(rng.uniform(5.0, 15.0), 2), "k_scale": round(rng.uniform(0.5, 2.0), 2)}
    kind = rng.choice(["static", "solve", "step", "step", "step", "step", "study", "gradient",
                       "batch", "host"])
    prec = rng.choice(["fp64", "mixed", "mixed"])
    most = 1 << (20 if prec == "fp64" else 22)
    if kind == "static":
        while True:
            n = tuple(log_int(8, 64) for _ in range(3))
            if n[0] * n[1] * n[2] <= 32768:
                break
    elif kind == "gradient":
        n = ragged(120000)
        more.update(steps=rng.randint(2, 4), every=2)
    elif kind == "batch":
        n = (128, 128, 128)
        more.update(precision="mixed",
                    sizes=" ".join(str(rng.choice([64, 96, 128])) for _ in range(rng.randint(2, 4))))
    elif kind == "study":
        n = pow2(most)
        more.update(precision="mixed", precond=rng.choice([1, 2]), steps=rng.randint(1, 3))
    else:
        jacobi = rng.random() < 0.4
        n = ragged(min(most, 1 << 20)) if jacobi else pow2(most)
        more.update(precision=prec, precond=0 if jacobi else rng.choice([1, 2, 2]))
        if kind == "step":
            more.update(steps=rng.randint(1, 2), model=1 if rng.random() < 0.15 else 0)
    c = _case("", kind, n, **more)
    del c["name"]
    return c


def _voxels(case):
    if case["kind"] == "batch":
        return sum(int(s) ** 3 for s in case["sizes"].split())
    return case["nx"] * case["ny"] * case["nz"]


def work(case):
    """Bytes: the state (or right-hand side) in and the results out, once, in 8-byte values.
    Operations: per step the transport's 10 tricubic interpolations (about 1700), reactions
    (300) and one application of each operator; a solve alone one application."""
    m, steps = _voxels(case), case.get("steps", 1)
    if case["kind"] in ("static", "solve"):
        return {"bytes": 8.0 * m * (7 + 3 + 3), "flops": 130.0 * m}
    if case["kind"] == "gradient":
        return {"bytes": 8.0 * m * (9 + 1 + 1), "flops": 5000.0 * m * steps}
    more = 3 if case["kind"] == "study" else 0
    return {"bytes": 8.0 * m * (15 + 14 + more), "flops": 2200.0 * m * steps}


# ------------------------------------------------------------------------------- inputs

def _phantom(n, seed, single=False):
    """Nested rough ellipsoids (white matter, gray matter, CSF, background) and a tumor with
    a hypoxic core: FP64 CUDA tensors (nz, ny, nx)."""
    nx, ny, nz = n
    rng = np.random.default_rng(seed)
    dev = torch.device("cuda")
    ax = [torch.arange(m, dtype=torch.float64, device=dev) * (TWO_PI / m) for m in (nx, ny, nz)]
    X, Y, Z = ax[0][None, None, :], ax[1][None, :, None], ax[2][:, None, None]

    def rough():
        k = rng.integers(-4, 5, size=(24, 3))
        c = rng.standard_normal(24) * np.exp(-(k * k).sum(1) / 16.0)
        c = c * np.exp(1j * rng.uniform(0, TWO_PI, 24)) / max(math.sqrt(0.5 * (c * c).sum()), 1e-9)
        k = torch.from_numpy(k.astype(np.float64)).to(dev)
        e = [torch.exp(1j * k[:, d, None] * ax[d][None, :]) for d in range(3)]
        yx = (e[1][:, :, None] * e[0][:, None, :]).reshape(len(k), -1)
        ez = e[2] * torch.from_numpy(c).to(dev)[:, None]
        return (ez.T @ yx).real.reshape(nz, ny, nx)

    def level(a):
        r = torch.sqrt(((X - math.pi) / a[0]) ** 2 + ((Y - math.pi) / a[1]) ** 2
                       + ((Z - math.pi) / a[2]) ** 2)
        return r - 1.0 + 0.04 * rough()

    h = sum(TWO_PI / m for m in n) / 3.0
    wm = level((1.5, 1.8, 1.3))
    gm = torch.minimum(level((2.2, 2.5, 2.0)), wm)
    cs = torch.minimum(level((2.4, 2.7, 2.2)), gm)
    s = [0.5 * (1.0 - torch.tanh(v / (1.5 * h))) for v in (wm, gm, cs)]
    at = [math.pi + o + rng.uniform(-0.15, 0.15) for o in (0.6, 0.4, 0.3)]
    width = max(2.0 * h, rng.uniform(0.2, 0.3))

    def wrapped(x, x0):
        return x - x0 - TWO_PI * torch.round((x - x0) / TWO_PI)

    G = torch.exp(-(wrapped(X, at[0]) ** 2 + wrapped(Y, at[1]) ** 2 + wrapped(Z, at[2]) ** 2)
                  / (2.0 * width * width))
    w, g = s[0], s[1] - s[0]
    healthy = g + w
    st = {"f": s[2] - s[1], "bg": 1.0 - s[2]}
    if single:
        st["p"] = 0.8 * G * healthy
        st["i"] = st["n"] = torch.zeros_like(G)
        taken = 0.8 * G
    else:
        st["p"], st["i"], st["n"] = 0.7 * G * healthy, 0.07 * G * healthy, 0.1 * G ** 4 * healthy
        taken = 0.77 * G + 0.1 * G ** 4
    st["g"], st["w"] = g * (1.0 - taken), w * (1.0 - taken)
    st["o"] = 1.0 - 0.45 * G * healthy
    st["l"] = 0.25 * G * healthy
    for k in U + V:
        st[k] = torch.zeros_like(G)
    return {k: v.contiguous() for k, v in st.items()}


def _grid(case):
    return case["nx"], case["ny"], case["nz"]


def _rhs(n, seed):
    """A smooth, localised load (the residual of a force balance, say)."""
    b = _phantom(n, seed + 7)
    t = b["p"] + b["l"]
    return [2.0e3 * (torch.roll(t, -1, 2 - d) - torch.roll(t, 1, 2 - d)) * (1.0 + b["w"])
            for d in range(3)]


def _copy_into(dst, src):
    torch._foreach_copy_(dst, src)


def prepare(case, seed):
    kind, n, P = case["kind"], _grid(case), _params(case)
    single = case.get("model", 0) == 1
    if kind == "batch":
        sims = [((m, m, m), _params(dict(case, precond=2 if m & (m - 1) == 0 else 0)),
                 _phantom((m, m, m), seed + 100 * k))
                for k, m in enumerate(int(s) for s in case["sizes"].split())]
        batch = Batch(sims, concurrent=True, precision=case["precision"])
        torch.cuda.synchronize()
        live, kept = [], []
        for st in batch.states:
            for a in range(3):
                st[V[a]].copy_(GROWTH * st[U[a]])
            live += [st[k] for k in FIELDS]
            kept += [st[k].clone() for k in FIELDS]
        torch.cuda.synchronize()
        return {"kind": kind, "batch": batch, "live": live, "kept": kept}
    if kind == "gradient":
        st = _phantom(n, seed)
        r = _phantom(n, seed + 3)
        return {"kind": kind, "n": n, "P": P, "state": st, "lam": (r["p"] - 0.9 * st["p"]),
                "theta": torch.tensor(rollout.theta_of(P), device="cuda"),
                "steps": case["steps"], "every": case["every"]}
    if kind == "static":
        st = _phantom(n, seed)
        u = [torch.zeros_like(st["p"]) for _ in range(3)]
        cs = _tg.tg_state()
        for k in ("p", "i", "n", "g", "w", "f", "o", "l", "bg"):
            setattr(cs, k, st[k].data_ptr())
        for a in range(3):
            cs.u[a] = st[U[a]].data_ptr()
            cs.v[a] = st[V[a]].data_ptr()
        return {"kind": kind, "grid": _tg.make_grid(n), "params": _tg.make_params(P), "cs": cs,
                "state": st, "u": u}
    sim = Simulation(n, P, _phantom(n, seed, single), precision=case["precision"])
    s = {"kind": kind, "sim": sim, "steps": case.get("steps", 1)}
    if kind == "solve":
        s["rhs"] = _rhs(n, seed)
        s["u"] = [torch.zeros_like(sim.state["p"]) for _ in range(3)]
        return s
    for a in range(3):
        sim.state[V[a]].copy_(GROWTH * sim.state[U[a]])
    if kind == "host":
        s["in"] = {k: v.cpu().pin_memory() for k, v in sim.state.items()}
        s["out"] = {k: torch.zeros_like(v).pin_memory() for k, v in s["in"].items()}
        return s
    s["live"] = [sim.state[k] for k in FIELDS]
    s["kept"] = [v.clone() for v in s["live"]]
    if kind == "study":
        s["params"] = _study_params(case)
        s["seed"] = tuple(math.pi + o for o in (0.6, 0.4, 0.3))
        s["threshold"] = 0.1 * sum(TWO_PI / m for m in n) / 3.0
    return s


def _study_params(case):
    P = _params(case)
    P["eta"] = [0.0, 3.0e3, 3.0e3, 3.0e3, 1.0e6]
    P["zeta"] = 2.0e4
    return P


# --------------------------------------------------------------------------------- passes

def run(s):
    kind = s["kind"]
    if kind == "static":
        for u in s["u"]:
            u.zero_()
        _tg.tg_solve_elasticity_static(s["grid"], s["params"], s["cs"], None,
                                       [u.data_ptr() for u in s["u"]],
                                       torch.cuda.current_stream().cuda_stream)
        return s["u"]
    if kind == "gradient":
        theta = s["theta"].clone().requires_grad_(True)
        state = {k: v.clone() for k, v in s["state"].items()}
        p = rollout.TumorRollout.apply(theta, s["n"], s["P"], state, s["steps"], DT, s["every"])
        p.backward(s["lam"])
        return {"p": p.detach(), "grad": theta.grad}
    if kind == "batch":
        _copy_into(s["live"], s["kept"])
        torch.cuda.current_stream().synchronize()   # the members step on streams of their own
        s["batch"].step(DT, 1)
        return s["live"]
    sim = s["sim"]
    if kind == "solve":
        for u in s["u"]:
            u.zero_()
        sim.solve_elasticity(s["rhs"], s["u"])
        return s["u"]
    if kind == "host":
        sim.reset_history()
        sim.step_host(s["in"], s["out"], DT)
        return {k: s["out"][k] for k in FIELDS}
    _copy_into(s["live"], s["kept"])
    if kind == "study":
        sim.set_params(s["params"])
        sim.step(DT, nsteps=s["steps"])
        d = sim.diagnostics(s["seed"], s["threshold"], fields=True)
        return {"diag": d, "state": s["live"]}
    sim.reset_history()
    sim.step(DT, nsteps=s["steps"])
    return s["live"]


# ------------------------------------------------------------- the same in plain torch, 64 bits

class _Model:
    def __init__(self, n, P, L=TWO_PI):
        self.n, self.P = n, P
        self.h = [L / m for m in n]

    @staticmethod
    def sh(x, d, s):
        """x at the node s steps further along axis d (0: x)."""
        return torch.roll(x, -s, 2 - d)

    # diffusion -------------------------------------------------------------------------
    def faces(self, st):
        P = self.P
        K = (P["k_scale"] * (P["k_g"] * st["g"] + P["k_w"] * st["w"] + P["k_f"] * st["f"])).clamp(min=0)
        out = []
        for d in range(3):
            b = self.sh(K, d, 1)
            s = K + b
            out.append(torch.where(s > 0, 2 * K * b / torch.where(s > 0, s, torch.ones_like(s)),
                                   torch.zeros_like(s)) * (0.5 * DT / self.h[d] ** 2))
        return out

    def diffuse(self, F, c):
        r = torch.zeros_like(c)
        for d in range(3):
            t = F[d] * (self.sh(c, d, 1) - c)
            r += t - self.sh(t, d, -1)
        return r

    def cn(self, F, c):
        diag = 1.0 + sum(f + self.sh(f, d, -1) for d, f in enumerate(F))
        return _pcg(lambda x: x - self.diffuse(F, x), lambda r: r / diag, c + self.diffuse(F, c), c)

    # elasticity ------------------------------------------------------------------------
    def lame(self, st):
        P = self.P
        iota = [st["p"] + st["i"] + st["n"], st["g"], st["w"], st["f"], st["bg"]]
        E = [P["E_scale"] * e for e in P["E"]]
        mu = sum(E[s] / (2 * (1 + P["nu"][s])) * iota[s] for s in range(5))
        lam = sum(P["nu"][s] * E[s] / ((1 - 2 * P["nu"][s]) * (1 + P["nu"][s])) * iota[s]
                  for s in range(5))
        return mu, lam, sum(P["eta"][s] * iota[s] for s in range(5))

    def elas(self, st):
        mu, lam, eta = self.lame(st)
        sh, h = self.sh, self.h
        mf = [0.5 * (mu + sh(mu, d, 1)) for d in range(3)]
        lf = [0.5 * (lam + sh(lam, d, 1)) + 2 * mf[d] for d in range(3)]
        dia = torch.stack([eta + sum((lf if d == a else mf)[d] / h[d] ** 2
                                     + sh((lf if d == a else mf)[d], d, -1) / h[d] ** 2
                                     for d in range(3)) for a in range(3)])

        def grad(x, d):
            return (sh(x, d, 1) - sh(x, d, -1)) / (2 * h[d])

        def A(u):
            out = []
            for a in range(3):
                r = eta * u[a]
                for d in range(3):
                    t = (lf if d == a else mf)[d] * (sh(u[a], d, 1) - u[a]) / h[d] ** 2
                    r -= t - sh(t, d, -1)
                    if d != a:
                        r -= grad(mu * grad(u[d], a), d) + grad(lam * grad(u[d], d), a)
                out.append(r)
            return torch.stack(out)

        m0, l0, e0 = (float(x.mean()) for x in (mu, lam, eta))
        th = [torch.arange(m, dtype=torch.float64, device=mu.device) * (TWO_PI / m) for m in self.n]
        shape = [(1, 1, -1), (1, -1, 1), (-1, 1, 1)]
        S = [((2 - 2 * torch.cos(th[d])) / h[d] ** 2).reshape(shape[d]) for d in range(3)]
        T = [(torch.sin(th[d]) / h[d]).reshape(shape[d]) for d in range(3)]
        D = [e0 + m0 * (S[0] + S[1] + S[2]) + (l0 + m0) * (S[a] - T[a] ** 2) for a in range(3)]
        den = 1 + (l0 + m0) * sum(T[a] ** 2 / D[a] for a in range(3))
        d0 = [e0 + sum(2 * (l0 + 2 * m0 if d == a else m0) / h[d] ** 2 for d in range(3))
              for a in range(3)]
        s = torch.stack([torch.sqrt(d0[a] / dia[a]) for a in range(3)])

        def M(r):
            w = [torch.fft.fftn(s[a] * r[a]) / D[a] for a in range(3)]
            c = (l0 + m0) * sum(T[a] * w[a] for a in range(3)) / den
            return torch.stack([s[a] * torch.fft.ifftn(w[a] - c * T[a] / D[a]).real
                                for a in range(3)])

        return A, M

    def force(self, st):
        s = st["p"] + st["n"]
        t = self.P["zeta"] * torch.tanh(s)
        return torch.stack([t * (self.sh(s, d, 1) - self.sh(s, d, -1)) / (2 * self.h[d])
                            for d in range(3)])

    def displacement(self, st, rhs=None, start=None):
        A, M = self.elas(st)
        b = -self.force(st) if rhs is None else torch.stack(list(rhs))
        return _pcg(A, M, b, torch.zeros_like(b) if start is None else start)

    # transport -------------------------------------------------------------------------
    def taps(self, X):
        idx, wgt = [], []
        for d in range(3):
            fl = torch.floor(X[d])
            t = X[d] - fl
            wgt.append([-t * (t - 1) * (t - 2) / 6, (t + 1) * (t - 1) * (t - 2) / 2,
                        -(t + 1) * t * (t - 2) / 2, (t + 1) * t * (t - 1) / 6])
            idx.append([(fl.long() + a) % self.n[d] for a in (-1, 0, 1, 2)])
        return idx, wgt

    def interp(self, taps, fields):
        idx, wgt = taps
        out = [torch.zeros_like(f) for f in fields]
        for c in range(4):
            for b in range(4):
                row = (idx[2][c] * self.n[1] + idx[1][b]) * self.n[0]
                wzy = wgt[2][c] * wgt[1][b]
                for a in range(4):
                    at, w = row + idx[0][a], wzy * wgt[0][a]
                    for o, f in zip(out, fields):
                        o += w * f.reshape(-1)[at]
        return out

    def transport(self, st):
        v = [st[k] for k in V]
        dev = v[0].device
        ax = [torch.arange(m, dtype=torch.float64, device=dev) for m in self.n]
        j = [ax[0][None, None, :], ax[1][None, :, None], ax[2][:, None, None]]
        div = sum((self.sh(v[d], d, 1) - self.sh(v[d], d, -1)) / (2 * self.h[d]) for d in range(3))
        vs = self.interp(self.taps([j[d] - DT * v[d] / self.h[d] for d in range(3)]), v)
        X = [j[d] - 0.5 * DT * (v[d] + vs[d]) / self.h[d] for d in range(3)]
        keys = ("p", "i", "n", "g", "w", "f")
        q = self.interp(self.taps(X), [div] + [st[k] for k in keys])
        dX = q[0]
        for k, x in zip(keys, q[1:]):
            if k == "f":
                st[k] = x
            else:
                gx = -x * dX
                st[k] = x + 0.5 * DT * (gx - (x + DT * gx) * div)

    # reactions -------------------------------------------------------------------------
    @staticmethod
    def share(g, w):
        s = g + w
        ok = s > 0
        d = torch.where(ok, s, torch.ones_like(s))
        return torch.where(ok, g / d, torch.zeros_like(s)), torch.where(ok, w / d, torch.zeros_like(s))

    def rates(self, rho, o, y):
        P = self.P
        p, i, n, g, w = y

        def H(x):
            return 1 / (1 + torch.exp(-2 * x / P["eps_H"]))

        h = P["gamma"] * H(P["o_hyp"] - o)
        al = P["alpha0"] * H(P["o_inv"] - o)
        be = P["beta0"] * H(P["sigma_b"] - p - i) * o
        mit = 0.5 * (P["o_hyp"] + P["o_inv"])
        mf = torch.where(o > P["o_inv"], torch.ones_like(o),
                         torch.where(o >= mit, (o - mit) / (P["o_inv"] - mit), torch.zeros_like(o)))
        R, Rt = rho * p * (1 - p) * mf, P["rho_i_frac"] * rho * i * (1 - i) * mf
        fg, fw = self.share(g, w)
        return [R - al * p + be * i - h * p, Rt + al * p - be * i - h * i, h * (p + i + g + w),
                -fg * (R + Rt) - h * g, -fw * (R + Rt) - h * w]

    def react(self, st, rho):
        P = self.P
        if P["model"] == 1:
            def rates(y):
                R = rho * y[0] * (1 - y[0])
                fg, fw = self.share(y[1], y[2])
                return [R, -fg * R, -fw * R]
            keys = ("p", "g", "w")
        else:
            def rates(y):
                return self.rates(rho, st["o"], y)
            keys = ("p", "i", "n", "g", "w")
        y = [st[k] for k in keys]
        k1 = rates(y)
        k2 = rates([a + DT * b for a, b in zip(y, k1)])
        for k, a, b, c in zip(keys, y, k1, k2):
            st[k] = a + 0.5 * DT * (b + c)
        if P["model"] == 1:
            return
        o, gw = st["o"], st["g"] + st["w"]
        k1 = -P["delta_p"] * st["p"] + P["delta_s"] * (P["o_heal"] - o) * gw
        k2 = -P["delta_p"] * st["p"] + P["delta_s"] * (P["o_heal"] - o - DT * k1) * gw
        st["o"] = o + 0.5 * DT * (k1 + k2)
        l, i = st["l"], st["i"]
        src = P["delta_e"] * i / (i + P["delta_half"]) * (1 - i)
        k1 = src - P["delta_l"] * l
        st["l"] = l + 0.5 * DT * (k1 + src - P["delta_l"] * (l + DT * k1))

    def step(self, st):
        P = self.P
        F = self.faces(st)
        rho = P["rho_g"] * st["g"] + P["rho_w"] * st["w"]
        self.transport(st)
        lead = "p" if P["model"] == 1 else "i"
        before = st[lead]
        for k in ((lead,) if P["model"] == 1 else (lead, "o", "l")):
            st[k] = self.cn(F, st[k])
        fg, fw = self.share(st["g"], st["w"])
        di = st[lead] - before
        st["g"], st["w"] = st["g"] - di * fg, st["w"] - di * fw
        self.react(st, rho)
        u0 = torch.stack([st[k] for k in U])
        u = self.displacement(st, start=u0)
        for a in range(3):
            st[U[a]] = u[a]
            st[V[a]] = (u[a] - u0[a]) / DT

    def start(self, st):
        """The checkpoint: u from the species, v = GROWTH u."""
        u = self.displacement(st)
        for a in range(3):
            st[U[a]], st[V[a]] = u[a], GROWTH * u[a]

    def diagnostics(self, st, seed, threshold):
        mu, lam, _ = self.lame(st)
        u = [st[k] for k in U]
        D = [[(self.sh(u[a], d, 1) - self.sh(u[a], d, -1)) / (2 * self.h[d]) for d in range(3)]
             for a in range(3)]
        tr = D[0][0] + D[1][1] + D[2][2]
        Fm = [[D[a][b] + (1.0 if a == b else 0.0) for b in range(3)] for a in range(3)]
        J = (Fm[0][0] * (Fm[1][1] * Fm[2][2] - Fm[1][2] * Fm[2][1])
             - Fm[0][1] * (Fm[1][0] * Fm[2][2] - Fm[1][2] * Fm[2][0])
             + Fm[0][2] * (Fm[1][0] * Fm[2][1] - Fm[1][1] * Fm[2][0]))
        trace = (3 * lam + 2 * mu) * tr
        shear = torch.sqrt((mu * (D[0][0] - D[1][1])) ** 2 + (mu * (D[0][1] + D[1][0])) ** 2)
        r2 = torch.zeros_like(tr)
        for d in range(3):
            x = torch.arange(self.n[d], dtype=torch.float64, device=tr.device) * self.h[d] - seed[d]
            x = x - TWO_PI * torch.floor(x / TWO_PI + 0.5)
            r2 = r2 + (x * x).reshape([(1, 1, -1), (1, -1, 1), (-1, 1, 1)][d])
        far = torch.sqrt(u[0] ** 2 + u[1] ** 2 + u[2] ** 2) >= threshold
        vol = self.h[0] * self.h[1] * self.h[2]
        return {"jac_min": float(J.min()), "jac_max": float(J.max()),
                "jac_dev_l2": math.sqrt(vol * float(((J - 1) ** 2).sum())),
                "trace_min": float(trace.min()), "trace_max": float(trace.max()),
                "shear_max": float(shear.max()),
                "d_max": math.sqrt(float(r2[far].max())) if bool(far.any()) else 0.0,
                "trace": trace, "shear": shear, "jacobian": J}


def _pcg(A, M, b, x, rtol=1e-12, maxit=2000):
    x = x.clone()
    r = b - A(x)
    z = M(r)
    p = z.clone()
    rz, bb = torch.sum(r * z), float(torch.sum(b * b))
    for it in range(maxit):
        if float(torch.sum(r * r)) <= rtol * rtol * bb:
            break
        q = A(p)
        al = rz / torch.sum(p * q)
        x += al * p
        r -= al * q
        z = M(r)
        new = torch.sum(r * z)
        p = z + (new / rz) * p
        rz = new
    return x


def exact(case, seed):
    kind, n, P = case["kind"], _grid(case), _params(case)
    if kind == "batch":
        out = []
        for k, m in enumerate(int(s) for s in case["sizes"].split()):
            st, model = _phantom((m, m, m), seed + 100 * k), _Model((m, m, m), P)
            model.start(st)
            model.step(st)
            out += [st[f] for f in FIELDS]
        return out
    st, model = _phantom(n, seed, case.get("model", 0) == 1), _Model(n, P)
    if kind in ("static", "solve"):
        return list(model.displacement(st, _rhs(n, seed) if kind == "solve" else None))
    if kind == "gradient":
        lam = _phantom(n, seed + 3)["p"] - 0.9 * st["p"]

        def final(P):
            s, model = dict(st), _Model(n, P)
            u = model.displacement(s)
            for a in range(3):
                s[U[a]], s[V[a]] = u[a], torch.zeros_like(u[a])
            for _ in range(case["steps"]):
                model.step(s)
            return s["p"]

        theta, g = rollout_theta(P), []
        for k in range(5):   # central differences: the truncation and the solves' 1e-12 are
            J = []           # both some 1e-9 of the derivative
            for sign in (1.0, -1.0):
                t = list(theta)
                t[k] *= 1.0 + sign * 3e-5
                J.append(float((lam * final(with_theta(P, t))).sum()))
            g.append((J[0] - J[1]) / (6e-5 * theta[k]))
        return {"p": final(P), "grad": torch.tensor(g, dtype=torch.float64, device="cuda")}
    model.start(st)
    if kind == "study":
        model = _Model(n, _study_params(case))
    for _ in range(case.get("steps", 1)):
        model.step(st)
    if kind == "host":
        return {k: st[k] for k in FIELDS}
    if kind == "study":
        d = model.diagnostics(st, tuple(math.pi + o for o in (0.6, 0.4, 0.3)),
                              0.1 * sum(TWO_PI / m for m in n) / 3.0)
        return {"diag": d, "state": [st[k] for k in FIELDS]}
    return [st[k] for k in FIELDS]


def rollout_theta(P):
    return [P["k_scale"], P["rho_w"], P["o_hyp"], P["o_inv"], P["E_scale"]]


def with_theta(P, t):
    return dict(P, k_scale=t[0], rho_g=t[1], rho_w=t[1], o_hyp=t[2], o_inv=t[3], E_scale=t[4])
