"""The work that a program using this library has it do, as cases to time.

Every case goes through the public entry points (JdProblem, JdServer, JumpDiffusionCost)
on the seeded problems of ``workloads``.  ``prepare`` builds the problem object and the
control that a program has in hand, ``run`` makes one call (or one J + backward, or one
stream of requests) and returns everything it computes.  ``exact`` gives the same numbers
from plain torch in 64 bits: the generator's counter-based draws, the jump-adapted Euler
scheme and its derivative step by step, without the library.
"""
import math

import numpy as np
import torch

import paper_2505_04328_gb300 as jd
import workloads
from paper_2505_04328_gb300.autograd import JumpDiffusionCost


def listed():
    return [
        # one short control loop on a small scalar problem in FP64 (the lq_scalar
        # configuration): every sweep is tiny, launches and latency are the time
        dict(name="lq_scalar optimize fp64", kind="optimize", model="lq_scalar", prec="fp64", mode="auto",
             M=1000, Nt=100, lam=2.0, iters=10),
        # one evaluation of J and its gradient on the headline configuration, stored states
        dict(name="double_well gradient", kind="gradient", model="double_well", prec="fp32", mode="stored",
             M=1 << 20, Nt=1000, lam=5.0),
        # a few projected-gradient iterations (gradients, paired and single line-search
        # trials) of a medium problem
        dict(name="double_well optimize", kind="optimize", model="double_well", prec="fp32", mode="auto",
             M=1 << 18, Nt=500, lam=5.0, iters=4),
        # the plan for problems whose states do not fit in memory; path and step counts
        # that divide by nothing
        dict(name="double_well recompute", kind="gradient", model="double_well_phase", prec="fp32",
             mode="recompute", M=499979, Nt=777, lam=5.0),
        # J(u, theta) and its backward inside a torch program, parameter gradients included
        dict(name="autograd theta", kind="autograd", model="double_well_autograd", prec="fp32", mode="recompute",
             M=1 << 20, Nt=1024, lam=5.0),
        # the paper's phase-space particle with Keilson-Storer velocity resets
        dict(name="ks_oscillator gradient", kind="gradient", model="ks_oscillator", prec="fp32", mode="stored",
             M=1 << 20, Nt=500, lam=math.sqrt(10.0 / math.pi)),
        # an eight-dimensional request of the serving mix, ragged
        dict(name="linear8 gradient", kind="gradient", model="linear8", prec="fp32", mode="auto",
             M=200003, Nt=313, lam=3.0),
        # d = 32 with the BF16 tensor-core drift
        dict(name="linear32 bf16 gradient", kind="gradient", model="linear32", prec="fp32", mode="stored", tc=1,
             M=1 << 18, Nt=500, lam=1.0),
        # d = 32 in FP32 on the CUDA cores, ragged
        dict(name="linear32 fp32 gradient", kind="gradient", model="linear32", prec="fp32", mode="stored", tc=0,
             M=50001, Nt=333, lam=2.5),
        # the FP64 form, where an answer is checked or the FP32 rounding is not enough
        dict(name="double_well fp64", kind="gradient", model="double_well", prec="fp64", mode="stored",
             M=1 << 17, Nt=400, lam=5.0),
        # the paper's feedback problem: dJ/dmu of 10x10 bump weights per step
        dict(name="feedback_centering gradient", kind="feedback", model="feedback_centering", prec="fp32",
             particles=0, M=1 << 20, Nt=100),
        # the small requests of the serving stream, submitted together
        dict(name="serving small requests", kind="serving", prec="fp32", requests=12, m_lo=12.0, m_hi=16.0,
             nt_lo=50, nt_hi=500, iters=3),
    ]


def _log_uniform(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["optimize", "gradient", "gradient", "gradient", "gradient", "autograd", "tensor", "fp64",
                       "feedback", "serving"])
    if kind == "optimize":
        if rng.random() < 0.5:
            return dict(kind="optimize", model="lq_scalar", prec=rng.choice(["fp64", "fp32"]), mode="auto",
                        M=_log_uniform(rng, 500, 40000), Nt=_log_uniform(rng, 50, 400),
                        lam=rng.uniform(0.5, 10.0), iters=rng.randint(2, 10))
        return dict(kind="optimize", model=rng.choice(["double_well", "ks_oscillator"]), prec="fp32",
                    mode=rng.choice(["auto", "recompute"]), M=_log_uniform(rng, 1 << 12, 1 << 18),
                    Nt=_log_uniform(rng, 50, 800), lam=rng.uniform(0.5, 8.0), iters=rng.randint(2, 4))
    if kind == "gradient":
        model = rng.choice(["double_well", "double_well_phase", "ks_oscillator", "lq_scalar", "linear4", "linear8",
                            "linear3"])
        top = 1 << 20 if model[-1] not in "348" else 1 << 18
        return dict(kind="gradient", model=model, prec="fp32", mode=rng.choice(["stored", "recompute", "auto"]),
                    M=_log_uniform(rng, 1 << 12, top), Nt=_log_uniform(rng, 50, 1000), lam=rng.uniform(0.5, 10.0))
    if kind == "autograd":
        return dict(kind="autograd", model="double_well_autograd", prec="fp32",
                    mode=rng.choice(["recompute", "stored"]), M=_log_uniform(rng, 1 << 14, 1 << 20),
                    Nt=_log_uniform(rng, 100, 1000), lam=rng.uniform(0.5, 8.0))
    if kind == "tensor":
        tc = rng.choice([0, 1, 2, 3])
        return dict(kind="gradient", model="linear32", prec="fp32", mode="stored", tc=tc,
                    M=_log_uniform(rng, 1 << 12, 1 << (18 if tc in (1, 2) else 17)),
                    Nt=_log_uniform(rng, 50, 480), lam=rng.uniform(0.5, 10.0))
    if kind == "fp64":
        return dict(kind="gradient", model=rng.choice(["double_well", "lq_scalar", "ks_oscillator", "linear4"]),
                    prec="fp64", mode=rng.choice(["stored", "recompute"]), M=_log_uniform(rng, 1 << 12, 90000),
                    Nt=_log_uniform(rng, 50, 400), lam=rng.uniform(0.5, 10.0))
    if kind == "feedback":
        ring = rng.choice([0, 0, 32, 27])
        M = _log_uniform(rng, 1 << 13, 1 << 20)
        return dict(kind="feedback", model="feedback_coupled" if ring else rng.choice(
            ["feedback_centering", "feedback_trajectory"]), prec="fp32", particles=ring,
            M=max(32, M // 32 * 32) if ring else M, Nt=_log_uniform(rng, 40, 100))
    lo = rng.uniform(12.0, 14.0)
    return dict(kind="serving", prec="fp32", requests=rng.randint(4, 14), m_lo=lo, m_hi=lo + rng.uniform(0.5, 2.0),
                nt_lo=50, nt_hi=rng.randint(150, 600), iters=rng.randint(2, 4))


# --- inputs ----------------------------------------------------------------------------
def _problem(case, seed):
    """(problem, feedback or None) of a case; seed keys the generator and the control."""
    name, M, Nt = case["model"], case["M"], case["Nt"]
    if name.startswith("linear"):
        return workloads.linear_family(int(name[6:]), M, Nt, lam=case["lam"], seed=seed), None
    if name == "feedback_coupled":
        return workloads.feedback_coupled(M=M, Nt=Nt, seed=seed, particles=case["particles"])
    if name.startswith("feedback"):
        return getattr(workloads, name)(M=M, Nt=Nt, seed=seed)
    p = getattr(workloads, name)(M=M, Nt=Nt, seed=seed)
    p.lam = case["lam"]
    return p, None


def _requests(case, seed):
    """The sizes and rates belong to the case, the generators' keys to the seed."""
    rng, keys = np.random.default_rng(case["requests"]), np.random.default_rng(seed)
    out = []
    for i in range(case["requests"]):
        M = int(np.round(2.0 ** rng.uniform(case["m_lo"], case["m_hi"])))
        Nt = int(rng.integers(case["nt_lo"], case["nt_hi"] + 1))
        p = workloads.lq_scalar(M=M, Nt=Nt) if rng.random() < 0.5 else workloads.double_well(M=M, Nt=Nt)
        p.lam = float(rng.uniform(0.5, 10.0))
        p.seed = int(keys.integers(1 << 31))
        out.append(p)
    return out


def prepare(case, seed):
    kind = case["kind"]
    if kind == "serving":
        return dict(case=case, server=jd.JdServer(max_slots=16), requests=_requests(case, seed))
    p, fb = _problem(case, seed)
    if kind == "autograd":
        u = torch.from_numpy(workloads.random_control(p, seed=seed, scale=0.5)).cuda().requires_grad_(True)
        theta = torch.tensor([0.5, 0.3, 0.2], dtype=torch.float64, requires_grad=True)
        # A[1][1] = -0.5 is the damping rho0 = 0.5 along dA
        return dict(case=case, cost=JumpDiffusionCost(p, rho0=0.5, prec=case["prec"], mode=case["mode"]), u=u,
                    theta=theta)
    prob = jd.JdProblem(p, prec=case["prec"], mode=case.get("mode", "auto"), use_tensor_cores=case.get("tc", 0))
    if kind == "feedback":
        mu = torch.from_numpy(workloads.random_mu(p, fb, seed=seed, scale=0.3)).cuda()
        return dict(case=case, prob=prob, fb=fb, mu=mu)
    return dict(case=case, prob=prob, u=workloads.random_control(p, seed=seed, scale=0.5))


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "gradient":
        J, g, _ = state["prob"].gradient(state["u"])
        return {"J": J, "grad": g}
    if kind == "optimize":
        u, res, hist = state["prob"].optimize(u0=state["u"], max_iter=case["iters"], tol_rel_grad=0.0)
        return {"u": u, "J": hist, "zeta": res["zeta"], "iters": res["iters"]}
    if kind == "autograd":
        J = state["cost"](state["u"], state["theta"])
        gu, gth = torch.autograd.grad(J, [state["u"], state["theta"]])
        return {"J": J.detach(), "grad_u": gu, "grad_theta": gth}
    if kind == "feedback":
        J, g = state["prob"].fb_gradient(state["fb"], state["mu"])
        return {"J": J, "grad": g}
    server = state["server"]
    tickets = [server.submit(p, prec=case["prec"], max_iter=case["iters"], tol_rel_grad=0.0)
               for p in state["requests"]]
    out = []
    for t in tickets:
        server.wait(t)
        u, res = server.poll(t)
        out.append({"u": u, "J": res["J"]})
    return out


# --- work ------------------------------------------------------------------------------
def _path_step_flops(d, du, cubic, adjoint=True):
    """Operations of one step of one path: the generator's blocks (20 wide multiplies and
    20 XORs each), uniforms and normals, drift, update and cost, and the adjoint's update,
    sensitivity and cost gradient."""
    P = (d + 1) // 2
    fwd = 40 * -(-(1 + 2 * P) // 4) + 13 * P + 2 * (d * d + d * du) + 4 * d + 5 * d + (2 * d * d + 2 * d) * cubic
    adj = 2 * (d * d + d * du) + 5 * d + (2 * d * d + 3 * d) * cubic
    return fwd + adj * adjoint


def work(case):
    kind = case["kind"]
    if kind == "serving":
        reqs = _requests(case, 1)
        steps = sum(p.M * p.Nt * _path_step_flops(p.d, p.du, p.drift == workloads.CUBIC) for p in reqs)
        return {"bytes": sum(16.0 * p.Nt for p in reqs), "flops": float(case["iters"]) * steps}
    p, fb = _problem(case, 1)
    per = _path_step_flops(p.d, p.du, p.drift == workloads.CUBIC)
    n = p.Nt * p.du
    if kind == "feedback":
        # 20 bumps with derivatives, three bilinear forms and the outer product
        per += 20 * 10 + 3 * 2 * fb.L + 2 * fb.L
        n = p.Nt * fb.L
    if kind == "autograd":
        per += 4 * p.d + 2 * p.d * p.d
    flops = float(per) * p.M * p.Nt
    if kind == "optimize":
        flops *= case["iters"]
    return {"bytes": 16.0 * n, "flops": flops}


# --- the same numbers in plain torch, 64 bits -------------------------------------------
_MASK = 0xFFFFFFFF


def _philox(c0, c1, c2, c3, seed):
    """Philox4x32-10 on int64 tensors holding 32-bit words: four words per counter."""
    k0, k1 = seed & _MASK, (seed >> 32) & _MASK
    for _ in range(10):
        p0, p1 = c0 * 0xD2511F53, c2 * 0xCD9E8D57
        c0, c1, c2, c3 = ((p1 >> 32) & _MASK) ^ c1 ^ k0, p1 & _MASK, ((p0 >> 32) & _MASK) ^ c3 ^ k1, p0 & _MASK
        k0, k1 = (k0 + 0x9E3779B9) & _MASK, (k1 + 0xBB67AE85) & _MASK
    return c0, c1, c2, c3


def _words(k, m, tag, epoch, seed, count):
    """The first `count` words of the stream with counters (k, m, tag | b, epoch)."""
    out = []
    zero = torch.zeros_like(k + m)
    for b in range(-(-count // 4)):
        out += _philox(zero + k, zero + m, zero + (tag | b), zero + epoch, seed)
    return out[:count]


def _u01(w):
    return ((w >> 9).double() + 0.5) * 2.0 ** -23


def _normals(w, d):
    z = []
    for a, b in zip(w[0::2], w[1::2]):
        r, ang = torch.sqrt(-2.0 * torch.log(_u01(a))), 2.0 * math.pi * _u01(b)
        z += [r * torch.cos(ang), r * torch.sin(ang)]
    return torch.stack(z[:d], dim=-1)


class _Exact:
    """One problem in 64-bit torch on the GPU."""

    def __init__(self, p, fb=None):
        self.p, self.fb = p, fb
        d, self.dev = p.d, torch.device("cuda")
        t = lambda a: torch.as_tensor(np.asarray(a, dtype=np.float64), device=self.dev)  # noqa: E731
        a = p.arrays()
        self.A, self.C, self.B = t(a["A"]), t(a["C"]), t(a["B"])
        self.sigma, self.q, self.xd = t(a["sigma"]), t(a["q"]), t(a["xd"])
        self.scale = t(p.jump_scale)
        self.cubic = p.drift == workloads.CUBIC
        self.dt = p.T / p.Nt
        self.P = (d + 1) // 2
        ring = fb is not None and fb.particles > 0
        if ring:
            self.N, lanes = fb.particles, 32
            self.m = (torch.arange(p.M // lanes, device=self.dev)[:, None] * lanes
                      + torch.arange(self.N, device=self.dev)).reshape(-1)
            ang = 2.0 * math.pi * torch.arange(self.N, device=self.dev).double() / self.N
            x0 = torch.stack([fb.ax * torch.cos(ang), fb.av * torch.sin(ang)], dim=-1)
            self.x0 = x0.repeat(p.M // lanes, 1)
        else:
            self.N = 0
            self.m = torch.arange(p.M, device=self.dev)
            self.x0 = t(a["x0"]).expand(p.M, d)
        self.paths = self.m.numel()
        # Poisson thresholds floor(2^32 F(n)), the pmf accumulated in order
        mu, thr, pn, F = p.lam * self.dt, [], math.exp(-p.lam * self.dt), math.exp(-p.lam * self.dt)
        for n in range(16):
            if n:
                pn = pn * mu / n
                F += pn
            thr.append(int(min(max(math.floor(F * 4294967296.0), 0.0), 4294967296.0)))
        self.thr = thr if p.jump_law != workloads.JUMP_NONE and p.lam > 0 else []
        self.chunk = max(1, min(p.Nt, (1 << 24) // (self.paths * self.P)))
        self.kept = None

    def draws(self, c):
        """Draws of the steps of chunk c: per step (z0, jump entries or None)."""
        if self.kept is not None and self.kept[0] == c:
            return self.kept[1]
        p, d, P = self.p, self.p.d, self.P
        ks = torch.arange(c * self.chunk, min(p.Nt, (c + 1) * self.chunk), device=self.dev)
        w = _words(ks[:, None], self.m[None, :], 0, p.epoch, p.seed, 1 + 2 * P)
        z0 = _normals(w[1:], d)
        n = torch.zeros_like(w[0])
        for T in self.thr:
            n += w[0] >= T
        step, path = torch.nonzero(n, as_tuple=True)
        n = n[step, path]
        del w
        top = int(n.max()) if n.numel() else 0
        if top:
            th, size, zn = [], [], []
            for i in range(top):
                s = _words(ks[step], self.m[path], (1 << 24) | ((i + 1) << 16), p.epoch, p.seed, 1 + 4 * P)
                th.append(torch.where(i < n, _u01(s[0]), 2.0))
                if p.jump_law == workloads.JUMP_UNIFORM:
                    size.append(torch.stack([2.0 * _u01(v) - 1.0 for v in s[1:1 + 2 * P]][:d], dim=-1))
                else:
                    size.append(_normals(s[1:1 + 2 * P], d))
                zn.append(_normals(s[1 + 2 * P:], d))
            th, order = torch.sort(torch.stack(th, 1), dim=1, stable=True)
            pick = order[:, :, None].expand(-1, -1, d)
            size, zn = torch.stack(size, 1).gather(1, pick), torch.stack(zn, 1).gather(1, pick)
        counts = torch.bincount(step, minlength=ks.numel()).tolist()
        out, at = [], 0
        for j, e in enumerate(counts):
            sel = slice(at, at + e)
            out.append((z0[j], (path[sel], n[sel], th[sel], size[sel], zn[sel]) if e else None))
            at += e
        self.kept = (c, out)
        return out

    def control(self, y, uk):
        """B u for the open-loop control, or the feedback mu^T phi(y); and u itself."""
        if self.fb is None:
            return uk @ self.B.T, None
        fb = self.fb

        def bumps(r, n, half):
            cen = (torch.arange(n, device=self.dev).double() + 0.5) * (2.0 * half / n) - half
            t = 1.0 - (fb.eps * (r[:, None] - cen)) ** 2
            inside = t > 0
            return torch.where(inside, torch.exp(-1.0 / torch.where(inside, t, 1.0)), 0.0)

        u = ((bumps(y[:, 0], fb.nx, fb.x_max) @ uk.view(fb.nx, fb.nv)) * bumps(y[:, 1], fb.nv, fb.v_max)).sum(1)
        return u[:, None] * self.B[:, 0], u

    def substep(self, y, de, z, uk, force, A, sigma):
        bu, u = self.control(y, uk)
        f = y @ A.T + bu
        if self.cubic:
            f = f + (y * y * y) @ self.C.T
        if force is not None:
            f = f + force
        cost = 0.0 if u is None else (0.5 * self.p.nu) * de[:, 0] * u * u
        return y + de * f + sigma * torch.sqrt(de) * z, cost

    def step(self, k, x, uk, draw, A, sigma, scale):
        """(X_{k+1}, summed cost of the step)."""
        z0, jumps = draw
        force = None
        if self.N:
            pos = x[:, 0].view(-1, self.N)
            f = self.fb.omega * (pos.roll(1, 1) + pos.roll(-1, 1)).reshape(-1)
            force = torch.stack([torch.zeros_like(f), f], dim=-1)
            A = A - 2.0 * self.fb.omega * torch.tensor([[0.0, 0.0], [1.0, 0.0]], device=self.dev).double()
        dt = torch.full((1, 1), self.dt, dtype=torch.float64, device=self.dev)
        out, cost = self.substep(x, dt, z0, uk, force, A, sigma)
        fb = self.fb
        if jumps is not None:
            idx, n, th, size, zn = jumps
            d, ks = self.p.d, self.p.jump_law == workloads.JUMP_KS
            gain = torch.ones(d, dtype=torch.float64, device=self.dev)
            moved = torch.ones_like(gain)
            if ks:
                gain[d // 2:] = self.p.jump_gain
                moved[:d // 2] = 0.0
            y, z, fj = x[idx], z0[idx], None if force is None else force[idx]
            prev, total = torch.zeros_like(th[:, :1]), 0.0
            for i in range(th.shape[1]):
                on = (i < n)[:, None]
                t = torch.where(on, th[:, i:i + 1], 1.0)
                yn, c = self.substep(y, torch.where(on, self.dt * (t - prev), self.dt), z, uk, fj, A, sigma)
                y = torch.where(on, gain * yn + moved * scale * size[:, i], y)
                if fb is not None:
                    total = total + torch.where(on[:, 0], c, 0.0)
                prev, z = torch.where(on, t, prev), torch.where(on, zn[:, i], z)
            y, c = self.substep(y, self.dt * (1.0 - prev), z, uk, fj, A, sigma)
            out = out.index_copy(0, idx, y)
            if fb is not None:
                cost = cost.index_copy(0, idx, total + c)
        e = out - self.xd[k + 1]
        if fb is None or fb.track == workloads.TRACK_QUAD:
            run_cost = 0.5 * (self.q * e * e).sum(1)
        elif fb.track == workloads.TRACK_GAUSS:
            run_cost = -torch.exp(-(self.q * e * e).sum(1) / (2.0 * fb.sigma_J ** 2))
        else:
            s = out[:, 0] ** 2 / fb.ax ** 2 + out[:, 1] ** 2 / fb.av ** 2 - 1.0
            run_cost = -torch.exp(-s * s / (2.0 * fb.sigma_J ** 2))
        total = self.dt * run_cost.sum()
        return out, total + (cost.sum() if fb is not None else 0.0)

    def coef(self, theta):
        if theta is None:
            return self.A, self.sigma, self.scale
        rho, s_sigma, s_jump = theta
        dA = torch.as_tensor(self.p.dA, device=self.dev)
        return self.A + (rho - 0.5) * dA, s_sigma.expand(self.p.d), s_jump

    def forward(self, u, keep=False, theta=None):
        x, J, X = self.x0, torch.zeros((), dtype=torch.float64, device=self.dev), []
        with torch.no_grad():
            for k in range(self.p.Nt):
                if keep:
                    X.append(x)
                x, c = self.step(k, x, u[k], self.draws(k // self.chunk)[k % self.chunk], *self.coef(theta))
                J = J + c
        J = J / self.paths
        if self.fb is None:
            J = J + 0.5 * self.p.nu * self.dt * (u * u).sum()
        return J, X

    def gradient(self, u, theta=None):
        J, X = self.forward(u, keep=True, theta=theta)
        g = torch.zeros_like(u)
        th = None if theta is None else [t.detach().requires_grad_(True) for t in theta]
        gth = None if theta is None else [torch.zeros_like(t) for t in theta]
        lam = torch.zeros_like(X[0])
        for k in range(self.p.Nt - 1, -1, -1):
            x, uk = X.pop().detach().requires_grad_(True), u[k].detach().requires_grad_(True)
            draw = self.draws(k // self.chunk)[k % self.chunk]
            with torch.enable_grad():
                out, c = self.step(k, x, uk, draw, *self.coef(th))
                got = torch.autograd.grad((out * lam).sum() + c, [x, uk] + (th or []))
            lam, g[k] = got[0], got[1] / self.paths
            for i in range(len(th or [])):
                gth[i] += got[2 + i] / self.paths
        if self.fb is None:
            g += self.p.nu * self.dt * u
        return J, g, gth

    def optimize(self, u, iters):
        """Projected gradient with the Armijo rule: (u, J of every iterate, last step)."""
        p, zeta, hist = self.p, 1.0, []
        for it in range(iters):
            J, g, _ = self.gradient(u)
            if it == 0:
                hist.append(J.item())
            else:
                zeta = min(2.0 * zeta, 1e3)
            g = g / self.dt
            for _ in range(41):
                v = torch.clamp(u - zeta * g, p.u_min, p.u_max)
                Jv = self.forward(v)[0]
                if Jv <= J + 1e-4 * self.dt * (g * (v - u)).sum():
                    break
                zeta *= 0.5
            u = v
            hist.append(Jv.item())
        return u, np.array(hist), zeta


def exact(case, seed):
    kind = case["kind"]
    if kind == "serving":
        return None
    p, fb = _problem(case, seed)
    # sums of a dozen torch operations per step: the largest sizes stay within some seconds
    if kind == "optimize" and (p.Nt * case["iters"] > 2500 or p.M * p.Nt * case["iters"] > 600e6):
        return None
    e = _Exact(p, fb)
    if kind == "feedback":
        J, g, _ = e.gradient(torch.from_numpy(workloads.random_mu(p, fb, seed=seed, scale=0.3)).cuda())
        return {"J": J, "grad": g}
    u = torch.from_numpy(workloads.random_control(p, seed=seed, scale=0.5)).cuda()
    if kind == "gradient":
        J, g, _ = e.gradient(u)
        return {"J": J, "grad": g}
    if kind == "autograd":
        theta = [torch.tensor(v, dtype=torch.float64, device="cuda") for v in (0.5, 0.3, 0.2)]
        J, g, gth = e.gradient(u, theta)
        return {"J": J, "grad_u": g, "grad_theta": torch.stack(gth)}
    u, hist, zeta = e.optimize(u, case["iters"])
    return {"u": u, "J": hist, "zeta": zeta, "iters": None}
