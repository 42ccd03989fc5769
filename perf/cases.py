"""The work a user of the library has it do, as timed cases.

Four kinds of call, each through the package's public entry points:
    step     a time-stepping run: ``Solver.set_state``, ``Solver.step`` per step, ``Solver.stress``
    coupled  the velocity and the stress in turn: ``Solver.stress``, ``NSSolver.step``, ``Solver.step`` per step
    implicit a run with the transport inside the global solve (above the explicit Courant limit)
    train    ``fractional_stress`` forward and its gradients in sigma0, grad_u, Wi and beta

``listed()`` names the cases, ``draw(rng)`` gives further ones of the same
ranges, ``prepare`` / ``run`` execute one, ``work`` counts what one pass cannot
do without and ``exact`` restates the scheme in plain FP64 torch: the memory
term is evaluated as the full history sum with scalar weights instead of m
modes per point (the same numbers, since the modes start at zero and obey a
linear recurrence with constant coefficients).
"""
from __future__ import annotations

import math

import numpy as np
import torch

B0, B1, B2 = 1.5, -2.0, 0.5                      # BDF2
PAIRS = {2: ((0, 0), (0, 1), (1, 1)), 3: ((0, 0), (1, 1), (2, 2), (1, 2), (0, 2), (0, 1))}
FP64, FP32, FP32_PLAIN = 0, 1, 2
# mode updates of the largest listed case, FP64 ones counted with their lower rate
BUDGET = 3.3e10


def _case(kind, n, precision, m, alpha, dt, steps, **kw):
    case = dict(kind=kind, dim=len(n), precision=precision, m=m, alpha=alpha, dt=dt, steps=steps, horizon=200,
                Wi=1.0, beta=0.5, transport="none", form="stress", stencil=0, diffusion=False, sigma0=True, K=50)
    for a, k in enumerate(n):
        case[f"n{a}"] = k
    case.update(kw)
    return case


def listed():
    return [
        # the small development run: Taylor-Green-sized grid in FP64, a hundred steps (launches and host time count)
        _case("step", (64, 64), FP64, 16, 0.5, 1e-3, 100, transport="explicit", name="step_2d_64_fp64"),
        # the 2D production grid in the FP32 storage form, with transport
        _case("step", (1024, 1024), FP32, 32, 0.5, 5e-4, 20, transport="explicit", sigma0=False,
              name="step_2d_1024_fp32"),
        # the same grid in the FP64 form it is validated against, pointwise law
        _case("step", (1024, 1024), FP64, 32, 0.8, 5e-4, 10, name="step_2d_1024_fp64"),
        # the headline: 3D 256^3 with transport, FP32 modes and compensated sum
        _case("step", (256, 256, 256), FP32, 32, 0.6, 2e-4, 10, transport="explicit", Wi=2.0, beta=0.9,
              sigma0=False, name="step_3d_256_fp32"),
        # a box whose sides fit no tile, central stencil and diffusion
        _case("step", (97, 61, 53), FP32, 16, 0.5, 5e-4, 30, transport="explicit", stencil=1, diffusion=True,
              name="step_3d_ragged_fp32"),
        # precision study: most modes, FP64, 3D
        _case("step", (160, 160, 160), FP64, 48, 0.9, 2e-4, 3, Wi=2.0, beta=0.9, name="step_3d_160_fp64_m48"),
        # the paper's own variable in 3D
        _case("step", (192, 192, 192), FP32, 32, 0.6, 2e-4, 8, form="paper", Wi=2.0, beta=0.9,
              name="paper_3d_192_fp32"),
        # unit-RMS velocity on the 2D production grid: transport has to be implicit
        _case("implicit", (1024, 1024), FP32, 32, 0.5, 5e-4, 2, transport="implicit", sigma0=False,
              name="implicit_2d_1024_fp32"),
        # flow and stress together
        _case("coupled", (1024, 1024), FP32, 32, 0.5, 5e-4, 10, transport="explicit", Wi=2.0, beta=0.9,
              sigma0=False, name="coupled_2d_1024_fp32"),
        # parameter and field fitting, FP32 storage, checkpoint every 50 steps
        _case("train", (512, 512), FP32, 32, 0.5, 5e-4, 100, name="train_2d_512_fp32"),
        # the same in FP64 on a smaller ragged grid (gradient checks, small inverse problems)
        _case("train", (250, 198), FP64, 32, 0.5, 5e-4, 60, K=20, name="train_2d_250x198_fp64"),
        # fitting with the stress carried along by the flow, 3D
        _case("train", (64, 64, 64), FP32, 24, 0.6, 5e-4, 40, K=20, transport="explicit",
              name="train_3d_64_fp32_transport"),
    ]


def draw(rng):
    kind = rng.choice(["step"] * 6 + ["train"] * 3 + ["coupled", "implicit"])
    alpha = rng.choice([0.3, 0.5, 0.6, 0.8, 0.9])
    dt = rng.choice([2e-4, 5e-4, 1e-3])
    m = rng.choice([8, 16, 24, 32, 48])

    def side(lo, hi, ragged):
        k = int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))
        return k if ragged else max(32, 32 * ((k + 16) // 32))

    ragged = rng.random() < 0.5
    if kind == "coupled":
        n = (2 ** rng.randint(6, 10), 2 ** rng.randint(6, 10))
        return _case(kind, n, rng.choice([FP64, FP32, FP32]), min(m, 32), 0.5, 5e-4, rng.randint(3, 10),
                     transport="explicit", Wi=2.0, beta=0.9, sigma0=False)
    if kind == "implicit":
        n = tuple(side(96, 900, ragged) for _ in range(2))
        return _case(kind, n, rng.choice([FP64, FP32, FP32]), min(m, 32), 0.5, 5e-4, 2, transport="implicit",
                     sigma0=False)
    dim = rng.choice([2, 2, 3]) if kind == "train" else rng.choice([2, 3])
    precision = rng.choice([FP64, FP32, FP32] if kind == "train" else [FP64, FP32, FP32, FP32_PLAIN])
    transport = rng.choice(["none", "explicit"])
    form = "stress"
    if rng.random() < 0.2:
        form, transport = "paper", "none"
    if kind == "step" and rng.random() < 0.1:
        alpha, m, form = 1.0, 0, "stress"
    lo, hi = ((48, 1400) if kind == "step" else (32, 600)) if dim == 2 else ((16, 240) if kind == "step" else (12, 80))
    n = tuple(side(lo, hi, ragged) for _ in range(dim))
    N, nc = int(np.prod(n)), len(PAIRS[dim])
    rate = 7.0 if precision == FP64 else 1.0
    passes = 4.0 if kind == "train" else 1.0
    top = 100 if kind == "step" else 60
    cost = N * nc * max(m, 4) * rate * passes
    while cost * 2 > BUDGET:
        n = tuple(max(16, k - (1 if ragged else 32)) for k in n)
        N = int(np.prod(n))
        cost = N * nc * max(m, 4) * rate * passes
    steps = max(2, min(int(BUDGET / cost), int(round(math.exp(rng.uniform(math.log(2), math.log(top)))))))
    stencil = rng.choice([0, 0, 1])
    return _case(kind, n, precision, m, alpha, dt, steps, transport=transport, form=form, stencil=stencil,
                 diffusion=transport == "explicit" and rng.random() < 0.3, K=rng.choice([10, 20, 50]),
                 sigma0=rng.random() < 0.7, Wi=rng.choice([1.0, 2.0]), beta=rng.choice([0.5, 0.9]))


# ------------------------------------------------------------------ inputs
def _grid(case):
    return tuple(int(case[f"n{a}"]) for a in range(case["dim"]))


def _device():
    return torch.device("cuda", torch.cuda.current_device()) if torch.cuda.is_available() else torch.device("cpu")


def _soe(case):
    """Positive exponential table: the kernel's Laplace integral by the trapezoidal
    rule in log mu, the lowest node taking the tail below, and a last term that
    carries the kernel's missing mass near t = 0."""
    if case["alpha"] == 1.0:
        return None, None
    alpha = 1.0 - case["alpha"] if case["form"] == "paper" else case["alpha"]
    dt, T, k = case["dt"], case["horizon"] * case["dt"], case["m"] - 1
    lo, hi = math.log(0.02 / T), math.log(20.0 / dt)
    h = (hi - lo) / (k - 1)
    s = math.sin(math.pi * alpha) / math.pi
    mu = np.exp(lo + h * np.arange(k))
    w = h * s * mu ** alpha
    w[0] += s * math.exp(alpha * (lo - h / 2)) / alpha
    missing = T ** (1.0 - alpha) / math.gamma(2.0 - alpha) - float(np.sum(w * -np.expm1(-mu * T) / mu))
    fast = 1e12 / dt
    return np.append(mu, fast), np.append(w, max(missing, 0.0) * fast)


def _velocity(n, gen, dev):
    """Divergence-free random velocity with a k^-5/3 spectrum at unit RMS and its gradient, FP64."""
    dim = len(n)
    kmax = min(32 if dim == 2 else 24, min(n) // 3)
    shape = n[::-1]                                               # x fastest
    axes = [torch.fft.fftfreq(k, 1.0 / k, dtype=torch.float64, device=dev) for k in shape]
    kv = torch.meshgrid(*axes, indexing="ij")[::-1]               # kx, ky(, kz)
    kk = sum(k * k for k in kv).sqrt()
    safe = torch.where(kk > 0, kk, torch.ones_like(kk))
    amp = torch.where((kk > 0) & (kk <= kmax), safe ** (-5.0 / 6.0 - 0.5 * (dim - 1)), torch.zeros_like(kk))
    uh = [amp * torch.fft.fftn(torch.randn(shape, generator=gen, device=dev, dtype=torch.float64))
          for _ in range(dim)]
    kdu = sum(kv[a] * uh[a] for a in range(dim)) / safe ** 2
    uh = [uh[a] - kv[a] * kdu for a in range(dim)]
    u = torch.stack([torch.fft.ifftn(f).real.reshape(-1) for f in uh])
    kap = torch.stack([torch.fft.ifftn(1j * kv[j] * uh[i]).real.reshape(-1) for i in range(dim) for j in range(dim)])
    scale = 1.0 / float((u * u).sum(0).mean().sqrt())
    return u * scale, kap * scale


def _smooth(n, rows, gen, dev, amplitude):
    """A constant and three low Fourier modes per row, FP64."""
    xs = torch.meshgrid(*[torch.arange(k, dtype=torch.float64, device=dev) * (2 * math.pi / k) for k in n[::-1]],
                        indexing="ij")[::-1]
    r = torch.randn(rows, 3, 3 + len(n), generator=gen, device=dev, dtype=torch.float64).cpu().tolist()
    out = []
    for c in range(rows):
        f = torch.full_like(xs[0], r[c][0][0])
        for mode in r[c]:
            f = f + 0.3 * mode[1] * torch.cos(sum(round(mode[3 + a]) * xs[a] for a in range(len(n))) + 3 * mode[2])
        out.append(amplitude * f.reshape(-1))
    return torch.stack(out)


def _inputs(case, seed):
    dev, n, dim = _device(), _grid(case), case["dim"]
    gen = torch.Generator(device=dev).manual_seed(int(seed))
    dtype = torch.float64 if case["precision"] == FP64 else torch.float32
    nc = len(PAIRS[dim])
    mu, w = _soe(case)
    dt = case["dt"]
    eta = B0 if mu is None else float(np.sum(B0 * w * dt / (B0 + mu * dt)))
    inv_h = [k / (2 * math.pi) for k in n]
    u, kap = _velocity(n, gen, dev)
    if case["transport"] == "explicit":
        # about a third of the explicit transport's limit, dt sum |u_a|/h_a ~ 0.3 eta (0.27 for alpha = 1)
        top = 0.1 * min(eta, 1.0)
        f = top / (dt * float((u.abs() * torch.tensor(inv_h, device=dev, dtype=torch.float64)[:, None]).sum(0).max()))
        u, kap = u * f, kap * f
        kap = kap * min(1.0, 0.1 * eta / (dt * float(kap.abs().max())))
    elif case["transport"] == "none":
        kap = kap * min(0.1, 0.1 * eta / (dt * float(kap.abs().max())))
    eps = 0.02 * min(eta, 1.0) / (dt * sum(h * h for h in inv_h)) if case["diffusion"] else 0.0
    inp = dict(mu=mu, w=w, eps=eps, u=u.to(dtype), kap=kap.to(dtype), kap_prev=(0.98 * kap).to(dtype), sigma0=None)
    if case["sigma0"] or case["kind"] == "train":
        inp["sigma0"] = _smooth(n, nc, gen, dev, 0.1).to(dtype)
    if case["kind"] == "train":
        inp["target"] = _smooth(n, nc, gen, dev, 0.1).to(dtype)
    return inp


# ------------------------------------------------------------- the library
def prepare(case, seed):
    from paper_2411_17294_gb300 import tfs
    inp = _inputs(case, seed)
    n, dim = _grid(case), case["dim"]
    state = dict(case=case, **inp)
    if case["kind"] == "train":
        state["sigma0"] = inp["sigma0"].requires_grad_(True)
        state["kap"] = inp["kap"].requires_grad_(True)
        state["Wi"] = torch.tensor(case["Wi"], dtype=torch.float64, requires_grad=True)
        state["beta"] = torch.tensor(case["beta"], dtype=torch.float64, requires_grad=True)
        return state
    transport = {"none": False, "explicit": True, "implicit": "implicit"}[case["transport"]]
    state["solver"] = tfs.Solver(dim, n, case["alpha"], case["Wi"], case["beta"], case["dt"],
                                 m=0 if inp["mu"] is None else case["m"], precision=case["precision"], mu=inp["mu"],
                                 w=inp["w"], transport=transport, eps=inp["eps"], stencil=case["stencil"],
                                 form=case["form"])
    if case["kind"] == "coupled":
        state["ns"] = tfs.NSSolver(n, (2 * math.pi, 2 * math.pi), case["beta"], 100.0, case["dt"],
                                   precision=case["precision"])
    return state


def run(state):
    case = state["case"]
    if case["kind"] == "train":
        from paper_2411_17294_gb300.autograd import fractional_stress
        leaves = (state["sigma0"], state["kap"], state["Wi"], state["beta"])
        moving = case["transport"] == "explicit"
        out = fractional_stress(*leaves, dim=case["dim"], n=_grid(case), alpha=case["alpha"], dt=case["dt"],
                                steps=case["steps"], K=case["K"], mu=state["mu"], w=state["w"],
                                u=state["u"] if moving else None, precision=case["precision"], eps=state["eps"],
                                stencil=case["stencil"], form=case["form"])
        loss = ((out - state["target"]) ** 2).sum()
        return (out.detach(),) + torch.autograd.grad(loss, leaves)
    s = state["solver"]
    s.set_state(state["sigma0"])
    if case["kind"] == "coupled":
        ns = state["ns"]
        ns.set_state(state["u"])
        for _ in range(case["steps"]):
            u, kap = ns.step(s.stress())
            s.step(kap, kap, u)
        return u, kap, s.stress()
    u = None if case["transport"] == "none" else state["u"]
    for _ in range(case["steps"]):
        s.step(state["kap"], state["kap_prev"], u)
    return s.stress()


def work(case):
    """Stepping: the state does not stay on the chip between calls, so each step reads both levels of
    every mode and of the stress and writes the new ones, and reads its inputs.  Training is one call:
    its inputs and results."""
    dim, steps, m = case["dim"], case["steps"], case["m"]
    N, nc = float(np.prod(_grid(case))), len(PAIRS[dim])
    s = 8 if case["precision"] == FP64 else 4
    solve = 2 * nc ** 3 / 3 + 2 * nc ** 2
    flops = N * (8 * m * nc + solve + 10 * nc)
    if case["kind"] == "train":
        return {"bytes": N * s * (2 * nc + dim * dim + nc) + N * s * (nc + dim * dim), "flops": 2 * steps * flops}
    words = 3 * m * nc + 3 * nc + 2 * dim * dim
    if case["transport"] != "none":
        words += dim
        flops += N * nc * 8 * dim
    if case["sigma0"]:
        words += nc
    nbytes = N * s * words
    if case["kind"] == "coupled":
        # velocity, gradient and stress exchanged; FP64 spectra: two levels of u and of its explicit terms
        nbytes += N * (s * (2 + 4 + 3) + 16 * (2 * 2 + 2 * 2))
        flops += N * (9 * 2.5 * math.log2(N) + 60)
    return {"bytes": steps * nbytes, "flops": steps * flops}


# ------------------------------------------- the same numbers in plain FP64
def _shift(f, n, axis, k):
    """f [..., N] at offset k along an axis, periodic."""
    g = f.reshape(f.shape[:-1] + n[::-1])
    return torch.roll(g, -k, dims=g.dim() - 1 - axis).reshape(f.shape)


def _transport(case, inp, E):
    """u . grad E - eps Lap E."""
    n, u = _grid(case), inp["u"].double()
    out = torch.zeros_like(E)
    for a in range(case["dim"]):
        h = 2 * math.pi / n[a]
        f = {k: _shift(E, n, a, k) for k in (-2, -1, 1, 2)}
        if case["stencil"] == 1:
            d = (f[1] - f[-1]) / (2 * h)
        else:
            d = torch.where(u[a] >= 0, f[-2] - 6 * f[-1] + 3 * E + 2 * f[1], -2 * f[-1] - 3 * E + 6 * f[1] - f[2]) / (6 * h)
        out = out + u[a] * d
        if inp["eps"]:
            out = out - inp["eps"] * (f[-1] - 2 * E + f[1]) / h ** 2
    return out


def _upper(K, s, dim):
    """kappa S + S kappa^T of packed components, kappa [d*d][N]."""
    P = PAIRS[dim]
    at = {}
    for c, (i, j) in enumerate(P):
        at[i, j] = at[j, i] = c
    return torch.stack([sum(K[i * dim + l] * s[at[l, j]] + K[j * dim + l] * s[at[i, l]] for l in range(dim))
                        for i, j in P])


def _sym(K, dim):
    return torch.stack([K[i * dim + j] + K[j * dim + i] for i, j in PAIRS[dim]])


class _Law:
    """One run of the stress law from zero modes, the memory as a history sum."""

    def __init__(self, case, inp, Wi, beta):
        self.case, self.inp, self.Wi, self.beta = case, inp, Wi, beta
        self.dim, self.dt, self.alpha = case["dim"], case["dt"], case["alpha"]
        self.paper, self.classic = case["form"] == "paper", case["alpha"] == 1.0
        self.G = (1.0 - beta) / Wi
        dt = self.dt
        if self.classic:
            self.eta = B0
        else:
            mu, w = inp["mu"], inp["w"]
            c = 1.0 / (B0 + mu * dt)
            g = [np.ones_like(c)]                                    # response of a mode to a unit drive
            for _ in range(case["steps"]):
                g.append(-c * (B1 * g[-1] + B2 * (g[-2] if len(g) > 1 else 0.0)))
            tail = [B1 * g[k] + (B2 * g[k - 1] if k > 0 else 0.0) for k in range(case["steps"])]
            drive = dt * c if self.paper else w * dt * c
            read = w * mu * c if self.paper else mu * dt * c
            self.weight = [float(np.sum(read * t * drive)) for t in tail]   # lag 1, 2, ...
            self.eta = float(np.sum(B0 * w * c)) if self.paper else float(np.sum(B0 * w * dt * c))
        s0 = inp["sigma0"]
        N = int(np.prod(_grid(case)))
        self.s0 = s0.double() if s0 is not None else torch.zeros((len(PAIRS[self.dim]), N), dtype=torch.float64,
                                                                 device=inp["kap"].device)
        self.cur, self.prev = self.s0, self.s0
        self.hist, self.index, self.inverse = [], 0, None
        self.psi, self.psi_prev = torch.zeros_like(self.s0), torch.zeros_like(self.s0)

    def system(self, K):
        a, scale = (B0 + self.dt * self.eta / self.Wi, self.dt * self.eta) if self.paper else \
            (self.eta + self.dt / self.Wi, self.dt)
        nc = len(PAIRS[self.dim])
        cols = []
        for k in range(nc):
            e = torch.zeros((nc, K.shape[1]), dtype=torch.float64, device=K.device)
            e[k] = 1.0
            cols.append(a * e - scale * _upper(K, e, self.dim))
        return torch.stack(cols, dim=1)                              # [row][column][N]

    def solve(self, M, R):
        if self.inverse is None:
            Mt = M.detach().permute(2, 0, 1)
            self.inverse = torch.cat([torch.linalg.inv(b) for b in Mt.split(1 << 19)]).permute(1, 2, 0).contiguous()
        mul = lambda A, x: torch.stack([sum(A[i, j] * x[j] for j in range(x.shape[0])) for i in range(x.shape[0])])
        x = mul(self.inverse, R.detach())
        x = x + mul(self.inverse, R.detach() - mul(M.detach(), x))
        if not (M.requires_grad or R.requires_grad):
            return x
        return _Solve.apply(M, R, x, self.inverse)

    def memory(self):
        if not self.hist:
            return torch.zeros_like(self.s0)
        k = len(self.hist)
        return sum(self.weight[k - 1 - i] * self.hist[i] for i in range(k))

    def step(self, K, M=None, keep=True):
        dt, Wi = self.dt, self.Wi
        if M is None:
            M = self.system(K)
            self.inverse = None if not keep else self.inverse
        t = (self.index + 1) * dt
        src = dt * self.G * _sym(K, self.dim)
        moving = self.case["transport"] == "explicit"
        if self.paper:
            k = self.index
            psi0 = self.eta + sum(self.weight[k - 1 - i] for i in range(k))
            h = self.memory()
            R = -B1 * self.cur - B2 * self.prev + dt * (_upper(K, h, self.dim) - h / Wi) + src * psi0
            if moving:
                R = R - dt * _transport(self.case, self.inp, 2 * self.psi - self.psi_prev)
        else:
            if self.classic:
                R, g = -B1 * self.cur - B2 * self.prev, 1.0
            else:
                R, g = self.eta * self.s0 - self.memory(), t ** (self.alpha - 1.0) / math.gamma(self.alpha)
            R = R + src * g
            if moving:
                R = R - dt * _transport(self.case, self.inp, 2 * self.cur - self.prev)
        new = self.implicit(M, R) if self.case["transport"] == "implicit" else self.solve(M, R)
        if self.paper:
            self.psi_prev, self.psi = self.psi, self.eta * new + h
        self.hist.append(new if self.paper else new - self.s0)
        self.prev, self.cur, self.index = self.cur, new, self.index + 1
        return self.stress()

    def stress(self):
        return self.psi if self.paper else self.cur

    def implicit(self, M, R):
        """BiCGStab on the global system, right-preconditioned by the point blocks."""
        mul = lambda A, x: torch.stack([sum(A[i, j] * x[j] for j in range(x.shape[0])) for i in range(x.shape[0])])
        if self.inverse is None:
            h = [2 * math.pi / k for k in _grid(self.case)]
            lead = 3.0 / 6.0 if self.case["stencil"] == 0 else 0.0
            diag = sum(self.dt * lead * self.inp["u"][a].double().abs() / h[a] for a in range(self.dim))
            blocks = M.permute(2, 0, 1) + diag[:, None, None] * torch.eye(M.shape[0], dtype=M.dtype, device=M.device)
            self.inverse = torch.cat([torch.linalg.inv(b) for b in blocks.split(1 << 19)]).permute(1, 2, 0).contiguous()
        op = lambda x: mul(M, x) + self.dt * _transport(self.case, self.inp, x)
        x = 2 * self.cur - self.prev
        goal = 1e-13 * float(R.norm())
        for _ in range(6):                                           # restarts from the true residual
            r = R - op(x)
            if float(r.norm()) <= goal:
                break
            r0, p = r.clone(), r.clone()
            rho = torch.dot(r0.flatten(), r.flatten())
            for it in range(3000):
                y = mul(self.inverse, p)
                v = op(y)
                al = rho / torch.dot(r0.flatten(), v.flatten())
                s = r - al * v
                z = mul(self.inverse, s)
                q = op(z)
                om = torch.dot(q.flatten(), s.flatten()) / torch.dot(q.flatten(), q.flatten())
                x = x + al * y + om * z
                r = s - om * q
                if it % 16 == 15 and not float(r.norm()) > 0.3 * goal:
                    break
                new = torch.dot(r0.flatten(), r.flatten())
                p = r + (new / rho) * (al / om) * (p - om * v)
                rho = new
        return x


class _Solve(torch.autograd.Function):
    """x = M^-1 R with the solution in hand; the adjoint solves the transposed systems."""

    @staticmethod
    def forward(ctx, M, R, x, inverse):
        ctx.save_for_backward(M.detach(), x, inverse)
        return x.clone()

    @staticmethod
    def backward(ctx, g):
        M, x, inv = ctx.saved_tensors
        nc = x.shape[0]
        mulT = lambda A, v: torch.stack([sum(A[i, j] * v[i] for i in range(nc)) for j in range(nc)])
        lam = mulT(inv, g)
        lam = lam + mulT(inv, g - mulT(M, lam))
        gM = -torch.stack([torch.stack([lam[i] * x[j] for j in range(nc)]) for i in range(nc)])
        return gM, lam, None, None


class _Flow:
    """The projection step on the periodic square with spectral derivatives."""

    def __init__(self, n, nu, dt, u0):
        self.n, self.nu, self.dt = n, nu, dt
        d = []
        for k in n:
            f = torch.fft.fftfreq(k, 1.0 / k, dtype=torch.float64, device=u0.device)
            f[k // 2] = 0.0
            d.append(f)
        self.kx, self.ky = d[0][None, :].expand(n[1], n[0]), d[1][:, None].expand(n[1], n[0])
        self.k2 = self.kx ** 2 + self.ky ** 2
        self.safe = torch.where(self.k2 > 0, self.k2, torch.ones_like(self.k2))
        self.uh = self.project(*[self.hat(u0[a]) for a in range(2)])
        self.uh_prev, self.f_prev = self.uh, None

    def hat(self, f):
        return torch.fft.fft2(f.reshape(self.n[1], self.n[0]))

    def real(self, f):
        return torch.fft.ifft2(f).real.reshape(-1)

    def project(self, a, b):
        q = (self.kx * a + self.ky * b) / self.safe
        return a - self.kx * q, b - self.ky * q

    def fields(self):
        a, b = self.uh
        u = torch.stack([self.real(a), self.real(b)])
        kap = torch.stack([self.real(1j * k * f) for f in (a, b) for k in (self.kx, self.ky)])
        return u, kap

    def step(self, s):
        u, k = self.fields()
        sx, sm, sy = [self.hat(s[c]) for c in range(3)]
        f = (1j * (self.kx * sx + self.ky * sm) - self.hat(u[0] * k[0] + u[1] * k[1]),
             1j * (self.kx * sm + self.ky * sy) - self.hat(u[0] * k[2] + u[1] * k[3]))
        old = f if self.f_prev is None else self.f_prev
        r = [2 * f[a] - old[a] - (B1 * self.uh[a] + B2 * self.uh_prev[a]) / self.dt for a in range(2)]
        new = [v / (B0 / self.dt + self.nu * self.k2) for v in self.project(*r)]
        self.f_prev, self.uh_prev, self.uh = f, self.uh, tuple(new)
        return self.fields()


def exact(case, seed):
    inp = _inputs(case, seed)
    if case["kind"] == "train":
        inp["sigma0"] = inp["sigma0"].double().requires_grad_(True)
        kap = inp["kap"].double().requires_grad_(True)
        Wi = torch.tensor(case["Wi"], dtype=torch.float64, device=kap.device, requires_grad=True)
        beta = torch.tensor(case["beta"], dtype=torch.float64, device=kap.device, requires_grad=True)
        law = _Law(case, inp, Wi, beta)
        M = law.system(kap)
        for _ in range(case["steps"]):
            out = law.step(kap, M)
        loss = ((out - inp["target"].double()) ** 2).sum()
        grads = torch.autograd.grad(loss, (inp["sigma0"], kap, Wi, beta))
        return (out.detach(), grads[0], grads[1], grads[2].cpu(), grads[3].cpu())
    law = _Law(case, inp, case["Wi"], case["beta"])
    if case["kind"] == "coupled":
        flow = _Flow(_grid(case), case["beta"] / 100.0, case["dt"], inp["u"].double())
        for _ in range(case["steps"]):
            u, kap = flow.step(law.stress())
            inp["u"] = u
            law.step(kap, keep=False)
        return u, kap, law.stress()
    K = 2.0 * inp["kap"].double() - inp["kap_prev"].double()
    M = law.system(K)
    for _ in range(case["steps"]):
        law.step(K, M)
    return law.stress()
