"""The work a user of this package has it do, as measured cases.

A program makes a solver for its grid once (``prepare``) and then calls it many
times (``run``): single transforms and operators, elliptic solves, right-hand
sides, whole stretches of RK4 steps, an ensemble, and the training and the use
of the learned start's network. Sizes are those of the package's workloads (the
256x16 soliton, the 1024x256 transverse-stability grid, the ensemble's uneven
grids, the 2048^2 localized hump, the 128^2 coarse network).
"""
import math

import numpy as np
import torch

from paper_2306_09731_gb300 import sgn as S
from paper_2306_09731_gb300 import unet as U

DEV = "cuda"
F64 = torch.float64
# the four-level network of 471,873 parameters and the library's default one
ARCHS = {"spec": (4, (32, 64, 64, 96)), "default": (3, (16, 32, 32))}


def listed():
    return [
        # the smallest call: L[sigma] without a handle on the soliton's grid,
        # for a host program that cannot allocate
        dict(name="noalloc_256x16", kind="noalloc", Nx=256, Ny=16, Lx=80.0, Ly=10.0),
        # a spectrum and the field back from it (post-processing, filters)
        dict(name="fft2_1024x256", kind="fft2", Nx=1024, Ny=256, Lx=120.0, Ly=30.0),
        # the gradient of a large field (u = v - grad(sigma)/h, vorticity checks)
        dict(name="gradient_2048", kind="gradient", Nx=2048, Ny=2048, Lx=100.0, Ly=100.0),
        # one application of the elliptic operator in double-float
        dict(name="elliptic_1024x512_p2", kind="elliptic", Nx=1024, Ny=512, Lx=120.0, Ly=60.0, precision=2),
        # one elliptic solve from a zero start, mixed precision, large grid
        dict(name="solve_2048_p2", kind="solve", Nx=2048, Ny=2048, Lx=100.0, Ly=100.0, precision=2),
        # one right-hand side for a caller's own time stepper, accurate mode
        dict(name="rhs_1024x256_p3", kind="rhs", Nx=1024, Ny=256, Lx=120.0, Ly=30.0, precision=3),
        # the line soliton with the paper's method: small grid, many launches
        dict(name="rk4_256x16_p0", kind="rk4", Nx=256, Ny=16, Lx=80.0, Ly=10.0, precision=0, guess=0, graph=0,
             steps=5, dt=5e-3),
        # transverse stability with the paper's method
        dict(name="rk4_1024x256_p0", kind="rk4", Nx=1024, Ny=256, Lx=120.0, Ly=30.0, precision=0, guess=0, graph=0,
             steps=3, dt=2e-3),
        # the localized hump in mixed precision, polynomial start, step graphs
        dict(name="rk4_2048_p2", kind="rk4", Nx=2048, Ny=2048, Lx=100.0, Ly=100.0, precision=2, guess=3, graph=1,
             steps=10, dt=1e-3),
        # perturbed solitons on uneven grids, stepped together
        dict(name="ensemble_12", kind="ensemble", members=12, precision=2, guess=3, graph=1, steps=8, dt=2e-3),
        # training the learned start: loss and gradients of one batch
        dict(name="train_128_b8", kind="train", n=128, batch=8, arch="spec"),
        # using it: one sample per corrected stage
        dict(name="infer_128_b1", kind="infer", n=128, batch=1, arch="spec"),
    ]


def _pow2(rng, lo, hi):
    return 1 << rng.randint(lo, hi)


def _grid(rng, lo, hi, most):
    """Sides 2^lo..2^hi with at most 2^most points."""
    while True:
        a, b = rng.randint(lo, hi), rng.randint(lo, hi)
        if a + b <= most:
            break
    # grid spacings of the package's workloads (~0.05 to 0.3 depths)
    return dict(Nx=1 << a, Ny=1 << b, Lx=(1 << a) * rng.uniform(0.05, 0.3), Ly=(1 << b) * rng.uniform(0.05, 0.3))


def draw(rng):
    kind = rng.choice(["noalloc", "fft2", "gradient", "elliptic", "solve", "rhs", "rk4", "rk4", "ensemble", "train",
                       "infer"])
    if kind == "noalloc":
        return dict(kind=kind, **_grid(rng, 4, 12, 16))
    if kind in ("fft2", "gradient"):
        return dict(kind=kind, **_grid(rng, 4, 12, 22))
    if kind == "elliptic":
        return dict(kind=kind, precision=rng.choice([0, 1, 2, 3]), **_grid(rng, 4, 12, 22))
    if kind == "solve":
        return dict(kind=kind, precision=rng.choice([0, 1, 2, 3]), **_grid(rng, 4, 11, 20))
    if kind == "rhs":
        return dict(kind=kind, precision=rng.choice([0, 1, 2, 3]), **_grid(rng, 4, 11, 20))
    if kind == "rk4":
        p = rng.choice([0, 2, 3])
        return dict(kind=kind, precision=p, guess=rng.choice([0, 2, 3]), graph=rng.choice([0, 1]),
                    steps=rng.randint(1, 6), dt=10 ** rng.uniform(-3.3, -2.3), **_grid(rng, 4, 10, 16 if p == 0 else 19))
    if kind == "ensemble":
        return dict(kind=kind, members=rng.randint(2, 16), precision=rng.choice([0, 2]), guess=rng.choice([2, 3]),
                    graph=1, steps=rng.randint(1, 4), dt=2e-3)
    n = _pow2(rng, 5, 8)
    return dict(kind=kind, n=n, batch=rng.randint(1, min(16, (1 << 17) // (n * n))), arch=rng.choice(["spec", "default"]))


# ------------------------------------------------------------------- inputs

def _rng(seed, *salt):
    return np.random.default_rng([int(seed) & 0x7fffffff, *salt])


def _axes(c):
    x = -0.5 * c["Lx"] + c["Lx"] * torch.arange(c["Nx"], dtype=F64, device=DEV) / c["Nx"]
    y = -0.5 * c["Ly"] + c["Ly"] * torch.arange(c["Ny"], dtype=F64, device=DEV) / c["Ny"]
    return x, y


def _band(c, r, amp, kx=6, ky=6):
    """A smooth periodic field: random modes |m| <= k with amplitudes amp/(1+|m|^2)."""
    x, y = _axes(c)
    mx = torch.arange(0, min(kx, c["Nx"] // 2 - 1) + 1, device=DEV)
    k = min(ky, c["Ny"] // 2 - 1)
    my = torch.arange(-k, k + 1, device=DEV)
    C = r.standard_normal((len(my), len(mx))) + 1j * r.standard_normal((len(my), len(mx)))
    C = torch.tensor(C, device=DEV) * amp / (1.0 + (my[:, None] ** 2 + mx[None, :] ** 2).to(F64))
    C[k, 0] = 0.0
    two_pi = 2.0 * math.pi
    ex = torch.exp(1j * two_pi * (mx[None, :] * (x[:, None] / c["Lx"])))
    ey = torch.exp(1j * two_pi * (my[None, :] * (y[:, None] / c["Ly"])))
    return (ey @ C @ ex.T).real.contiguous()


def _state(c, seed):
    """A depth and a curl-free velocity: a perturbed line solitary wave where the
    box is a channel long enough for its tails, else a localized hump."""
    r = _rng(seed, 1)
    x, y = _axes(c)
    X, Y = x[None, :], y[:, None]
    a = float(r.uniform(0.2, 0.8))
    if c["Lx"] >= 40.0 and c["Lx"] > 2.0 * c["Ly"]:
        kap = math.sqrt(3.0 * a / (4.0 * (1.0 + a)))
        cc = math.sqrt(1.0 + a)
        T = torch.tanh(kap * X)
        s = 1.0 - T * T
        h0 = 1.0 + a * s
        h1, h2 = a * (-2.0 * kap * s * T), a * kap * kap * (4.0 * s - 6.0 * s * s)
        v = cc - cc / h0 * (1.0 + (2.0 * (h1 * h1 + h0 * h2)) / 6.0)
        phi = float(r.uniform(0.0, 2.0 * math.pi))
        h = h0 + 1e-2 * torch.exp(-X * X) * torch.cos(2.0 * math.pi * Y / c["Ly"] + phi)
        vx, vy = v.expand(c["Ny"], c["Nx"]).contiguous(), torch.zeros((c["Ny"], c["Nx"]), dtype=F64, device=DEV)
    else:
        # centre and width in units of the smaller period, so that every grid resolves it
        w = min(c["Lx"], c["Ly"]) / float(r.uniform(9.0, 14.0))
        x0, y0 = (float(r.uniform(-0.1, 0.1)) * c[k] for k in ("Lx", "Ly"))
        g = torch.exp(-((X - x0) ** 2 + (Y - y0) ** 2) / (w * w))
        h = 1.0 + a * g
        b = float(r.uniform(0.05, 0.15)) * w
        vx, vy = -2.0 * b * (X - x0) / (w * w) * g, -2.0 * b * (Y - y0) / (w * w) * g
    return h.contiguous(), vx.contiguous(), vy.contiguous()


def _net_inputs(c, seed):
    """Network parameters and a batch of smooth coarse fields of unit size with their targets."""
    r = _rng(seed, 2)
    p = []
    for ci, co, k, last in _layers(ARCHS[c["arch"]][1]):
        b = math.sqrt(6.0 / (ci * k * k)) * (0.1 if last else 1.0)
        p += [r.uniform(-b, b, co * ci * k * k), r.uniform(-0.05, 0.05, co)]
    p = torch.tensor(np.concatenate(p).astype(np.float32), device=DEV)
    g = dict(Nx=c["n"], Ny=c["n"], Lx=1.0, Ly=1.0)
    f = torch.stack([_band(g, r, 1.0, 10, 10) for _ in range(5 * c["batch"])]).to(torch.float32)
    f = f.reshape(c["batch"], 5, c["n"], c["n"])
    return p, f[:, :4].contiguous(), f[:, 4:].contiguous()


def _layers(w):
    """(Ci, Co, kernel, is the output layer) in the order of the parameters."""
    D, out = len(w), []
    for l in range(D - 1):
        out += [(w[l - 1] if l else 4, w[l], 3, False), (w[l], w[l], 3, False)]
    out += [(w[D - 2], w[D - 1], 3, False), (w[D - 1], w[D - 1], 3, False)]
    out += [(w[l + 1] + w[l], w[l], 3, False) for l in range(D - 2, -1, -1)]
    return out + [(w[0], 1, 1, True)]


# the ensemble's uneven grids, in turn
GRIDS = [(256, 256, 60.0, 60.0), (512, 256, 120.0, 60.0), (1024, 512, 120.0, 60.0)]


def _members(c):
    out = []
    for i in range(c["members"]):
        Nx, Ny, Lx, Ly = GRIDS[i % len(GRIDS)]
        out.append(dict(c, Nx=Nx, Ny=Ny, Lx=Lx, Ly=Ly))
    return out


def _solver(c):
    o = {k: c[k] for k in ("precision", "guess", "graph") if k in c}
    return S.Solver(c["Nx"], c["Ny"], c["Lx"], c["Ly"], **o)


def _operands(c, seed):
    """(h, sigma or right-hand side) of an elliptic call."""
    h = _state(c, seed)[0]
    return h, _band(c, _rng(seed, 3), 0.1)


def prepare(case, seed):
    c, k = case, case["kind"]
    st = dict(case=c)
    if k == "noalloc":
        h, f = _operands(c, seed)
        # the first call on a device loads the library's code there
        return dict(st, h=h, f=f, out=torch.empty_like(h))
    if k in ("fft2", "gradient"):
        return dict(st, s=_solver(c), f=_state(c, seed)[0] + _band(c, _rng(seed, 3), 0.1))
    if k in ("elliptic", "solve"):
        h, f = _operands(c, seed)
        return dict(st, s=_solver(c), h=h, f=f)
    if k in ("rhs", "rk4"):
        h, vx, vy = _state(c, seed)
        init = [h, vx, vy, torch.zeros_like(h)]
        return dict(st, s=_solver(c), init=init, work=[t.clone() for t in init])
    if k == "ensemble":
        init, solvers, streams = [], [], []
        for i, m in enumerate(_members(c)):
            h, vx, vy = _state(m, seed * 100 + i)
            init.append([h, vx, vy, torch.zeros_like(h)])
            solvers.append(_solver(m))
            streams.append(torch.cuda.Stream())
            solvers[-1].set_stream(streams[-1])
        return dict(st, solvers=solvers, streams=streams, init=init, work=[[t.clone() for t in f] for f in init])
    p, x, t = _net_inputs(c, seed)
    net = U.UNet(c["n"], max_batch=c["batch"], bf16=True, seed=0, arch=ARCHS[c["arch"]])
    net.set_params(p)
    return dict(st, net=net, x=x, t=t)


# --------------------------------------------------------------------- runs

def run(state):
    c, k = state["case"], state["case"]["kind"]
    if k == "noalloc":
        S.sgn_elliptic_apply_noalloc(c["Nx"], c["Ny"], c["Lx"], c["Ly"], state["h"], state["f"], state["out"],
                                     torch.cuda.current_stream().cuda_stream)
        return state["out"]
    if k == "fft2":
        fh = state["s"].fft2(state["f"])
        return fh, state["s"].ifft2(fh)
    if k == "gradient":
        return state["s"].derivative(state["f"])
    if k == "elliptic":
        return state["s"].elliptic_apply(state["h"], state["f"])
    if k == "solve":
        return state["s"].gmres_solve(state["h"], state["f"])[0]
    if k == "rhs":
        h, vx, vy, sg = state["init"]
        state["work"][3].copy_(sg)
        return (*state["s"].rhs(h, vx, vy, state["work"][3]), state["work"][3])
    if k == "rk4":
        for w, i in zip(state["work"], state["init"]):
            w.copy_(i)
        state["s"].rk4_step(*state["work"], c["dt"], c["steps"])
        return state["work"]
    if k == "ensemble":
        cur = torch.cuda.current_stream()
        for ws, fs in zip(state["work"], state["init"]):
            for w, i in zip(ws, fs):
                w.copy_(i)
        for t in state["streams"]:
            t.wait_stream(cur)
        S.sgn_rk4_step_batch([s.handle for s in state["solvers"]], state["work"], c["dt"], c["steps"])
        return state["work"]
    if k == "train":
        y = state["net"].forward(state["x"])
        loss = state["net"].backward(state["t"])
        return y, loss, state["net"].grads()
    return state["net"].infer(state["x"])


def _spec(c):
    return c["Ny"] * (c["Nx"] // 2 + 1) * 16


def _fft_flops(c):
    """One real 2D transform: 2.5 N log2 N."""
    n = c["Nx"] * c["Ny"]
    return 2.5 * n * math.log2(n)


def work(case):
    c, k = case, case["kind"]
    if k == "ensemble":
        ws = [work(dict(m, kind="rk4")) for m in _members(c)]
        return {key: sum(w[key] for w in ws) for key in ("bytes", "flops")}
    if k in ("train", "infer"):
        macs, w, n = 0.0, ARCHS[c["arch"]][1], c["n"]
        D = len(w)
        lv = [l for l in range(D - 1) for _ in range(2)] + [D - 1] * 2 + list(range(D - 2, -1, -1)) + [0]
        size = 0
        for (ci, co, kk, _), l in zip(_layers(w), lv):
            macs += ci * co * kk * kk * (n >> l) ** 2
            size += co * ci * kk * kk + co
        px = 4.0 * c["batch"] * n * n
        if k == "infer":
            return {"bytes": px * 5 + 4.0 * size, "flops": 2.0 * macs * c["batch"]}
        return {"bytes": px * 6 + 8.0 * size, "flops": 6.0 * macs * c["batch"]}
    n = 8.0 * c["Nx"] * c["Ny"]
    f = _fft_flops(c)
    if k == "fft2":
        return {"bytes": 2 * n + 2.0 * _spec(c), "flops": 2 * f}
    if k == "gradient":
        return {"bytes": 3 * n, "flops": 3 * f}
    # L[sigma]: sigma_hat, three inverse and three forward transforms, the field back
    apply = 8 * f
    if k in ("noalloc", "elliptic"):
        return {"bytes": 3 * n, "flops": apply}
    if k == "solve":  # a residual and one Krylov step at the least
        return {"bytes": 3 * n, "flops": 12 * f + 4 * f}
    # one stage: 1/h, one residual of L, the right-hand side (5 inverse, 3 forward)
    stage = (1 + 6 + 8) * f
    if k == "rhs":
        return {"bytes": 8 * n, "flops": stage + 8 * f}
    return {"bytes": 8 * n, "flops": 4 * c["steps"] * stage + 8 * f}


# ------------------------------------------------- what it comes to in 64 bits

class _Ref:
    """The spectral method in torch's own float64 transforms: zeroed Nyquist
    wavenumbers, the elliptic equation solved by preconditioned conjugate
    gradients to rounding, classic RK4."""

    def __init__(self, c):
        Nx, Ny = c["Nx"], c["Ny"]
        two_pi = 2.0 * math.pi
        kx = two_pi * torch.arange(Nx // 2 + 1, dtype=F64, device=DEV) / c["Lx"]
        kx[-1] = 0.0
        m = torch.arange(Ny, device=DEV)
        ky = two_pi * torch.where(m < Ny // 2, m, m - Ny).to(F64) / c["Ly"]
        ky[Ny // 2] = 0.0
        self.kx, self.ky, self.shape = kx[None, :], ky[:, None], (Ny, Nx)
        self.M = 3.0 + self.kx ** 2 + self.ky ** 2

    def fwd(self, f):
        return torch.fft.rfft2(f)

    def inv(self, F):
        return torch.fft.irfft2(F, s=self.shape)

    def grad(self, f):
        F = self.fwd(f)
        return self.inv(1j * self.kx * F), self.inv(1j * self.ky * F)

    def div(self, a, b):
        return self.inv(1j * self.kx * self.fwd(a) + 1j * self.ky * self.fwd(b))

    def L(self, h, s):
        sx, sy = self.grad(s)
        return 3.0 * s / h ** 3 - self.div(sx / h, sy / h)

    def solve(self, h, b):
        x = torch.zeros_like(b)
        r = b.clone()
        z = self.inv(self.fwd(r) / self.M)
        p, rz = z, float((r * z).sum())
        stop = 1e-32 * rz
        for _ in range(200):
            if not rz > stop:
                break
            q = self.L(h, p)
            a = rz / float((p * q).sum())
            x = x + a * p
            r = r - a * q
            z = self.inv(self.fwd(r) / self.M)
            new = float((r * z).sum())
            p, rz = z + (new / rz) * p, new
        return x

    def rhs(self, h, vx, vy):
        s = self.solve(h, -self.div(vx, vy))
        sx, sy = self.grad(s)
        ht = -self.div(h * vx - sx, h * vy - sy)
        F = 0.5 * (vx * vx + vy * vy) - 0.5 * (sx * sx + sy * sy) / h ** 2 + (h - 1.0) - 4.5 * s * s / h ** 4
        fx, fy = self.grad(F)
        return ht, -fx, -fy, s

    def rk4(self, u, dt, steps):
        s = None
        for _ in range(steps):
            acc, us = None, u
            for w, nxt in ((1.0, 0.5), (2.0, 0.5), (2.0, 1.0), (1.0, None)):
                *k, s = self.rhs(*us)
                acc = [w * a for a in k] if acc is None else [a + w * b for a, b in zip(acc, k)]
                if nxt is not None:
                    us = [a + nxt * dt * b for a, b in zip(u, k)]
            u = [a + dt / 6.0 * b for a, b in zip(u, acc)]
        return [*u, s]


def _net(params, x, widths):
    """The periodic U-Net in the dtype of its arguments."""
    D, off, wb = len(widths), 0, []
    for ci, co, k, _ in _layers(widths):
        n = co * ci * k * k
        wb.append((params[off:off + n].reshape(co, ci, k, k), params[off + n:off + n + co]))
        off += n + co

    def conv(v, i):
        v = torch.nn.functional.pad(v, (1, 1, 1, 1), mode="circular")
        return torch.relu(torch.nn.functional.conv2d(v, *wb[i]))

    skips = []
    for l in range(D - 1):
        x = conv(conv(x, 2 * l), 2 * l + 1)
        skips.append(x)
        x = torch.nn.functional.avg_pool2d(x, 2)
    x = conv(conv(x, 2 * D - 2), 2 * D - 1)
    for l in range(D - 2, -1, -1):
        x = x.repeat_interleave(2, -1).repeat_interleave(2, -2)
        x = conv(torch.cat([x, skips[l]], 1), 2 * D + D - 2 - l)
    return torch.nn.functional.conv2d(x, *wb[-1])


def exact(case, seed):
    c, k = case, case["kind"]
    if k in ("train", "infer"):
        p, x, t = (v.to(F64) for v in _net_inputs(c, seed))
        w = ARCHS[c["arch"]][1]
        if k == "infer":
            with torch.no_grad():
                return _net(p, x, w)
        p.requires_grad_(True)
        y = _net(p, x, w)
        loss = ((y - t) ** 2).mean()
        loss.backward()
        return y.detach(), float(loss), p.grad
    if k == "ensemble":
        out = []
        for i, m in enumerate(_members(c)):
            out.append(_Ref(m).rk4(list(_state(m, seed * 100 + i)), c["dt"], c["steps"]))
        return out
    R = _Ref(c)
    if k == "fft2":
        f = _state(c, seed)[0] + _band(c, _rng(seed, 3), 0.1)
        return R.fwd(f), f
    if k == "gradient":
        return R.grad(_state(c, seed)[0] + _band(c, _rng(seed, 3), 0.1))
    if k in ("noalloc", "elliptic"):
        return R.L(*_operands(c, seed))
    if k == "solve":
        return R.solve(*_operands(c, seed))
    if k == "rhs":
        return R.rhs(*_state(c, seed))
    return R.rk4(list(_state(c, seed)), c["dt"], c["steps"])
