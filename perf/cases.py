"""Workloads of the stability library for performance measurement, each one
call of a public entry point as a user's program makes it.

Kinds (``case["kind"]``):

* ``propagator``  ``Stepper.apply_expTL`` about a base flow that was set once:
  the product with M = exp(T A) that every Krylov iteration makes;
* ``march``       ``Stepper.step_nonlinear``: the nonlinear map, as base-flow
  marching and selective frequency damping run it, in place;
* ``tangent``     ``Stepper.apply_tangent``: the exact Jacobian product of the
  Newton-Krylov base-flow solve;
* ``cgs2``        ``cgs2_orthogonalize``: one Gram-Schmidt step of a new Krylov
  vector against the basis;
* ``arnoldi``     ``Stepper.arnoldi_eigs``: a whole m-step factorisation with its
  Ritz values and residuals;
* ``unet_forward``, ``unet_gradient``: the learned base-flow guess, prediction
  and training direction.

Steppers of precision 64 (FP64), 48 (double-float) and 32 (FP32) are used with
the launch plans they are created with.  Every entry point takes and returns
float64 fields; an FP32 stepper's results are float32 values widened to
float64, so they are handed out as the float32 tensors they are (an exact
conversion).
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_1804_03859_gb300 import learned_guess, nsstab

LX, LY = 16.0, 8.0      # the box of the cylinder wake


def listed():
    return [
        # the 128x64 cylinder workload's product with M (T = 0.5): the smallest grid in use, short serial kernels
        dict(name="propagator 128x64 f64", kind="propagator", nx=128, ny=64, prec=64, sets=1, per=1, steps=50),
        # the 512x256 workload's product with M (T = 0.5), which the eigen-solves spend their time in
        dict(name="propagator 512x256 f64", kind="propagator", nx=512, ny=256, prec=64, sets=1, per=1, steps=200),
        # the same in double-float arithmetic, the faster FP64-class stepper of the same solve
        dict(name="propagator 512x256 df64", kind="propagator", nx=512, ny=256, prec=48, sets=1, per=1, steps=200),
        # one Jacobian product (T = 0.4) of the 512x256 Newton-Krylov base flow, FP32 inside the FP64 iteration
        dict(name="tangent 512x256 f32", kind="tangent", nx=512, ny=256, prec=32, sets=1, per=2, steps=160),
        # FP64 base-flow marching on a fine grid
        dict(name="march 2048x1024 f64", kind="march", nx=2048, ny=1024, prec=64, sets=1, per=1, steps=10),
        # a Reynolds sweep of 16 flows in one batch, FP32 (T = 0.5)
        dict(name="sweep16 512x256 f32", kind="propagator", nx=512, ny=256, prec=32, sets=16, per=1, steps=200),
        # one fine-grid FP32 product (an eighth of T = 0.5)
        dict(name="propagator 2048x1024 f32", kind="propagator", nx=2048, ny=1024, prec=32, sets=1, per=1, steps=100),
        # block Krylov round of a fine-grid sweep: 4 Reynolds numbers x blocks of 8 vectors, far beyond L2
        dict(name="block4x8 2048x1024 f32", kind="propagator", nx=2048, ny=1024, prec=32, sets=4, per=8, steps=20),
        # Gram-Schmidt of a long vector of odd length against a basis beyond L2, odd number of columns
        dict(name="cgs2 1000003x129", kind="cgs2", n=1000003, j=129),
        # a whole call: the 128x64 workload's Arnoldi factorisation (m 64, leading 4), host work included
        dict(name="arnoldi 128x64 f64", kind="arnoldi", nx=128, ny=64, prec=64, sets=1, per=1, steps=50, m=64, nev=4),
        # the trained network's prediction for one flow on the 512x256 grid
        dict(name="unet forward 512x256", kind="unet_forward", nx=512, ny=256, width=24, batch=1),
        # one training pass of the network at its training size: loss and gradients of a batch of 16
        dict(name="unet gradient 128x64 b16", kind="unet_gradient", nx=128, ny=64, width=24, batch=16),
    ]


def draw(rng):
    kind = rng.choice(["propagator"] * 5 + ["march", "march", "tangent", "cgs2", "cgs2", "unet_forward",
                                            "unet_gradient"])
    if kind == "cgs2":
        j = int(round(math.exp(rng.uniform(math.log(1), math.log(200)))))
        n = int(round(math.exp(rng.uniform(math.log(2000), math.log(min(2.0e6, 1.2e8 / j))))))
        return dict(kind=kind, n=n | rng.randint(0, 1), j=j)
    if kind.startswith("unet"):
        lx, ly = rng.randint(6, 9), rng.randint(5, 8)
        width = rng.choice([8, 12, 16, 24, 32])
        bmax = max(1, min(16, (1 << 18) // (1 << (lx + ly))))
        return dict(kind=kind, nx=1 << lx, ny=1 << ly, width=width, batch=rng.randint(1, bmax))
    prec = rng.choice([64, 64, 48, 32, 32, 32])
    lx = rng.randint(6, 11)
    ly = rng.randint(max(5, lx - 2), min(10, lx + 1))
    pts = 1 << (lx + ly)
    sets, per = 1, 1
    if kind == "tangent":
        per = 2
    elif kind == "propagator" and rng.random() < 0.6:
        most = max(1, min(32, (1 << (25 if prec == 32 else 21)) // pts))
        sets = rng.randint(1, min(16, most))
        per = rng.randint(1, min(8, most // sets))
    budget = (1 << 29) if prec == 32 else (1 << 26)      # grid-point steps of all members
    steps = int(round(math.exp(rng.uniform(math.log(4), math.log(200)))))
    steps = max(4, min(steps, budget // (pts * sets * per)))
    return dict(kind=kind, nx=1 << lx, ny=1 << ly, prec=prec, sets=sets, per=per, steps=steps)


# ------------------------------------------------------------------ inputs

def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed) * 7919 + 17)


def _wake(nx, ny, count, g):
    """Developed-wake-shaped vorticity fields [count][ny][nx]: two shear layers
    of opposite sign behind the cylinder (at x = y = 4) plus random modes of
    low wavenumber, mean removed."""
    x = torch.arange(nx, dtype=torch.float64, device="cuda") * (LX / nx)
    y = torch.arange(ny, dtype=torch.float64, device="cuda") * (LY / ny)
    down = ((x - 4).clamp(0, 1) * torch.exp(-(x - 4).clamp(min=0) / 6))[None, :]
    layer = (torch.exp(-((y - 4.5) / 0.25) ** 2) - torch.exp(-((y - 3.5) / 0.25) ** 2))[:, None]
    k = torch.arange(-6, 7, dtype=torch.float64, device="cuda")
    ex = torch.exp(2j * math.pi * k[:, None] * x[None, :] / LX)
    ey = torch.exp(2j * math.pi * k[:, None] * y[None, :] / LY)
    a = torch.randn(count, 13, 13, 2, dtype=torch.float64, device="cuda", generator=g)
    a = torch.view_as_complex(a) / (1 + k[:, None] ** 2 + k[None, :] ** 2)
    pert = torch.matmul(torch.matmul(ey.T, a), ex).real
    f = 2 * down * layer + 0.05 * pert / pert.abs().amax(dim=(1, 2), keepdim=True)
    return (f - f.mean(dim=(1, 2), keepdim=True)).contiguous()


def _gauss(nx, ny, count, g):
    """Krylov start vectors: Gaussian, mean removed, unit norm."""
    f = torch.randn(count, ny, nx, dtype=torch.float64, device="cuda", generator=g)
    f -= f.mean(dim=(1, 2), keepdim=True)
    return f / f.square().sum(dim=(1, 2), keepdim=True).sqrt()


def _reynolds(case):
    return [float(r) for r in np.linspace(40.0, 100.0, case["sets"])] if case["sets"] > 1 else [60.0]


def _dt(case):
    return 0.01 * 128 / case["nx"]


def _fields(case, seed):
    """(base flows or trajectory start [sets][ny][nx], vectors [members][ny][nx])"""
    g = _gen(seed)
    nx, ny = case["nx"], case["ny"]
    return _wake(nx, ny, case["sets"], g), _gauss(nx, ny, case["sets"] * case["per"], g)


def _basis(case, seed):
    """Columns of unit norm, nearly orthogonal (random signs and magnitudes), and the new vector."""
    g = _gen(seed)
    n, j = case["n"], case["j"]
    V = torch.randn(j, n, dtype=torch.float64, device="cuda", generator=g)
    V /= math.sqrt(n)
    w = torch.randn(n, dtype=torch.float64, device="cuda", generator=g) + V.sum(dim=0)
    return V, w


def _unet_data(case, seed):
    """Flow features (cylinder bump, Re and D planes) of seeded flows, wake-shaped targets, He-normal weights."""
    g = _gen(seed)
    nx, ny, B = case["nx"], case["ny"], case["batch"]
    r = np.random.default_rng(seed)
    x = (torch.arange(nx, dtype=torch.float64, device="cuda") * (LX / nx) - 4 + LX / 2) % LX - LX / 2
    y = (torch.arange(ny, dtype=torch.float64, device="cuda") * (LY / ny) - 4 + LY / 2) % LY - LY / 2
    r2 = x[None, :] ** 2 + y[:, None] ** 2
    f = torch.empty(B, 3, ny, nx, dtype=torch.float64, device="cuda")
    for b in range(B):
        Re, D = r.uniform(40, 150), r.uniform(0.8, 1.2)
        f[b, 0] = torch.exp(-r2 / (0.5 * D) ** 2)
        f[b, 1] = (Re - 95.0) / 55.0
        f[b, 2] = (D - 1.0) / 0.2
    theta = torch.from_numpy(learned_guess.he_init(3, case["width"], seed)).cuda()
    return f.float(), _wake(nx, ny, B, g).float(), theta


def prepare(case, seed):
    kind = case["kind"]
    if kind == "cgs2":
        V, w = _basis(case, seed)
        return dict(kind=kind, n=case["n"], j=case["j"], V=V, product=w, w=torch.empty_like(w))
    if kind.startswith("unet"):
        x, target, theta = _unet_data(case, seed)
        net = nsstab.UNet(3, case["width"], case["ny"], case["nx"], max_batch=case["batch"])
        net.unet_set_params(theta)
        s = dict(kind=kind, net=net, x=x)
        if kind == "unet_forward":
            s["y"] = torch.empty(case["batch"], case["ny"], case["nx"], dtype=torch.float32, device="cuda")
        else:
            s.update(target=target, grad=torch.empty_like(theta))
        return s
    base, v = _fields(case, seed)
    kw = dict(nx=case["nx"], ny=case["ny"], dt=_dt(case), precision=case["prec"], per_set=case["per"])
    Re = _reynolds(case)
    st = nsstab.Stepper(Re=Re if case["sets"] > 1 else Re[0], **kw)
    s = dict(kind=kind, st=st, prec=case["prec"], steps=case["steps"], T=case["steps"] * _dt(case))
    if kind == "march":
        return dict(s, omega=base)
    if kind == "tangent":
        return dict(s, q=base[:1].contiguous(), v=v[:1].contiguous(), out=torch.empty_like(v[:1]))
    if kind == "arnoldi":
        return dict(s, base=base[0].contiguous(), v=v[0].contiguous(), m=case["m"], nev=case["nev"])
    st.stepper_set_base(base)
    return dict(s, v=v, out=torch.empty_like(v))


def run(s):
    kind = s["kind"]
    if kind == "propagator":
        s["st"].apply_expTL(None, s["v"], s["out"], s["T"])
        return s["out"].float() if s["prec"] == 32 else s["out"]
    if kind == "march":
        s["st"].step_nonlinear(s["omega"], s["steps"])
        return s["omega"].float() if s["prec"] == 32 else s["omega"]
    if kind == "tangent":
        s["st"].apply_tangent(s["q"], s["v"], s["out"], s["T"])
        return s["out"].float() if s["prec"] == 32 else s["out"]
    if kind == "cgs2":
        s["w"].copy_(s["product"])          # the product M v that the step orthogonalises
        h, beta = nsstab.cgs2_orthogonalize(s["V"], s["n"], s["j"], s["w"])
        return {"h": h, "beta": beta, "w": s["w"]}
    if kind == "arnoldi":
        r = s["st"].arnoldi_eigs(s["base"], s["v"], m=s["m"], nev=s["nev"], tol=1e-8, T=s["T"])
        pad = s["nev"] + 1 - len(r.mu)      # nev or nev + 1 values (a conjugate pair is never split)
        return {"mu": np.pad(r.mu, (0, pad)), "residual": np.pad(r.residual, (0, pad)), "products": r.n_matvec}
    if kind == "unet_forward":
        s["net"].unet_forward(s["x"], s["y"])
        return s["y"]
    loss = s["net"].unet_gradient(s["x"], s["target"], s["grad"])
    return {"loss": loss, "grad": s["grad"]}


# ------------------------------------------------------------------- work

def _unet_convs(case):
    """(level, input channels, output channels) of the 3x3 convolutions"""
    c = [case["width"] << l for l in range(4)]
    convs, ci = [], 3
    for l in range(4):
        convs += [(l, ci, c[l]), (l, c[l], c[l])]
        ci = c[l]
    for l in (2, 1, 0):
        convs += [(l, c[l + 1] + c[l], c[l]), (l, c[l], c[l])]
    return convs


def work(case):
    kind = case["kind"]
    if kind == "cgs2":
        n, j = case["n"], case["j"]
        return {"bytes": 8.0 * n * (j + 2), "flops": 8.0 * n * j + 2.0 * n}
    if kind.startswith("unet"):
        pts = case["nx"] * case["ny"] * case["batch"]
        convs = _unet_convs(case)
        weights = sum(9 * a * b for _, a, b in convs)
        fl = sum(18.0 * (pts >> (2 * l)) * a * b for l, a, b in convs)
        if kind == "unet_forward":
            return {"bytes": 4.0 * pts * 4 + 2 * weights, "flops": fl}
        return {"bytes": 4.0 * pts * 4 + 6 * weights, "flops": 3 * fl - 18.0 * pts * 3 * case["width"]}
    n = case["nx"] * case["ny"]
    members = case["sets"] * case["per"]
    cell = {64: 8, 48: 8, 32: 4}[case["prec"]]
    # a time step: omega and the advection history read and written, the base flow's omega and psi (read once
    # per parameter set) or nothing; five real 2D transforms of 2.5 n log2 n and about 30 pointwise operations
    lin = 2.0 * case["sets"] / members if kind != "march" else 0.0
    step_bytes = members * n * cell * (4.0 + lin)
    step_flops = members * n * (12.5 * math.log2(n) + 30.0)
    w = {"bytes": case["steps"] * step_bytes, "flops": case["steps"] * step_flops}
    if kind == "arnoldi":
        m = case["m"]
        w = {"bytes": m * w["bytes"] + 8.0 * n * m * m / 2, "flops": m * w["flops"] + 4.0 * n * m * m}
    return w


# ------------------------------------------------------------------ exact

class _Exact:
    """The time-stepper's definition in plain torch, 64 bits, batched over members."""

    def __init__(self, case):
        nx, ny = case["nx"], case["ny"]
        self.nx, self.ny, self.dt = nx, ny, _dt(case)
        self.dx, self.dy = LX / nx, LY / ny
        dev = dict(dtype=torch.float64, device="cuda")
        kx, ky = torch.arange(nx // 2 + 1, **dev), torch.arange(ny, **dev)
        lam = (-(4 / self.dx ** 2) * torch.sin(math.pi * kx / nx) ** 2)[None, :] \
            - ((4 / self.dy ** 2) * torch.sin(math.pi * ky / ny) ** 2)[:, None]
        nu = torch.tensor([1 / r for r in _reynolds(case)], **dev).repeat_interleave(case["per"])[:, None, None]
        b = 1 - 0.5 * nu * self.dt * lam
        self.A, self.B = (1 + 0.5 * nu * self.dt * lam) / b, self.dt / b
        lam[0, 0] = 1.0
        self.P = -1 / lam
        self.P[0, 0] = 0.0
        self.A[:, 0, 0] = 0.0
        self.B[:, 0, 0] = 0.0
        x, y = torch.arange(nx, **dev) * self.dx, torch.arange(ny, **dev) * self.dy
        r = torch.sqrt(((x - 4 + LX / 2) % LX - LX / 2)[None, :] ** 2 + ((y - 4 + LY / 2) % LY - LY / 2)[:, None] ** 2)
        w = self.dx                                            # half of the smoothed edge of two cells
        chi = 0.5 * (1 - torch.sin(math.pi * (r - 0.5) / (2 * w)))
        chi = torch.where(r <= 0.5 - w, 1.0, torch.where(r >= 0.5 + w, 0.0, chi))
        sig = torch.where(x >= 0.9 * LX, 10 * torch.sin(math.pi * (x - 0.9 * LX) / (0.1 * LX)) ** 2, 0.0)[None, :]
        s = self.dt * (chi / 1e-3 + sig)
        self.cS, self.cG = s / (1 + s), (self.dt * sig / (1 + s)).expand(ny, nx)

    def ddx(self, f):
        return (torch.roll(f, -1, -1) - torch.roll(f, 1, -1)) / (2 * self.dx)

    def ddy(self, f):
        return (torch.roll(f, -1, -2) - torch.roll(f, 1, -2)) / (2 * self.dy)

    def phys(self, fh):
        return torch.fft.irfft2(fh, s=(self.ny, self.nx))

    def base(self, om):
        psi = self.phys(torch.fft.rfft2(om) * self.P)
        return 1 + self.ddy(psi), -self.ddx(psi), self.ddx(om), self.ddy(om)

    def step(self, w, prev, base):
        """One step (prev: last step's advection spectrum or None); base None: nonlinear."""
        wh = torch.fft.rfft2(w)
        psi = self.phys(wh * self.P)
        u, v = self.ddy(psi), -self.ddx(psi)
        if base is None:
            N = -((1 + u) * self.ddx(w) + v * self.ddy(w))
        else:
            Ub, Vb, Ox, Oy = base
            N = -(Ub * self.ddx(w) + Vb * self.ddy(w) + u * Ox + v * Oy)
        Nh = torch.fft.rfft2(N)
        wh = self.A * wh + self.B * (Nh if prev is None else 1.5 * Nh - 0.5 * prev)
        psi = self.phys(wh * self.P)
        u, v = self.ddy(psi), -self.ddx(psi)
        du = -self.cS * u if base is not None else self.cG - self.cS * (1 + u)
        dv = -self.cS * v
        return self.phys(wh) + self.ddx(dv) - self.ddy(du), Nh

    def linear(self, v, base, steps):
        prev = None
        for _ in range(steps):
            v, prev = self.step(v, prev, base)
        return v


def _exact_unet(case, seed):
    """The network in 64 bits with its stated storage (bfloat16 input, weights and activations)."""
    x, target, theta = _unet_data(case, seed)
    theta = theta.double()
    q = lambda t: t + (t.float().bfloat16().double() - t).detach()       # noqa: E731  rounded, gradient passed on
    c = [case["width"] << l for l in range(4)]
    params, k = [], 0

    def take(*shape):
        nonlocal k
        n = math.prod(shape)
        t = theta[k:k + n].reshape(shape).clone().requires_grad_()
        k += n
        params.append(t)
        return t

    def conv(h, co):
        w, b = take(co, h.shape[1], 3, 3), take(co)
        h = torch.cat([h[..., -1:, :], h, h[..., :1, :]], dim=-2)
        h = torch.cat([h[..., -1:], h, h[..., :1]], dim=-1)
        H, W = h.shape[-2] - 2, h.shape[-1] - 2
        wq = q(w)
        z = b[None, :, None, None]
        for a in range(3):
            for e in range(3):
                z = z + torch.einsum("oi,biyx->boyx", wq[:, :, a, e], h[..., a:a + H, e:e + W])
        return q(torch.relu(z))

    def pool(h):
        B, C, H, W = h.shape
        return h.reshape(B, C, H // 2, 2, W // 2, 2).mean(dim=(3, 5))

    h, skips = q(x.double()), []
    for l in range(4):
        h = conv(conv(h, c[l]), c[l])
        if l < 3:
            skips.append(h)
            h = q(pool(h))
    for l in (2, 1, 0):
        h = torch.cat([h.repeat_interleave(2, dim=-2).repeat_interleave(2, dim=-1), skips[l]], dim=1)
        h = conv(conv(h, c[l]), c[l])
    w, b = take(1, c[0]), take(1)
    y = torch.einsum("c,bcyx->byx", q(w)[0], h) + b
    if case["kind"] == "unet_forward":
        return y.detach()
    loss = (y - target.double()).square().mean()
    grads = torch.autograd.grad(loss, params)
    return {"loss": float(loss), "grad": torch.cat([g.reshape(-1) for g in grads])}


def exact(case, seed):
    kind = case["kind"]
    if kind == "cgs2":
        V, w = _basis(case, seed)
        h1 = V @ w
        w = w - h1 @ V
        h2 = V @ w
        w = w - h2 @ V
        return {"h": (h1 + h2).cpu().numpy(), "beta": float(w.norm()), "w": w}
    if kind.startswith("unet"):
        return _exact_unet(case, seed)
    ex = _Exact(case)
    base, v = _fields(case, seed)
    steps, per = case["steps"], case["per"]
    if kind == "march":
        prev, w = None, base
        for _ in range(steps):
            w, prev = ex.step(w, prev, None)
        return w
    if kind == "tangent":
        ex.A, ex.B = ex.A[:1], ex.B[:1]
        q, d, pq, pd = base[:1], v[:1], None, None
        for _ in range(steps):
            b = ex.base(q)
            d, pd = ex.step(d, pd, b)
            q, pq = ex.step(q, pq, None)
        return d
    if kind == "propagator":
        out = torch.empty_like(v)
        A, B = ex.A, ex.B
        for k in range(case["sets"]):                # one parameter set at a time, for memory
            m = slice(k * per, (k + 1) * per)
            ex.A, ex.B = A[m], B[m]
            out[m] = ex.linear(v[m], ex.base(base[k:k + 1]), steps)
        return out
    m, nev = case["m"], case["nev"]
    b = ex.base(base[:1])
    V = torch.zeros(m + 1, v[0].numel(), dtype=torch.float64, device="cuda")
    H = np.zeros((m + 1, m))
    V[0] = v[0].reshape(-1) / v[0].norm()
    for k in range(m):
        w = ex.linear(V[k].reshape(1, case["ny"], case["nx"]), b, steps).reshape(-1)
        h = V[:k + 1] @ w
        w = w - h @ V[:k + 1]
        h2 = V[:k + 1] @ w
        w = w - h2 @ V[:k + 1]
        H[:k + 1, k] = (h + h2).cpu().numpy()
        H[k + 1, k] = float(w.norm())
        V[k + 1] = w / w.norm()
    mu, Y = np.linalg.eig(H[:m])
    order = sorted(range(m), key=lambda i: (-round(abs(mu[i]), 10), -mu[i].imag))
    keep = nev
    if mu[order[nev - 1]].imag > 0 and abs(mu[order[nev]] - np.conj(mu[order[nev - 1]])) < 1e-9:
        keep += 1
    order = order[:keep]
    res = np.array([abs(H[m, m - 1] * Y[m - 1, i]) / np.linalg.norm(Y[:, i]) for i in order])
    pad = nev + 1 - keep
    return {"mu": np.pad(mu[order], (0, pad)), "residual": np.pad(res, (0, pad)), "products": None}
