"""Performance cases: the calls a user of this library makes, over the sizes that they make them at.

Four kinds of case, each through a public entry point of the package:

  train     Problem.train_steps (points drawn on the device, Adam in mid-run state)
  grad      Problem.loss_grad   (drawn points, or the caller's own)
  residual  Problem.residual    (forward only, per-point squared residuals)
  grid, points   Problem.eval_grid, Problem.eval_points (a trained pair evaluated)
  cg, refined    Problem.grid_cg_solve, Problem.grid_solve_refined (the plain method)

`exact` restates the method in 64 bits with torch alone: Philox points, Kuhn-split cell
geometry, direct evaluation of the networks at the stencil points, autograd, Adam, and a
Jacobi-scaled CG of the grid rows.
"""
import math

import numpy as np
import torch

import paper_2210_14907_gb300 as nbm

PREC = {"fp32": nbm.PREC_FP32, "bf16": nbm.PREC_BF16, "fp16": nbm.PREC_FP16}
LR, BETA1, BETA2, EPS = 1e-3, 0.9, 0.999, 1e-8
STEP0 = 500  # Adam steps already taken by a training state


def _case(name, kind, **kw):
    c = {"name": name, "kind": kind, "geometry": "sphere", "prec": "bf16", "width": 128, "layers": 3, "cells": 128,
         "n": 0, "steps": 1, "mu_plus": 10.0, "band": 0.0, "refine": 0, "own_points": False, "sec41": False}
    c.update(kw)
    return c


def listed():
    return [
        # a small run: plain FP32 pair, sphere, a few thousand points, several steps per call (launches count)
        _case("train small fp32", "train", prec="fp32", width=64, layers=2, cells=32, n=4096, steps=10),
        # the convergence study's sine networks (5 x 10 units, variable coefficients), its mini-batch of 32 x 32 x 16
        _case("train sine narrow", "train", prec="fp32", width=10, layers=5, cells=32, n=16384, steps=2, sec41=True),
        # the mixed-precision training step, the package's main use
        _case("train mixed", "train", n=262144, steps=2),
        # loss and gradient on the flower interface, many cut cells, a million drawn points
        _case("grad mixed flower", "grad", geometry="flower", layers=4, cells=256, n=1048576, mu_plus=100.0, band=0.3),
        # fine resolution: FP64 rows, the largest batch
        _case("grad mixed fine", "grad", layers=4, cells=1024, n=4194304),
        # the plain FP32 path on the caller's own points, an odd batch
        _case("grad fp32 own points", "grad", prec="fp32", n=200003, own_points=True),
        # forward only with per-point residuals, implicit refinement over four spacings (the finest in FP64 rows)
        _case("residual refined", "residual", cells=64, n=50001, refine=3, own_points=True),
        # a trained pair on a dense grid
        _case("grid fp16", "grid", geometry="flower", prec="fp16", layers=4, n=512),
        # a trained pair at scattered points in the default precision
        _case("points fp32", "points", prec="fp32", n=200000),
        # a few points (probes of a solution): the call's fixed cost
        _case("points fp16 few", "points", geometry="flower", prec="fp16", layers=4, n=1000),
        # the plain mesh method, FP64 CG
        _case("cg 128", "cg", n=128),
        # the same rows on a finer grid by FP32 corrections of FP64 residuals
        _case("refined 256", "refined", n=256),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["train", "grad", "grad", "residual", "grid", "points", "cg", "refined"])
    flower = rng.random() < 0.4
    c = {"geometry": "flower" if flower else "sphere", "mu_plus": 100.0 if flower else 10.0}
    if kind in ("cg", "refined"):
        c.update(n=_log(rng, 24, 176 if kind == "cg" else 240))
        c["mu_plus"] = 10.0
    elif kind in ("grid", "points"):
        c["prec"] = rng.choice(["fp16", "bf16", "fp32"])
        c["layers"] = rng.choice([2, 3, 4])
        c["width"] = rng.choice([64, 128]) if c["prec"] == "fp32" else 128
        top = 500000 if c["prec"] == "fp32" else 60000000
        n = _log(rng, 300, top)
        c["n"] = n if kind == "points" else max(6, int(round(n ** (1 / 3))))
    else:
        path = rng.choice(["bf16", "bf16", "fp32", "sine"])
        c["layers"] = rng.choice([2, 3, 4])
        c["cells"] = rng.choice([32, 64, 128, 256])
        if path == "bf16":
            c["cells"] = rng.choice([64, 128, 256, 1024])
            c["n"] = _log(rng, 600, 1000000)
        elif path == "fp32":
            c.update(prec="fp32", width=rng.choice([64, 128]), n=_log(rng, 600, 200000))
        else:
            c.update(geometry="sphere", prec="fp32", width=10, layers=5, sec41=True, cells=rng.choice([8, 16, 32, 64]),
                     n=_log(rng, 500, 60000))
        c["refine"] = rng.choice([0, 0, 0, 1, 2]) if c["cells"] <= 128 else 0
        c["own_points"] = kind != "train" and rng.random() < 0.5
        c["band"] = 0.0 if c["own_points"] else rng.choice([0.0, 0.0, 0.3])
        c["steps"] = rng.choice([1, 2, 4]) if kind == "train" else 1
    c = _case("", kind, **c)
    del c["name"]
    return c


# ---------------------------------------------------------------- inputs

def _radius(c, seed):
    """Radius of the interface: 1/2, and for the grid solves (which take no other input) drawn about it."""
    if c["kind"] not in ("cg", "refined"):
        return 0.5
    return 0.45 + 0.1 * float(torch.rand(1, generator=torch.Generator().manual_seed(int(seed)), dtype=torch.float64))


def _desc(c, seed=0):
    step = c["kind"] in ("train", "grad", "residual")
    return nbm.ProblemDesc(
        geometry=nbm.GEOM_FLOWER if c["geometry"] == "flower" else nbm.GEOM_SPHERE, n_hidden=c["layers"],
        width=c["width"], precision=PREC[c["prec"]] if step else nbm.PREC_FP32, r0=_radius(c, seed), mu_minus=1.0,
        mu_plus=c["mu_plus"], h=2.0 / c["cells"], band_fraction=c["band"], refine_levels=c["refine"],
        solution=nbm.SOL_SEC41 if c["sec41"] else nbm.SOL_BENCH,
        activation=nbm.ACT_SIN if c["sec41"] else nbm.ACT_TANH)


def _device():
    return torch.device("cuda" if torch.cuda.is_available() else "cpu")


def _params(c, gen):
    """Glorot-uniform weights and small biases of the network pair, the flat FP32 vector."""
    H, parts = c["width"], []
    for _ in range(2):
        for i, o in [(3, H)] + [(H, H)] * (c["layers"] - 1) + [(H, 1)]:
            a = math.sqrt(6.0 / (i + o))
            parts.append((2 * torch.rand(i * o, generator=gen, dtype=torch.float64) - 1) * a)
            parts.append((2 * torch.rand(o, generator=gen, dtype=torch.float64) - 1) * 0.1)
    return torch.cat(parts).float()


def _inputs(c, seed):
    """(params, points or None, m, v) on the device, from the seed alone."""
    gen = torch.Generator().manual_seed(1000003 * int(seed) + 17)
    p = _params(c, gen)
    m = 1e-5 * torch.randn(p.numel(), generator=gen)
    v = 1e-8 * (0.5 + torch.rand(p.numel(), generator=gen))
    pts = None
    if c["kind"] == "points" or c["own_points"]:
        # lattice points of the cube, a tenth of them in a shell across the interface
        n = c["n"]
        k = torch.randint(1, 2 ** 23, (n, 3), generator=gen).double()
        d = torch.randn(n, 3, generator=gen, dtype=torch.float64)
        d = d / d.norm(dim=1, keepdim=True) * (0.35 + 0.3 * torch.rand(n, 1, generator=gen, dtype=torch.float64))
        k = torch.where(torch.rand(n, 1, generator=gen) < 0.1, torch.round((d + 1) * 4194304.0), k)
        pts = (k / 4194304.0 - 1).float()
    dev = _device()
    return p.to(dev), None if pts is None else pts.to(dev), m.to(dev), v.to(dev)


def prepare(case, seed):
    p, pts, m, v = _inputs(case, seed)
    s = {"case": case, "prob": nbm.Problem(_desc(case, seed)), "params": p, "pts": pts, "seed": int(seed) + 1}
    if case["kind"] == "train":
        s.update(m=m, v=v, step=STEP0, hist=torch.zeros(case["steps"], device=p.device))
    return s


def run(s):
    c, prob = s["case"], s["prob"]
    if c["kind"] == "train":
        s["step"] = prob.train_steps(s["params"], s["m"], s["v"], s["step"], c["steps"], c["n"], lr=LR, beta1=BETA1,
                                     beta2=BETA2, eps=EPS, seed=s["seed"], loss_hist=s["hist"])
        return {"params": s["params"], "m": s["m"], "v": s["v"], "loss": s["hist"]}
    if c["kind"] == "grad":
        loss, g = prob.loss_grad(s["params"], pts=s["pts"], n=c["n"], seed=s["seed"])
        return {"loss": loss, "grad": g}
    if c["kind"] == "residual":
        loss, r2 = prob.residual(s["params"], pts=s["pts"], n=c["n"], seed=s["seed"])
        return {"loss": loss, "r2": r2}
    if c["kind"] == "grid":
        return prob.eval_grid(s["params"], c["n"], precision=PREC[c["prec"]])
    if c["kind"] == "points":
        return prob.eval_points(s["params"], s["pts"], precision=PREC[c["prec"]])
    solve = prob.grid_cg_solve if c["kind"] == "cg" else prob.grid_solve_refined
    u, _, _, ok = solve(c["n"], rtol=1e-12)
    return {"u": u, "converged": ok}


def work(case):
    c, H, n = case, case["width"], case["n"]
    mlp = 2 * (3 * H + (c["layers"] - 1) * H * H + H)  # one network at one point
    P = nbm.param_count(_desc(c))
    if c["kind"] in ("train", "grad", "residual"):
        one = 7 * mlp * n * (1 if c["kind"] == "residual" else 3) * (1 + c["refine"])
        moved = (12 * n if c["own_points"] else 0) + (4 * n if c["kind"] == "residual" else 0)
        moved += P * {"train": 24, "grad": 8, "residual": 4}[c["kind"]]
        return {"bytes": moved * c["steps"], "flops": one * c["steps"]}
    if c["kind"] == "grid":
        return {"bytes": 4 * (n + 1) ** 3 + 4 * P, "flops": mlp * (n + 1) ** 3}
    if c["kind"] == "points":
        return {"bytes": 16 * n + 4 * P, "flops": mlp * n}
    # about 3.7 n iterations of 13 multiply-adds per unknown
    return {"bytes": 8 * (n + 1) ** 3, "flops": 26 * 3.7 * n * (n - 1) ** 3}


# ---------------------------------------------------------------- the method in 64 bits

class _Pair:
    """Level set, manufactured pair and coefficients on tensors [..., 3]."""

    def __init__(self, c, r0=0.5):
        self.r0 = r0
        self.flower, self.sec41 = c["geometry"] == "flower", c["sec41"]
        self.mu_c = (1.0, c["mu_plus"])

    def phi(self, x):
        r = x.norm(dim=-1)
        if not self.flower:
            return r - self.r0
        th, ps = torch.atan2(x[..., :2].norm(dim=-1), x[..., 2]), torch.atan2(x[..., 1], x[..., 0])
        return r - self.r0 - 0.1 * torch.sin(5 * th) * torch.cos(3 * ps)

    def grad_phi(self, x):
        r = x.norm(dim=-1, keepdim=True)
        g = x / r
        if self.flower:
            rho = x[..., :2].norm(dim=-1, keepdim=True)
            X, Y, Z = x[..., :1], x[..., 1:2], x[..., 2:]
            th, ps = torch.atan2(rho, Z), torch.atan2(Y, X)
            dth = torch.cat([Z * X / (r * r * rho), Z * Y / (r * r * rho), -rho / (r * r)], -1)
            dps = torch.cat([-Y / rho ** 2, X / rho ** 2, torch.zeros_like(X)], -1)
            g = g - 0.5 * torch.cos(5 * th) * torch.cos(3 * ps) * dth + 0.3 * torch.sin(5 * th) * torch.sin(3 * ps) * dps
        return g

    def u(self, s, x):
        X, Y, Z = x[..., 0], x[..., 1], x[..., 2]
        if self.sec41:
            return torch.exp(Z) if s == 0 else torch.cos(X) * torch.sin(Y)
        return torch.exp(X) * torch.cos(Y) * torch.sin(Z) if s == 0 else X * X + Y * Y + Z * Z

    def grad_u(self, s, x):
        X, Y, Z = x[..., 0], x[..., 1], x[..., 2]
        o = torch.zeros_like(X)
        if self.sec41:
            g = (o, o, torch.exp(Z)) if s == 0 else (-torch.sin(X) * torch.sin(Y), torch.cos(X) * torch.cos(Y), o)
        elif s == 0:
            e = torch.exp(X)
            g = (e * torch.cos(Y) * torch.sin(Z), -e * torch.sin(Y) * torch.sin(Z), e * torch.cos(Y) * torch.cos(Z))
        else:
            return 2 * x
        return torch.stack(g, -1)

    def mu(self, s, x):
        if not self.sec41:
            return torch.full_like(x[..., 0], self.mu_c[s])
        return x[..., 1] ** 2 * torch.log(x[..., 0] + 2) + 4 if s == 0 else torch.exp(-x[..., 2])

    def f(self, s, x):
        """-div(mu grad u); the reaction coefficients are 0 in every case."""
        if self.sec41:
            return -self.mu(0, x) * self.u(0, x) if s == 0 else 2 * torch.exp(-x[..., 2]) * self.u(1, x)
        return self.mu_c[0] * self.u(0, x) if s == 0 else torch.full_like(x[..., 0], -6 * self.mu_c[1])

    def alpha(self, x):
        return self.u(1, x) - self.u(0, x)

    def beta(self, x):
        g = self.grad_phi(x)
        d = self.mu(1, x)[..., None] * self.grad_u(1, x) - self.mu(0, x)[..., None] * self.grad_u(0, x)
        return (d * g).sum(-1) / g.norm(dim=-1)


def _fraction(f):
    """Share with phi <= 0 of triangles [m, 3] or tetrahedra [m, 4] with linear phi."""
    f = torch.sort(f, dim=-1).values
    neg, k = (f <= 0).sum(-1), f.shape[-1]
    lo = torch.stack([f[..., 0] / (f[..., 0] - f[..., i]) for i in range(1, k)]).prod(0)
    hi = 1 - torch.stack([f[..., -1] / (f[..., -1] - f[..., i]) for i in range(k - 1)]).prod(0)
    out = torch.where(neg == 1, lo, torch.where(neg == k - 1, hi, torch.zeros_like(lo)))
    if k == 4:
        A, B, C, D = -f[..., 0], -f[..., 1], f[..., 2], f[..., 3]
        two = (C * D * (A * A + A * B + B * B) + (C + D) * A * B * (A + B) + A * A * B * B) / (
            (C + A) * (D + A) * (C + B) * (D + B))
        out = torch.where(neg == 2, two, out)
    return torch.where(neg == k, torch.ones_like(out), torch.where(neg == 0, torch.zeros_like(out), out))


def _interface(X, f):
    """(area, area x centroid) of phi = 0 inside tetrahedra X [m, 4, 3] with values f [m, 4]."""
    f, at = torch.sort(f, dim=-1)
    X = torch.gather(X, 1, at[..., None].expand(-1, -1, 3))
    neg = (f <= 0).sum(-1)

    def zero(i, j):
        t = f[:, i] / (f[:, i] - f[:, j])
        return X[:, i] + t[:, None] * (X[:, j] - X[:, i])

    def tri(a, b, c):
        ar = 0.5 * torch.linalg.cross(b - a, c - a).norm(dim=-1)
        return ar, ar[:, None] * (a + b + c) / 3

    one, three = tri(zero(0, 1), zero(0, 2), zero(0, 3)), tri(zero(0, 3), zero(1, 3), zero(2, 3))
    q = (zero(0, 2), zero(0, 3), zero(1, 3), zero(1, 2))
    t1, t2 = tri(q[0], q[1], q[2]), tri(q[0], q[2], q[3])
    out = []
    for k in range(2):
        o, sel = torch.zeros_like(one[k]), (lambda n: (neg == n) if k == 0 else (neg == n)[:, None])
        for n, val in ((1, one[k]), (2, t1[k] + t2[k]), (3, three[k])):
            o = torch.where(sel(n), val, o)
        out.append(o)
    return out


def _corners(p, h):
    bits = torch.tensor([[(c >> a) & 1 for a in range(3)] for c in range(8)], dtype=p.dtype, device=p.device)
    return p[:, None] + h * (bits - 0.5)


def _geometry(pair, p, h):
    """Of cut cells: volume fraction, face fractions [m, 6], area / h^2, interface point, has a jump row."""
    C = _corners(p, h)
    F = pair.phi(C)
    V, S, W = 0, 0, 0
    for a, b in ((0, 1), (0, 2), (1, 0), (1, 2), (2, 0), (2, 1)):
        idx = [0, 1 << a, (1 << a) | (1 << b), 7]
        V = V + _fraction(F[:, idx]) / 6
        ar, w = _interface(C[:, idx], F[:, idx])
        S, W = S + ar, W + w
    A = []
    for f in range(6):
        a, sd = f >> 1, f & 1
        j, k = (a + 1) % 3, (a + 2) % 3
        b0 = sd << a
        c10, c01 = b0 | (1 << j), b0 | (1 << k)
        c11 = c10 | (1 << k)
        A.append(0.5 * (_fraction(F[:, [b0, c10, c11]]) + _fraction(F[:, [b0, c01, c11]])))
    jump = S > 0
    x = torch.where(jump[:, None], W / S.clamp_min(1e-300)[:, None], p)
    for _ in range(3):
        g = pair.grad_phi(x)
        x = torch.where(jump[:, None], x - (pair.phi(x) / (g * g).sum(-1))[:, None] * g, x)
    return V, torch.stack(A, -1), S / (h * h), x, jump


def _net(c, theta, s, x):
    """Network s of the flat FP64 pair at points [m, 3]."""
    H, at = c["width"], s * (theta.numel() // 2)
    a = x
    for i in [3] + [H] * (c["layers"] - 1):
        W, b = theta[at:at + i * H].view(H, i), theta[at + i * H:at + i * H + H]
        at += i * H + H
        a = torch.addmm(b, a, W.t())
        a = torch.sin(a) if c["sec41"] else torch.tanh(a)
    return a @ theta[at:at + H] + theta[at + H]


def _residual(c, pair, theta, p, h):
    """Squared residuals of the points p [m, 3] (without refinement), r^2 = (B / D)^2 + J^2."""
    neg = (pair.phi(_corners(p, h)) <= 0).sum(-1)
    cut = (neg > 0) & (neg < 8)
    q = p[:, None].repeat(1, 7, 1)  # the point and its six neighbours, face f = 2 axis + (side > 0)
    for f in range(6):
        q[:, 1 + f, f >> 1] += h if f & 1 else -h
    B, D, J = (torch.zeros_like(p[:, 0]) for _ in range(3))
    V = (neg == 8).to(p.dtype)
    A = V[:, None].repeat(1, 6)
    if cut.any():
        Vc, Ac, S, xg, jump = _geometry(pair, p[cut], h)
        V, A = V.masked_scatter(cut, Vc), A.masked_scatter(cut[:, None].expand(-1, 6), Ac)
        B = B.masked_scatter(cut, torch.where(jump, h * S * pair.beta(xg), torch.zeros_like(S)))
        Jc = torch.where(jump, _net(c, theta, 1, xg) - _net(c, theta, 0, xg) - pair.alpha(xg), torch.zeros_like(S))
        J = J.masked_scatter(cut, Jc)
    for s in range(2):
        mine = cut | (neg == (8 if s == 0 else 0))
        if not mine.any():
            continue
        qs, Vs, As = q[mine], V[mine], A[mine]
        if s == 1:
            Vs, As = 1 - Vs, 1 - As
        U = _net(c, theta, s, qs.reshape(-1, 3)).view(-1, 7)
        out = qs[:, 1:].abs().amax(-1) >= 1
        dU = torch.where(out, pair.u(1, qs[:, 1:]), U[:, 1:]) - U[:, :1]
        w = As * pair.mu(s, 0.5 * (qs[:, :1] + qs[:, 1:]))
        B = B.index_put((mine.nonzero()[:, 0],), -h * h * Vs * pair.f(s, qs[:, 0]) - (w * dU).sum(-1), accumulate=True)
        D = D.index_put((mine.nonzero()[:, 0],), w.sum(-1), accumulate=True)
    return (B / D) ** 2 + J ** 2


def _drawn(c, seed, step):
    """The points that step `step` draws (Philox4x32-10), as FP64."""
    n, mask = c["n"], np.uint64(0xFFFFFFFF)
    r = [np.arange(n, dtype=np.uint64), np.full(n, step & 0xFFFFFFFF, np.uint64), np.full(n, step >> 32, np.uint64),
         np.full(n, 0x4E424D31, np.uint64)]
    k0, k1 = seed & 0xFFFFFFFF, seed >> 32
    for _ in range(10):
        a, b = np.uint64(0xD2511F53) * r[0], np.uint64(0xCD9E8D57) * r[2]
        r = [(b >> np.uint64(32)) ^ r[1] ^ np.uint64(k0), b & mask, (a >> np.uint64(32)) ^ r[3] ^ np.uint64(k1), a & mask]
        k0, k1 = (k0 + 0x9E3779B9) & 0xFFFFFFFF, (k1 + 0xBB67AE85) & 0xFFFFFFFF
    x = np.stack([-1 + (1 + ((w * np.uint64(8388607)) >> np.uint64(32)).astype(np.float64)) / 4194304 for w in r[:3]], -1)
    nb = int(math.floor(c["band"] * n + 0.5))
    if nb:
        u = [((w[n - nb:] >> np.uint64(8)).astype(np.float64) + 0.5) / 16777216 for w in r[:3]]
        ct, ps = 1 - 2 * u[0], 2 * math.pi * u[1]
        st = np.sqrt(np.maximum(0, 1 - ct * ct))
        R = 0.5 + (0.1 * np.sin(5 * np.arccos(ct)) * np.cos(3 * ps) if c["geometry"] == "flower" else 0.0)
        R = R + (2 * u[2] - 1) * 4 * (2.0 / c["cells"])
        v = np.stack([R * st * np.cos(ps), R * st * np.sin(ps), R * ct], -1)
        x[n - nb:] = -1 + np.clip(np.floor((v + 1) * 4194304 + 0.5), 1, 8388607) / 4194304
    return torch.from_numpy(x).to(_device())


def _loss(c, theta, pts, grad):
    """(loss, gradient or None, r^2) over the points and refinement levels."""
    pair, n = _Pair(c), pts.shape[0]
    theta = theta.double().requires_grad_(grad)
    g = torch.zeros_like(theta) if grad else None
    r2 = torch.zeros(n, dtype=torch.float64, device=pts.device)
    with torch.set_grad_enabled(grad):
        for lv in range(1 + c["refine"]):
            for a in range(0, n, 131072):
                e = _residual(c, pair, theta, pts[a:a + 131072], 2.0 / c["cells"] / 2 ** lv)
                if grad:
                    g += torch.autograd.grad(e.sum() / n, theta)[0]
                r2[a:a + 131072] += e.detach()
    return r2.mean(), g, r2


def _solve(c, seed):
    """The grid rows (exact node jump) solved to rounding; node values x fastest."""
    pair, n, dev = _Pair(c, _radius(c, seed)), c["n"], _device()
    h, m1 = 2.0 / n, c["n"] - 1
    ax = -1 + torch.arange(n + 1, dtype=torch.float64, device=dev) * h
    node = torch.stack(torch.meshgrid(ax, ax, ax, indexing="ij"), -1).flip(-1)  # [k, j, i] -> (x, y, z)
    half = ax[:-1] + 0.5 * h
    neg = (pair.phi(torch.stack(torch.meshgrid(half, half, half, indexing="ij"), -1).flip(-1)) <= 0).to(torch.int8)
    cnt = sum(neg[k:k + m1, j:j + m1, i:i + m1] for i in range(2) for j in range(2) for k in range(2))
    inner = (slice(1, n),) * 3
    minus = pair.phi(node) <= 0
    J = pair.alpha(node)
    corr = torch.stack([torch.where(minus, torch.zeros_like(J), -J), torch.where(minus, J, torch.zeros_like(J))])
    for d in range(3):  # boundary nodes carry their Dirichlet value alone
        for e in (0, n):
            corr[(slice(None),) + tuple(e if d == q else slice(None) for q in range(3))] = 0
    p = node[inner]
    V = (cnt == 8).double()
    A = V[..., None].repeat(1, 1, 1, 6)
    known = torch.zeros_like(V)
    cut = (cnt > 0) & (cnt < 8)
    if cut.any():
        Vc, Ac, S, xg, jump = _geometry(pair, p[cut], h)
        V[cut], A[cut] = Vc, Ac
        known[cut] = torch.where(jump, h * S * pair.beta(xg), torch.zeros_like(S))
    for s in range(2):
        known -= h * h * (1 - V if s else V) * pair.f(s, p)
    diag, w = torch.zeros_like(V), []
    for f in range(6):
        d, sg = 2 - (f >> 1), 1 if f & 1 else -1  # tensor dimension of axis f / 2
        to = tuple(slice(1 + sg, n + sg) if d == q else slice(1, n) for q in range(3))
        fc = p.clone()
        fc[..., f >> 1] += 0.5 * sg * h
        wf = torch.zeros_like(V)
        for s in range(2):
            a = (1 - A[..., f] if s else A[..., f]) * pair.mu(s, fc)
            wf += a
            known -= a * (corr[s][to] - corr[s][inner])
        diag += wf
        edge = tuple((-1 if sg > 0 else 0) if d == q else slice(None) for q in range(3))
        known[edge] -= wf[edge] * pair.u(1, node[to][edge])
        w.append((wf, d))
    root = diag.sqrt()
    ws = []
    for f in (1, 3, 5):  # weights to the next node of each axis, of the scaled system
        wf, d = w[f]
        lo, hi = ([slice(None)] * 3 for _ in range(2))
        lo[d], hi[d] = slice(0, m1 - 1), slice(1, m1)
        ws.append((wf[tuple(lo)] / (root[tuple(lo)] * root[tuple(hi)]), tuple(lo), tuple(hi)))
    b = -known / root
    x, r = torch.zeros_like(b), b.clone()
    d, rr = r.clone(), (r * r).sum()
    stop = 1e-26 * rr
    for it in range(12 * n + 200):
        y = d.clone()
        for wf, lo, hi in ws:
            y[lo] -= wf * d[hi]
            y[hi] -= wf * d[lo]
        al = rr / (d * y).sum()
        x += al * d
        r -= al * y
        new = (r * r).sum()
        d = r + new / rr * d
        rr = new
        if it % 50 == 0 and bool(rr <= stop):
            break
    u = pair.u(1, node)
    u[inner] = x / root
    return u.reshape(-1)


def exact(case, seed):
    c = case
    if c["kind"] in ("cg", "refined"):
        return {"u": _solve(c, seed), "converged": None}
    p, pts, m, v = _inputs(c, seed)
    if c["kind"] in ("grid", "points"):
        if c["kind"] == "grid":
            # node coordinates as FP32 holds them, with one rounding
            i = torch.arange(c["n"] + 1, device=p.device).double()
            ax = (-1 + i * float(np.float32(2.0) / np.float32(c["n"]))).float().double()
            pts = torch.stack(torch.meshgrid(ax, ax, ax, indexing="ij"), -1).flip(-1).reshape(-1, 3)
        pair, th, out = _Pair(c), p.double(), []
        for a in range(0, pts.shape[0], 1 << 21):
            x = pts[a:a + (1 << 21)].double()
            minus, u = pair.phi(x) <= 0, torch.zeros(x.shape[0], dtype=torch.float64, device=x.device)
            u[minus], u[~minus] = _net(c, th, 0, x[minus]), _net(c, th, 1, x[~minus])
            out.append(u)
        return torch.cat(out)
    points = [pts.double()] if pts is not None else [
        _drawn(c, int(seed) + 1, (STEP0 + 1 + k) if c["kind"] == "train" else 1) for k in range(c["steps"])]
    if c["kind"] == "residual":
        loss, _, r2 = _loss(c, p, points[0], False)
        return {"loss": loss, "r2": r2}
    if c["kind"] == "grad":
        loss, g, _ = _loss(c, p, points[0], True)
        return {"loss": loss, "grad": g}
    p, m, v, hist = p.double(), m.double(), v.double(), []
    lr, b1, b2, eps = (float(np.float32(z)) for z in (LR, BETA1, BETA2, EPS))
    for k, x in enumerate(points):
        loss, g, _ = _loss(c, p.detach(), x, True)
        t = STEP0 + 1 + k
        m, v = b1 * m + (1 - b1) * g, b2 * v + (1 - b2) * g * g
        p = p.detach() - lr * (m / (1 - b1 ** t)) / ((v / (1 - b2 ** t)).sqrt() + eps)
        hist.append(loss)
    return {"params": p, "m": m, "v": v, "loss": torch.stack(hist)}
