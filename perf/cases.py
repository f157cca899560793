"""Timed cases of the library: what a simulation program has it do, end to end
through the Python binding.

A pass is one call sequence of such a program: load a state (device tensor, or
host array), advance it a few steps with Courant time steps, read the state back;
or, for the gradient cases, a differentiable rollout with its backward pass; or a
batch of independent problems advanced together.  Initial states are seeded random
flows (a few Fourier modes in every primitive, a divergence-free field from a
random potential, and, where the limiter is on, steep shear layers a few cells
wide), formed on the device as P1 coefficients.

The results of the FP32 path are returned as float32: that is the type its
derivative coefficients are stored in and its fluxes are computed in (float64 is
only the container of the exchange layout).
"""
import math

import numpy as np
import torch

from paper_1305_5536_gb300 import dg

KMAX, MODES = 6, 6  # Fourier modes of the initial flow


def _case(name, kind, eq, n, precision, steps, integrator="rk2", limiter=1, gamma=5.0 / 3.0,
          face_points=0, problems=0):
    nx, ny, nz = (tuple(n) + (0,))[:3]
    c = {"kind": kind, "eq": eq, "nx": nx, "ny": ny, "nz": nz, "precision": precision,
         "steps": steps, "integrator": integrator, "limiter": limiter, "gamma": gamma,
         "face_points": face_points, "problems": problems}
    return dict(c, name=name) if name else c


def listed():
    return [
        # a small 2D Euler problem in FP64, the size of a convergence study: launch
        # latency and too few tiles to fill the chip
        _case("euler2d_64_fp64", "advance", "euler", (64, 64), "fp64", 10),
        # the headline: 2D MHD turbulence at 512^2, SSP-RK2 with the min/max limiter
        _case("mhd2d_512_fp32", "advance", "mhd", (512, 512), "fp32", 4),
        # the same in FP64, as the verification runs use it
        _case("mhd2d_512_fp64", "advance", "mhd", (512, 512), "fp64", 2),
        # the paper's own integrator on the same grid
        _case("mhd2d_512_mh_fp32", "advance", "mhd", (512, 512), "fp32", 4, integrator="mh"),
        # an odd-sized 2D Euler run with the WENO-type limiter (the paper's choice)
        _case("euler2d_531x277_weno_fp32", "advance", "euler", (531, 277), "fp32", 3, limiter=2,
              gamma=1.4),
        # the large 3D Kelvin-Helmholtz-like run, far beyond L2
        _case("euler3d_256_fp32", "advance", "euler", (256, 256, 256), "fp32", 2),
        # a 3D verification run in FP64
        _case("euler3d_64_fp64", "advance", "euler", (64, 64, 64), "fp64", 1),
        # a ragged 3D box with MUSCL-Hancock
        _case("euler3d_150x101x77_mh_fp32", "advance", "euler", (150, 101, 77), "fp32", 4,
              integrator="mh", gamma=1.4),
        # 3D MHD with the 11-function field basis, SSP-RK2
        _case("mhd3d_128_fp32", "advance", "mhd", (128, 128, 128), "fp32", 2),
        # many independent 2D MHD problems in one context (parameter studies)
        _case("mhd2d_batch48_fp32", "batch", "mhd", (32, 512), "fp32", 2, problems=48),
        # inverse problems: recorded rollout and its checkpointed adjoint
        _case("euler2d_256_gradient_fp32", "gradient", "euler", (256, 256), "fp32", 20, limiter=0),
        # a restart through host arrays (numpy in, numpy out), FP64
        _case("euler2d_200x120_host_fp64", "host", "euler", (200, 120), "fp64", 2),
    ]


def _size(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["2d", "2d", "2d", "3d", "3d", "batch", "gradient", "host"])
    precision = rng.choice(["fp32", "fp32", "fp64"])
    gamma = rng.choice([5.0 / 3.0, 1.4])
    integrator = rng.choice(["rk2", "mh"])
    fp = rng.choice([1, 2]) if integrator == "mh" else 0
    eq = rng.choice(["euler", "mhd"])
    limiter = rng.choice([1, 1, 2])
    if kind == "2d":
        hi = 540 if precision == "fp32" else 256
        n = (_size(rng, 48, hi), _size(rng, 48, hi))
        return _case(None, "advance", eq, n, precision, rng.randint(1, 4), integrator, limiter, gamma, fp)
    if kind == "3d":
        hi = 128 if precision == "fp32" else 44
        n = tuple(_size(rng, 20, hi) for _ in range(3))
        return _case(None, "advance", eq, n, precision, rng.randint(1, 2), integrator, limiter, gamma, fp)
    if kind == "batch":
        hi = 360 if precision == "fp32" else 96
        return _case(None, "batch", eq, (_size(rng, 24, 48), _size(rng, 64, hi)), precision, 2,
                     "rk2", limiter, gamma, 0, rng.randint(3, 32))
    if kind == "gradient":
        n = (_size(rng, 40, 256), _size(rng, 40, 200)) if precision == "fp32" else (_size(rng, 24, 64), _size(rng, 24, 64))
        return _case(None, "gradient", "euler", n, precision, rng.randint(4, 16), "rk2", 0, gamma)
    n = (_size(rng, 40, 220), _size(rng, 40, 220))
    return _case(None, "host", eq, n, precision, rng.randint(1, 3), integrator, 1, gamma, fp)


# ---------------------------------------------------------------------------
# initial states
# ---------------------------------------------------------------------------
def _device():
    return torch.device("cuda" if torch.cuda.is_available() else "cpu")


def _grids(case):
    """Grid sizes (nx, ny[, nz]) of the problems of a case."""
    if case["kind"] == "batch":
        k, lo, hi = case["problems"], case["nx"], case["ny"]
        return [(int(round(lo * (hi / lo) ** (i / max(1, k - 1)))),) * 2 for i in range(k)]
    n = (case["nx"], case["ny"]) + ((case["nz"],) if case["nz"] else ())
    return [n]


def _modes(gen, n):
    """Random amplitudes, integer wave vectors (8 cells per wave at least) and phases."""
    dim = len(n)
    a = torch.rand(MODES, generator=gen, dtype=torch.float64) + 0.25
    a = (a / a.sum()).tolist()
    top = torch.tensor([max(1, min(KMAX, q // 8)) for q in n])
    k = torch.randint(0, 1 << 20, (MODES, dim), generator=gen) % (2 * top + 1) - top
    k[:, 0] += (k.abs().sum(1) == 0).long()
    ph = (2 * math.pi * torch.rand(MODES, generator=gen, dtype=torch.float64)).tolist()
    return list(zip(a, k.tolist(), ph))


def _field(modes, x, second=False):
    """Value, gradient and (if asked) second derivatives of a sum of sines at the
    cell centres; x: coordinates per axis, broadcastable."""
    dim = len(x)
    f, g, h = 0.0, [0.0] * dim, [[0.0] * dim for _ in range(dim)]
    for a, k, ph in modes:
        w = [2 * math.pi * kk for kk in k]
        th = sum(w[d] * x[d] for d in range(dim)) + ph
        s, c = torch.sin(th), torch.cos(th)
        f = f + a * s
        for d in range(dim):
            g[d] = g[d] + a * w[d] * c
            if second:
                for e in range(dim):
                    h[d][e] = h[d][e] - a * w[d] * w[e] * s
    return f, g, h


def _initial(eq, n, gamma, steep, gen, device):
    """P1 coefficients (exchange layout, float64) of a random flow on the unit box."""
    dim = len(n)
    shape = tuple(reversed(n))
    x = []
    for d in range(dim):
        v = (torch.arange(n[d], device=device, dtype=torch.float64) + 0.5) / n[d]
        x.append(v.reshape([n[d] if e == d else 1 for e in reversed(range(dim))]))

    def full(t):
        return t.expand(shape) if torch.is_tensor(t) else torch.full(shape, t, device=device, dtype=torch.float64)

    def scaled(base, amp):
        f, g, _ = _field(_modes(gen, n), x)
        return base + amp * f, [amp * q for q in g]

    rho, drho = scaled(1.0, 0.2)
    p, dp = scaled(1.0 if eq == "euler" else 0.6, 0.15)
    v, dv = zip(*[scaled(0.0, 0.5) for _ in range(dim)])
    v, dv = list(v), [list(q) for q in dv]
    if steep:  # two shear layers in y with a density contrast
        w = max(0.03, 4.0 / n[1])
        t = torch.tanh(torch.sin(2 * math.pi * x[1]) / w)
        dt = (1 - t * t) * (2 * math.pi / w) * torch.cos(2 * math.pi * x[1])
        rho, v[0] = rho + 0.3 * t, v[0] + 0.3 * t
        drho[1], dv[0][1] = drho[1] + 0.3 * dt, dv[0][1] + 0.3 * dt
    B = dB = None
    if eq == "mhd":
        amp = 0.1 / (2 * math.pi)
        if dim == 2:  # B = curl (A e_z) plus a mean field
            _, g, h = _field(_modes(gen, n), x, True)
            B = [0.2 + amp * g[1], 0.1 - amp * g[0]]
            dB = [[amp * h[1][0], amp * h[1][1]], [-amp * h[0][0], -amp * h[0][1]]]
        else:
            A = [_field(_modes(gen, n), x, True) for _ in range(3)]
            B, dB = [], []
            for i in range(3):
                j, k = (i + 1) % 3, (i + 2) % 3  # B_i = d_j A_k - d_k A_j
                B.append(0.1 * (i + 1) + amp * (A[k][1][j] - A[j][1][k]))
                dB.append([amp * (A[k][2][j][d] - A[j][2][k][d]) for d in range(3)])
    planes = []

    def taylor(val, grad):
        planes.append(full(val))
        planes.extend(full(q) for q in grad)

    taylor(rho, drho)
    for i in range(dim):
        taylor(rho * v[i], [rho * dv[i][d] + v[i] * drho[d] for d in range(dim)])
    v2 = sum(q * q for q in v)
    E = p / (gamma - 1) + 0.5 * rho * v2
    dE = [dp[d] / (gamma - 1) + 0.5 * v2 * drho[d] + rho * sum(v[i] * dv[i][d] for i in range(dim))
          for d in range(dim)]
    if B is not None:
        E = E + 0.5 * sum(b * b for b in B)
        dE = [dE[d] + sum(B[i] * dB[i][d] for i in range(dim)) for d in range(dim)]
    taylor(E, dE)
    if B is not None:
        planes.extend(full(b) for b in B)
        if dim == 2:
            planes.extend(full(q) for q in (dB[0][1], dB[1][0], dB[0][0]))
        else:
            planes.extend(full(q) for q in (dB[0][1], dB[0][2], dB[1][0], dB[1][2], dB[2][0],
                                            dB[2][1], -dB[1][1], -dB[2][2]))
    return torch.stack(planes).contiguous()


def _inputs(case, seed):
    device = _device()
    gen = torch.Generator().manual_seed(int(seed))
    return [_initial(case["eq"], n, case["gamma"], case["limiter"] != 0, gen, device)
            for n in _grids(case)]


def _weights(case, seed):
    """Gradient of the objective with respect to the final state (gradient cases)."""
    gen = torch.Generator().manual_seed(int(seed) + 77)
    n = _grids(case)[0]
    return torch.randn((12, n[1], n[0]), generator=gen, dtype=torch.float64).to(_device())


# ---------------------------------------------------------------------------
# a pass through the binding
# ---------------------------------------------------------------------------
def prepare(case, seed):
    us = _inputs(case, seed)
    opt = dict(gamma=case["gamma"], limiter=case["limiter"], precision=case["precision"],
               integrator=case["integrator"], face_points=case["face_points"])
    s = {"case": case, "f32": case["precision"] == "fp32"}
    grids = _grids(case)
    dim = len(grids[0])
    if case["kind"] == "batch":
        s["solver"] = dg.batch([dg.make_config(case["eq"], dim, n, **opt) for n in grids])
        s["u"] = torch.cat([u.reshape(-1) for u in us])
    elif case["kind"] == "gradient":
        s["solver"] = dg.DGSolver(case["eq"], dim, grids[0], ckpt_every=10, **opt)
        s["u"], s["w"] = us[0], _weights(case, seed)
    else:
        s["solver"] = dg.DGSolver(case["eq"], dim, grids[0], **opt)
        s["u"] = us[0].cpu().numpy() if case["kind"] == "host" else us[0]
    if case["kind"] != "gradient":
        s["out"] = np.empty_like(s["u"]) if case["kind"] == "host" else torch.empty_like(s["u"])
    return s


def run(state):
    case, solver = state["case"], state["solver"]
    if case["kind"] == "gradient":
        u = state["u"].detach().requires_grad_(True)
        final = dg.rollout(u, solver, case["steps"])
        final.backward(state["w"])
        out = {"final": final.detach(), "grad": u.grad}
    else:
        solver.set_state(state["u"])
        solver.step(case["steps"])
        out = {"state": solver.get_state(out=state["out"])}
    if state["f32"]:
        if case["kind"] == "host":
            return {k: v.astype(np.float32) for k, v in out.items()}
        return {k: v.float() for k, v in out.items()}
    return out


def work(case):
    """State read and written once per pass, and the arithmetic of the steps: per cell
    and right-hand side, the face fluxes at their Gauss points (evaluation and Riemann
    solve), the volume fluxes, the limiter and the update."""
    grids = _grids(case)
    dim = len(grids[0])
    mhd = case["eq"] == "mhd"
    planes = (12, 20)[dim - 2] if not mhd else (17, 31)[dim - 2]
    cells = sum(math.prod(n) for n in grids)
    mh = case["integrator"] == "mh"
    points = 1 if mh and case["face_points"] != 2 else 2 ** (dim - 1)
    solve = (120 if not mhd else 180) + 4 * planes
    nv = dim + 2 + (dim if mhd else 0)
    volume = 2 ** dim * (2 * planes + dim * 4 * nv)
    limiter = 0 if case["limiter"] == 0 else nv * (4 * dim + 10) + 6 * planes
    flops = (dim * points * solve + volume + limiter + 6 * planes) * cells * (1 if mh else 2) * case["steps"]
    data = 16 * planes * cells
    if case["kind"] == "gradient":  # the adjoint: recomputation and about twice the arithmetic
        flops, data = 4 * flops, 2 * data
    return {"bytes": data, "flops": flops}


# ---------------------------------------------------------------------------
# the same method in 64 bits, in plain torch
# ---------------------------------------------------------------------------
class _Exact:
    """One periodic unit box: cell averages `a` [nv, ...] and derivatives
    `g` [nv, dim, ...] of (rho, m, E[, B]) (grid axes last, x fastest)."""

    def __init__(self, case, n):
        self.mhd, self.n, self.dim = case["eq"] == "mhd", n, len(n)
        self.gam, self.lim = case["gamma"], case["limiter"]
        self.mh = case["integrator"] == "mh"
        self.points = 1 if self.mh and case["face_points"] != 2 else 2
        self.h = [1.0 / q for q in n]
        self.nv = self.dim + 2 + (self.dim if self.mhd else 0)

    def unpack(self, u):
        d, nt = self.dim, self.dim + 2
        t = u[:nt * (d + 1)].reshape((nt, d + 1) + u.shape[1:])
        a, g = [t[:, 0]], [t[:, 1:]]
        if self.mhd:
            m = u[nt * (d + 1):]
            a.append(m[:d])
            g.append(self.basis(m[d:]))
        return torch.cat(a), torch.cat(g)

    def basis(self, c):
        """Field gradients [dim, dim, ...] of the divergence-free coefficients."""
        if self.dim == 2:
            return torch.stack([torch.stack([c[2], c[0]]), torch.stack([c[1], -c[2]])])
        return torch.stack([torch.stack([c[6] + c[7], c[0], c[1]]), torch.stack([c[2], -c[6], c[3]]),
                            torch.stack([c[4], c[5], -c[7]])])

    def coefficients(self, G):
        """L2 projection of field gradients G[i][d] onto the divergence-free basis."""
        h2 = [q * q for q in self.h]
        if self.dim == 2:
            return torch.stack([G[0][1], G[1][0], (h2[0] * G[0][0] - h2[1] * G[1][1]) / (h2[0] + h2[1])])
        P, Q = h2[0] * G[0][0] - h2[1] * G[1][1], h2[0] * G[0][0] - h2[2] * G[2][2]
        A, C = h2[0] + h2[1], h2[0] + h2[2]
        det = A * C - h2[0] ** 2
        return torch.stack([G[0][1], G[0][2], G[1][0], G[1][2], G[2][0], G[2][1],
                            (C * P - h2[0] * Q) / det, (A * Q - h2[0] * P) / det])

    def pack(self, a, g):
        d, nt = self.dim, self.dim + 2
        t = torch.cat([a[:nt, None], g[:nt]], 1).reshape((nt * (d + 1),) + a.shape[1:])
        return torch.cat([t, a[nt:], self.coefficients(g[nt:])]) if self.mhd else t

    # -- physics: W = (rho, v, p[, B])
    def prims(self, c):
        d = self.dim
        v = c[1:1 + d] / c[0]
        e = c[d + 1] - 0.5 * c[0] * (v * v).sum(0)
        if self.mhd:
            e = e - 0.5 * (c[d + 2:] ** 2).sum(0)
        return torch.cat([c[:1], v, ((self.gam - 1) * e)[None], c[d + 2:]])

    def prim_grads(self, W, g):
        d, rho, v = self.dim, W[0], W[1:1 + self.dim]
        gr = g[0]
        gv = (g[1:1 + d] - v[:, None] * gr[None]) / rho
        gp = g[d + 1] - 0.5 * (v * v).sum(0) * gr - rho * (v[:, None] * gv).sum(0)
        if self.mhd:
            gp = gp - (W[d + 2:, None] * g[d + 2:]).sum(0)
        return torch.cat([gr[None], gv, ((self.gam - 1) * gp)[None], g[d + 2:]])

    def cons_grads(self, W, q):
        d, rho, v = self.dim, W[0], W[1:1 + self.dim]
        gm = rho * q[1:1 + d] + v[:, None] * q[0][None]
        gE = q[d + 1] / (self.gam - 1) + 0.5 * (v * v).sum(0) * q[0] + rho * (v[:, None] * q[1:1 + d]).sum(0)
        if self.mhd:
            gE = gE + (W[d + 2:, None] * q[d + 2:]).sum(0)
        return torch.cat([q[:1], gm, gE[None], q[d + 2:]])

    def flux(self, W, d):
        n, rho, v, p = self.dim, W[0], W[1:1 + self.dim], W[1 + self.dim]
        E = p / (self.gam - 1) + 0.5 * rho * (v * v).sum(0)
        if not self.mhd:
            m = [rho * v[i] * v[d] + (p if i == d else 0) for i in range(n)]
            return torch.stack([rho * v[d]] + m + [(E + p) * v[d]])
        B = W[2 + n:]
        b2 = 0.5 * (B * B).sum(0)
        E, pT = E + b2, p + b2
        m = [rho * v[i] * v[d] - B[i] * B[d] + (pT if i == d else 0) for i in range(n)]
        return torch.stack([rho * v[d]] + m + [(E + pT) * v[d] - B[d] * (v * B).sum(0)]
                           + [B[i] * v[d] - v[i] * B[d] for i in range(n)])

    def fast(self, W, bn):
        n = self.dim
        a2 = self.gam * W[1 + n] / W[0]
        if not self.mhd:
            return a2.sqrt()
        s = a2 + (W[2 + n:] ** 2).sum(0) / W[0]
        return (0.5 * (s + (s * s - 4 * a2 * bn * bn / W[0]).clamp_min(0).sqrt())).sqrt()

    def riemann(self, L, R, d):
        return self.hlld(L, R, d) if self.mhd else self.godunov(L, R, d)

    def pressure(self, p, r, pK, c):
        g = self.gam
        A, B = 2 / ((g + 1) * r), (g - 1) / (g + 1) * pK
        q = (A / (p + B)).sqrt()
        fs, ds = (p - pK) * q, q * (1 - 0.5 * (p - pK) / (p + B))
        w = (p / pK) ** ((g - 1) / (2 * g))
        fr, dr = 2 * c / (g - 1) * (w - 1), w / (r * c * (p / pK))
        return torch.where(p > pK, fs, fr), torch.where(p > pK, ds, dr)

    def godunov(self, L, R, d):
        g, n = self.gam, self.dim
        rL, uL, pL, rR, uR, pR = L[0], L[1 + d], L[1 + n], R[0], R[1 + d], R[1 + n]
        cL, cR = (g * pL / rL).sqrt(), (g * pR / rR).sqrt()
        with torch.no_grad():
            p = (0.5 * (pL + pR) - 0.125 * (uR - uL) * (rL + rR) * (cL + cR))
            p = torch.maximum(p, 1e-3 * torch.minimum(pL, pR))
            for _ in range(12):
                fL, dL = self.pressure(p, rL, pL, cL)
                fR, dR = self.pressure(p, rR, pR, cR)
                p = torch.maximum(p - (fL + fR + uR - uL) / (dL + dR), 1e-10 * torch.minimum(pL, pR))
        fL, dL = self.pressure(p, rL, pL, cL)
        fR, dR = self.pressure(p, rR, pR, cR)
        p = p - (fL + fR + uR - uL) / (dL + dR).detach()  # carries the derivative of p*
        fL, fR = self.pressure(p, rL, pL, cL)[0], self.pressure(p, rR, pR, cR)[0]
        us = 0.5 * (uL + uR) + 0.5 * (fR - fL)
        left = us >= 0
        sg = torch.where(left, 1.0, -1.0).to(us.dtype)
        rK, pK, cK = torch.where(left, rL, rR), torch.where(left, pL, pR), torch.where(left, cL, cR)
        w, ws, x = sg * torch.where(left, uL, uR), sg * us, p / pK
        g6 = (g - 1) / (g + 1)
        shock = p > pK
        rs = torch.where(shock, rK * (x + g6) / (g6 * x + 1), rK * x ** (1 / g))
        still = torch.where(shock, w - cK * ((g + 1) / (2 * g) * x + (g - 1) / (2 * g)).sqrt(), w - cK) >= 0
        fan = ~shock & ~still & (ws - cK * x ** ((g - 1) / (2 * g)) >= 0)
        cf = (2 / (g + 1) * (cK + 0.5 * (g - 1) * w)).clamp_min(1e-3)
        rho = torch.where(still, rK, torch.where(fan, rK * (cf / cK) ** (2 / (g - 1)), rs))
        u = sg * torch.where(still, w, torch.where(fan, cf, ws))
        pp = torch.where(still, pK, torch.where(fan, pK * (cf / cK) ** (2 * g / (g - 1)), p))
        v = [u if i == d else torch.where(left, L[1 + i], R[1 + i]) for i in range(n)]
        return self.flux(torch.stack([rho] + v + [pp]), d)

    def hlld(self, L, R, d):
        n = self.dim
        bn = 0.5 * (L[2 + n + d] + R[2 + n + d])
        L, R = L.clone(), R.clone()
        L[2 + n + d] = bn
        R[2 + n + d] = bn
        t = [i for i in range(n) if i != d]

        def cons(W):
            E = W[1 + n] / (self.gam - 1) + 0.5 * W[0] * (W[1:1 + n] ** 2).sum(0) + 0.5 * (W[2 + n:] ** 2).sum(0)
            return torch.cat([W[:1], W[0] * W[1:1 + n], E[None], W[2 + n:]])

        def total(W):
            return W[1 + n] + 0.5 * (W[2 + n:] ** 2).sum(0)

        cm = torch.maximum(self.fast(L, bn), self.fast(R, bn))
        uL, uR, rL, rR = L[1 + d], R[1 + d], L[0], R[0]
        SL, SR = torch.minimum(uL, uR) - cm, torch.maximum(uL, uR) + cm
        dL, dR = SL - uL, SR - uR
        den = dR * rR - dL * rL
        pTL, pTR = total(L), total(R)
        SM = (dR * rR * uR - dL * rL * uL - pTR + pTL) / den
        pTs = (dR * rR * pTL - dL * rL * pTR + rL * rR * dR * dL * (uR - uL)) / den

        def star(W, S, dS, pT):
            r, u = W[0], W[1 + d]
            dd = r * dS * (S - SM) - bn * bn
            flat = dd.abs() < 1e-8 * (r * dS * dS + bn * bn)
            safe = torch.where(flat, torch.ones_like(dd), dd)
            rs = r * dS / (S - SM)
            vs, bs = {}, {}
            for i in t:
                vs[i] = torch.where(flat, W[1 + i], W[1 + i] - W[2 + n + i] * bn * (SM - u) / safe)
                bs[i] = torch.where(flat, W[2 + n + i], W[2 + n + i] * (r * dS * dS - bn * bn) / safe)
            E = cons(W)[1 + n]
            vB = u * bn + sum(W[1 + i] * W[2 + n + i] for i in t)
            vBs = SM * bn + sum(vs[i] * bs[i] for i in t)
            return rs, vs, bs, (dS * E - pT * u + pTs * SM + bn * (vB - vBs)) / (S - SM), vBs

        def vec(r, v, E, b):
            return torch.stack([r] + [r * (SM if i == d else v[i]) for i in range(n)] + [E]
                               + [bn if i == d else b[i] for i in range(n)])

        rsL, vL, bL, EL, vBL = star(L, SL, dL, pTL)
        rsR, vR, bR, ER, vBR = star(R, SR, dR, pTR)
        qL, qR, sg = rsL.sqrt(), rsR.sqrt(), torch.sign(bn)
        SsL, SsR = SM - bn.abs() / qL, SM + bn.abs() / qR
        vss = {i: (qL * vL[i] + qR * vR[i] + (bR[i] - bL[i]) * sg) / (qL + qR) for i in t}
        bss = {i: (qL * bR[i] + qR * bL[i] + qL * qR * (vR[i] - vL[i]) * sg) / (qL + qR) for i in t}
        vBss = SM * bn + sum(vss[i] * bss[i] for i in t)
        UL, UR = cons(L), cons(R)
        UsL, UsR = vec(rsL, vL, EL, bL), vec(rsR, vR, ER, bR)
        FL, FR = self.flux(L, d), self.flux(R, d)
        F1, F4 = FL + SL * (UsL - UL), FR + SR * (UsR - UR)
        F2 = F1 + SsL * (vec(rsL, vss, EL - qL * (vBL - vBss) * sg, bss) - UsL)
        F3 = F4 + SsR * (vec(rsR, vss, ER + qR * (vBR - vBss) * sg, bss) - UsR)
        w = torch.where
        F = w(SL > 0, FL, w(SR < 0, FR, w(SsL >= 0, F1, w(SsR <= 0, F4, w(SM >= 0, F2, F3)))))
        F[2 + n + d] = 0
        return F

    # -- limiter (on primitive gradients q)
    def nb(self, f, d, s):
        return torch.roll(f, -s, -1 - d)

    def alpha(self, phi, hi, lo, q):
        a = torch.stack([(q[d] * self.h[d] / 2).abs() for d in range(self.dim)]).amax(0)
        m = torch.minimum(hi - phi, phi - lo)
        return torch.where(a > 0, (m / torch.where(a > 0, a, torch.ones_like(a))).clamp_max(1), torch.ones_like(a))

    def limit(self, W, q):
        n = self.dim
        hi, lo = W, W
        for d in range(n):
            for s in (1, -1):
                hi, lo = torch.maximum(hi, self.nb(W, d, s)), torch.minimum(lo, self.nb(W, d, s))
        al = lambda k, g: self.alpha(W[k], hi[k], lo[k], g)  # noqa: E731
        if self.lim == 1:
            a = [al(k, q[k]) for k in range(self.nv)]
            if self.mhd:
                b = torch.stack(a[n + 2:]).amin(0)
                a[n + 2:] = [b] * n
            return q * torch.stack(a)[:, None]
        st = torch.stack([(self.nb(W, d, 1) - self.nb(W, d, -1)) / (2 * self.h[d]) for d in range(n)], 1)
        st = torch.stack([st[k] * al(k, st[k]) for k in range(self.nv)])
        if self.mhd:
            st = torch.cat([st[:n + 2], self.basis(self.coefficients(st[n + 2:]))])

        def weight(g):
            o = 0
            for d in range(n):
                a = g[:, d] * self.h[d] / 2
                o = o + 2 * a.abs() + (self.nb(W, d, 1) - (W + a)).abs() + (self.nb(W, d, -1) - (W - a)).abs()
            if self.mhd:
                o = torch.cat([o[:n + 2], o[n + 2:].sum(0, keepdim=True).expand_as(o[n + 2:])])
            return 1 / (2.220446049250313e-16 + o).sqrt()

        wd, ws = weight(q), weight(st)
        return (wd[:, None] * q + ws[:, None] * st) / (wd + ws)[:, None]

    # -- one right-hand side; at(point) gives the primitives at a local point
    def rhs(self, at):
        n, h = self.dim, self.h
        o = 0.5 / math.sqrt(3.0)
        ra, rg = 0, [0] * n
        for q in range(2 ** n):
            W = at([(o if q >> d & 1 else -o) * h[d] for d in range(n)])
            for d in range(n):
                rg[d] = rg[d] + (12 / h[d] ** 2) / 2 ** n * self.flux(W, d)
        for d in range(n):
            t = [e for e in range(n) if e != d]
            k = self.points ** len(t)
            for q in range(k):
                x = [0.0] * n
                for b, e in enumerate(t):
                    x[e] = 0.0 if self.points == 1 else (o if q >> b & 1 else -o) * h[e]
                L, R = list(x), list(x)
                L[d], R[d] = h[d] / 2, -h[d] / 2
                F = self.riemann(at(L), self.nb(at(R), d, 1), d) / k
                Fm = self.nb(F, d, -1)
                ra = ra - (F - Fm) / h[d]
                rg[d] = rg[d] - 6 / h[d] ** 2 * (F + Fm)
                for e in t:
                    if x[e]:
                        rg[e] = rg[e] - 12 / (h[e] ** 2 * h[d]) * x[e] * (F - Fm)
        rg = torch.stack(rg, 1)
        if self.mhd:
            rg = torch.cat([rg[:n + 2], self.basis(self.coefficients(rg[n + 2:]))])
        return ra, rg

    def limited(self, a, g):
        if self.lim == 0:
            return g
        W = self.prims(a)
        return self.cons_grads(W, self.limit(W, self.prim_grads(W, g)))

    def stage(self, a, g, dt):
        def at(x):
            return self.prims(a + sum(g[:, d] * x[d] for d in range(self.dim)))
        ra, rg = self.rhs(at)
        return a + dt * ra, g + dt * rg

    def hancock(self, a, g, dt):
        n = self.dim
        g = self.limited(a, g)
        W = self.prims(a)
        q = self.prim_grads(W, g)
        rho, v, p = W[0], W[1:1 + n], W[1 + n]
        div = sum(q[1 + i, i] for i in range(n))

        def along(f, grads):
            return (f[:, None] * grads.transpose(0, 1)).sum(0) if grads.dim() == f.dim() + 1 else (f * grads).sum(0)
        Wt = [-along(v, q[0]) - rho * div]
        for i in range(n):
            force = q[1 + n, i]
            if self.mhd:
                B = W[2 + n:]
                force = force + sum(B[j] * q[2 + n + j, i] for j in range(n)) - along(B, q[2 + n + i])
            Wt.append(-along(v, q[1 + i]) - force / rho)
        Wt.append(-along(v, q[1 + n]) - self.gam * p * div)
        if self.mhd:
            for i in range(n):
                Wt.append(along(B, q[1 + i]) - along(v, q[2 + n + i]) - B[i] * div)
        Wp = W + 0.5 * dt * torch.stack(Wt)
        ra, rg = self.rhs(lambda x: Wp + sum(q[:, d] * x[d] for d in range(n)))
        return a + dt * ra, g + dt * rg

    def step(self, a, g):
        n = self.dim
        W = self.prims(a)
        speed = sum((W[1 + d].abs() + self.fast(W, W[2 + n + d] if self.mhd else None)) / self.h[d] for d in range(n))
        dt = (0.3 / speed.max()).detach()
        if self.mh:
            return self.hancock(a, g, dt)
        g0 = self.limited(a, g)
        a1, g1 = self.stage(a, g0, dt)
        a2, g2 = self.stage(a1, self.limited(a1, g1), dt)
        return 0.5 * (a + a2), 0.5 * (g0 + g2)

    def advance(self, u, steps):
        a, g = self.unpack(u)
        for _ in range(steps):
            a, g = self.step(a, g)
        return self.pack(a, g)


def exact(case, seed):
    cells = sum(math.prod(n) for n in _grids(case)) * case["steps"]
    if cells > (6e7 if torch.cuda.is_available() else 4e4):
        return None
    us, grids = _inputs(case, seed), _grids(case)
    if case["kind"] == "gradient":
        u = us[0].requires_grad_(True)
        final = _Exact(case, grids[0]).advance(u, case["steps"])
        final.backward(_weights(case, seed))
        return {"final": final.detach(), "grad": u.grad}
    out = [_Exact(case, n).advance(u, case["steps"]) for n, u in zip(grids, us)]
    if case["kind"] == "batch":
        return {"state": torch.cat([u.reshape(-1) for u in out])}
    return {"state": out[0].cpu().numpy() if case["kind"] == "host" else out[0]}
