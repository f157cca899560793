"""The FP64 exact Riemann solver of the device code, flux by flux, against the exact
solution in extended precision.

The solver takes its star pressure from an FP32 iteration and one FP64 Halley step, so
it is accurate only if the step's second-order term is: the fluxes of random pairs of
states are compared with a Newton solution in ``numpy.longdouble``.  The device function
``exact_flux`` of ``csrc/dg_physics.cuh`` is compiled into a small library of its own.
"""
import ctypes
import os
import subprocess

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1305_5536_gb300", "csrc")
EPS = np.finfo(np.float64).eps

_SRC = r"""
#include "dg_physics.cuh"
using namespace dgk;
__global__ void flux_kernel(const double* s, double* F, unsigned* err, int n, Gas<double> G) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const double* a = s + 8 * (size_t)i;
  double f[4];
  unsigned e = 0;
  exact_flux<double, 1>(G, a[0], a[1], a[2], a + 3, a[4], a[5], a[6], a + 7, f, e);
  for (int k = 0; k < 4; ++k) F[4 * (size_t)i + k] = f[k];
  err[i] = e;
}
// s: n x (rho, u, p, v) left, then right; F: n x 4; all device pointers
extern "C" int fluxes(const double* s, double gamma, double* F, unsigned* err, int n) {
  Gas<double> G;
  G.set(gamma);
  flux_kernel<<<(n + 127) / 128, 128>>>(s, F, err, n, G);
  return (int)cudaDeviceSynchronize();
}
"""


@pytest.fixture(scope="module")
def fluxes(tmp_path_factory):
    import torch

    d = tmp_path_factory.mktemp("exact64")
    (d / "x.cu").write_text(_SRC)
    so = str(d / "libx.so")
    nvcc = "/usr/local/cuda/bin/nvcc" if os.path.exists("/usr/local/cuda/bin/nvcc") else "nvcc"
    subprocess.run([nvcc, "-gencode", "arch=compute_103a,code=sm_103a", "-O3", "-std=c++17",
                    "--expt-relaxed-constexpr", "-Xcompiler", "-fPIC", "-shared", "-I", CSRC,
                    str(d / "x.cu"), "-o", so, "-lcudart"], check=True, capture_output=True)
    L = ctypes.CDLL(so)
    vp = ctypes.c_void_p
    L.fluxes.argtypes = [vp, ctypes.c_double, vp, vp, ctypes.c_int]

    def run(s, gamma):
        t = torch.from_numpy(np.ascontiguousarray(s)).cuda()
        F = torch.empty((len(s), 4), dtype=torch.float64, device="cuda")
        e = torch.empty(len(s), dtype=torch.int32, device="cuda")
        torch.cuda.synchronize()
        assert L.fluxes(t.data_ptr(), gamma, F.data_ptr(), e.data_ptr(), len(s)) == 0
        return F.cpu().numpy(), e.cpu().numpy()

    return run


def _reference(s, gamma):
    """Exact-solver fluxes of the pairs s in longdouble (Toro's pressure function,
    Newton from the left of the root, where its concave branches converge monotonically)."""
    L = np.longdouble
    rL, uL, pL, vL, rR, uR, pR, vR = (s[:, k].astype(L) for k in range(8))
    g = L(np.float64(gamma))
    z, gm, gp = (g - 1) / (2 * g), g - 1, g + 1
    cL, cR = np.sqrt(g * pL / rL), np.sqrt(g * pR / rR)

    def f(p, r, pk, c):
        q = np.sqrt(2 / (gp * r) / (p + gm / gp * pk))
        w = np.power(p / pk, z)
        sh = p > pk
        return (np.where(sh, (p - pk) * q, 2 * c / gm * np.expm1(z * np.log(p / pk))),
                np.where(sh, q * (1 - (p - pk) / (2 * (p + gm / gp * pk))), c / g * w / p))

    p = np.minimum(pL, pR) * L(1e-9)
    for _ in range(200):
        a, da = f(p, rL, pL, cL)
        b, db = f(p, rR, pR, cR)
        step = -(a + b + uR - uL) / (da + db)
        p = np.maximum(p + step, p * L(1e-3))
        if (np.abs(step) < 64 * np.finfo(L).eps * p).all():
            break
    a, _ = f(p, rL, pL, cL)
    b, _ = f(p, rR, pR, cR)
    us = (uL + uR) / 2 + (b - a) / 2
    left = us >= 0
    sg = np.where(left, L(1), L(-1))
    r, pk, c, v = (np.where(left, x, y) for x, y in ((rL, rR), (pL, pR), (cL, cR), (vL, vR)))
    w, ws, x = sg * np.where(left, uL, uR), sg * us, p / pk
    shock = p > pk
    unpert = np.where(shock, w - c * np.sqrt(gp / (2 * g) * x + z) >= 0, w - c >= 0)
    fan = ~shock & ~unpert & (ws - c * np.power(x, z) >= 0)
    cf = np.where(fan, 2 / gp * (c + gm / 2 * w), c)
    rho = np.where(shock, r * (x + gm / gp) / (gm / gp * x + 1), r * np.power(x, 1 / g))
    rho = np.where(unpert, r, np.where(fan, r * np.power(cf / c, 2 / gm), rho))
    u = sg * np.where(unpert, w, np.where(fan, cf, ws))
    pp = np.where(unpert, pk, np.where(fan, pk * np.power(cf / c, 1 / z), p))
    e = pp / gm + rho * (u * u + v * v) / 2
    return np.stack([rho * u, rho * u * u + pp, rho * u * v, u * (e + pp)], 1)


def _scales(s, gamma):
    """Per component R a, R a^2, R a^2 and a (E + p) of the larger density R, the larger
    speed a = |u| + |v| + c and the larger pressure: u* carries the rounding of the faster
    side, whichever side is sampled."""
    r, p = (np.maximum(s[:, k], s[:, k + 4]) for k in (0, 2))
    a = np.maximum(*(np.abs(s[:, k + 1]) + np.abs(s[:, k + 3]) + np.sqrt(gamma * s[:, k + 2] / s[:, k])
                     for k in (0, 4)))
    return np.stack([r * a, r * a * a, r * a * a, a * (p * gamma / (gamma - 1) + 0.5 * r * a * a)], 1)


@pytest.mark.parametrize("gamma", [5.0 / 3.0, 1.4, 1.1])
@pytest.mark.parametrize("jump,mach", [(1e-3, 1e-3), (0.3, 0.5), (2.0, 1.5), (5.0, 0.8)])
def test_random_pairs(fluxes, gamma, jump, mach):
    rng = np.random.default_rng(11)
    n = 20000
    r, p = (np.exp(jump * rng.uniform(-1, 1, (n, 2))) for _ in range(2))
    c = np.sqrt(gamma * p / r)
    u, v = (mach * c * rng.uniform(-1, 1, (n, 2)) for _ in range(2))
    s = np.stack([r[:, 0], u[:, 0], p[:, 0], v[:, 0], r[:, 1], u[:, 1], p[:, 1], v[:, 1]], 1)
    # pairs well away from a vacuum
    s = s[(u[:, 1] - u[:, 0]) < 0.5 * 2 / (gamma - 1) * c.sum(1)]
    F, err = fluxes(s, gamma)
    assert (err == 0).all()
    # a pressure function is rounded to a few eps of 2 c / (g - 1) and its slope is about
    # c / (g p): p* to a few eps 2 g / (g - 1), and the fluxes with it
    tol = 4 * EPS * 2 * gamma / (gamma - 1)
    d = np.abs(F - _reference(s, gamma)) / _scales(s, gamma)
    assert d.max() < tol, (float(d.max()), tol)


@pytest.mark.parametrize("gamma", [5.0 / 3.0, 1.4, 1.1])
def test_strong_shocks(fluxes, gamma):
    """Pressure ratios up to 1e60 (the FP32 curvature once squared p*/pK), equal and unequal
    densities, at rest and with the hot gas driven into the cold one, from either side."""
    rng = np.random.default_rng(12)
    k = np.concatenate([np.arange(2, 61), rng.uniform(15, 45, 400)])
    r = np.exp(rng.uniform(-3, 3, k.size)) * (np.arange(k.size) % 2) + 1.0 * (np.arange(k.size) % 2 == 0)
    u = np.sqrt(gamma) * rng.uniform(0, 2, k.size) * (np.arange(k.size) % 3 > 0)
    one, zero = np.ones_like(k), np.zeros_like(k)
    s = np.stack([one, u, one, zero, r, zero, 10.0 ** -k, 0.5 * one], 1)
    m = s[:, [4, 5, 6, 7, 0, 1, 2, 3]] * np.array([1, -1, 1, 1, 1, -1, 1, 1])
    s = np.concatenate([s, m])
    F, err = fluxes(s, gamma)
    assert (err == 0).all() and np.isfinite(F).all()
    d = np.abs(F - _reference(s, gamma)) / _scales(s, gamma)
    assert d.max() < 4 * EPS * 2 * gamma / (gamma - 1), float(d.max())


@pytest.mark.parametrize("gamma", [5.0 / 3.0, 1.4, 1.1])
def test_sign_of_the_shock_speed(fluxes, gamma):
    """Shocks nearly at rest on the face (relative speeds down to 1e-13, Mach numbers up to
    3e5) and cold gas (pressure ratios up to 1e60) streaming against hot gas about as fast as
    the shock runs into it: on the wrong side of the shock the flux is off by its speed times
    the jump."""
    mach = np.array([1.5, 3, 30, 300, 3e3, 3e4, 3e5])
    eps = np.array([0] + [q * 10.0 ** -k for k in range(6, 14) for q in (1, -1, 3, -3)])
    m, e = (a.ravel() for a in np.meshgrid(mach, eps))
    u1 = m * np.sqrt(gamma)
    r2 = (gamma + 1) * m * m / ((gamma - 1) * m * m + 2)
    p2 = 1 + 2 * gamma / (gamma + 1) * (m * m - 1)
    one, zero = np.ones_like(m), np.zeros_like(m)
    stat = np.stack([one, u1 * (1 - e), one, zero, r2, u1 / r2 - e * u1, p2, zero], 1)
    rng = np.random.default_rng(13)
    n = 2000
    one, zero = np.ones(n), np.zeros(n)
    cold = np.stack([np.exp(rng.uniform(-2, 2, n)), rng.uniform(0, 6, n), 10.0 ** -rng.uniform(5, 60, n),
                     zero, one, zero, one, zero], 1)
    s = np.concatenate([stat, cold])
    s = np.concatenate([s, s[:, [4, 5, 6, 7, 0, 1, 2, 3]] * np.array([1, -1, 1, 1, 1, -1, 1, 1])])
    F, err = fluxes(s, gamma)
    assert (err == 0).all()
    d = np.abs(F - _reference(s, gamma)) / _scales(s, gamma)
    assert d.max() < 4 * EPS * 2 * gamma / (gamma - 1), float(d.max())
