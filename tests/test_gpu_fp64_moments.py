"""FP64 moments keep FP64's accuracy at high degrees: the recorded Q_diff of one particle near the equator,
where the terms of its sum grow with the degree, against extended precision. The ratio r_out / r^2 enters
to the power of the degree, so its last bits show: formed by a division (correctly rounded) the sum is
2.97 units of 2^-53 off (rms, from the same arithmetic on the host), from the squared reciprocal root 6.98."""
import math

import numpy as np
import pytest

from paper_2111_13072_gb300.inputs import Workload

pytestmark = pytest.mark.gpu

L, EPS, D = 24, 4.0, 0.001
W = Workload("equator", N=1, l_max=L, T_e_eV=2.0, n_e_m3=1e15, R_E_m=(1 - D) * 5e-3, R_D_m=5e-3, eps_D=EPS, outer_R=1.02,
             drive_kind=2, precision=0, seed=1)
LD = np.longdouble


def _canti(l, d):
    """Coefficient of r^-(l+1) P_l in Psi_anti, odd l."""
    k = (l + 1) // 2
    c = (-1.0) ** (k + 1) * 0.5 ** (k + 1) * (4.0 * k - 1) * math.prod(range(3, 2 * k - 2, 2)) / math.factorial(k)
    return c * (2 * l + 1) * EPS * (1 - d) ** (l + 1) / ((l + 1) * (EPS - 1) * (1 - d) ** (2 * l + 1) + l * EPS + l + 1)


def _fma(a, b, c):
    return (LD(a) * LD(b) + LD(c)).astype(np.float64)


def _sums(x, z, r_out, d):
    """sum over odd l of canti_l P_l(cos t) / r^(l+1): exact, and in the kernel's FP64 steps with a division."""
    r2, p0, p1 = LD(x) * x + LD(z) * z, LD(1), LD(z) / np.sqrt(LD(x) * x + LD(z) * z)
    r, c, exact = np.sqrt(r2), p1, LD(0)
    f2 = _fma(z, z, x * x)
    q, sc, zs, xs = r_out / f2, 1 / np.sqrt(f2), z / r_out, x / r_out
    s2, u0, u1, sums, nu = _fma(zs, zs, xs * xs), np.zeros_like(x), np.ones_like(x), np.zeros_like(x), [1.0, 1.0]
    for l in range(1, L + 1):
        if l > 1:
            p0, p1 = p1, ((2 * l - 1) * c * p1 - (l - 1) * p0) / l
            nu.append(nu[l - 2] * (l - 1) / l)
        u0, u1 = u1, _fma((2 * l - 1) / l * nu[l - 1] / nu[l] * zs, u1, -(s2 * u0))
        sc = sc * q
        if l % 2:
            exact = exact + LD(_canti(l, d)) * p1 * r ** -(l + 1)
            sums = sums + _canti(l, d) * (u1 * sc * nu[l])
    return exact, sums


def test_tally_of_one_particle_near_the_equator():
    import torch
    assert torch.cuda.is_available()
    from paper_2111_13072_gb300 import build, imrp
    build.build()
    rng = np.random.default_rng(5)
    n, t = 400, math.radians(85.0)
    r = 1.0005 + 0.019 * rng.random(n)
    x, z = np.round(r * math.sin(t) * 2 ** 20) / 2 ** 20, np.round(r * math.cos(t) * 2 ** 20) / 2 ** 20  # r^2 is exact
    q = np.zeros(n)
    with imrp.Sim(imrp.params_from_workload(W)) as sim:
        for k in range(n):
            sim.load(np.array([[x[k], 0.0, z[k]]]), np.zeros((1, 3)))
            q[k] = sim.step(1)[0][0]
        info = sim.info()
    exact, host = _sums(x, z, info.r_out, info.d)
    # one electron: Q = sum / n~. Its two roundings (of -1 / n~ and of the product) are far below the bound
    off = (q.astype(LD) * LD(info.n_tilde) - exact).astype(np.float64)
    best = (host - exact).astype(np.float64)
    assert np.sqrt(np.mean(off ** 2)) <= 1.5 * np.sqrt(np.mean(best ** 2))
