"""The transform of a recorded series (imrp_admittance) against the plain FP64 sums, at the edges of
its blocks of 32 samples, segments and warps of 32 frequencies.

Tolerance per frequency: each sample enters with a phase of at most w t_max, whose rounding (the
product w dt and its multiple, on both sides) and whose up to 32 chained rotations cost at most
(2 w t_max + 64) units of 2^-52 of the sample; the sum of n terms adds n 2^-53 of their magnitudes at
worst. Y = i w Q / U carries that relative to sum |q_n - q_0| dt and sum |k_n u_n|."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def imrp():
    import torch
    assert torch.cuda.is_available()
    from paper_2111_13072_gb300 import build, imrp as m
    build.build()
    return m


@pytest.mark.parametrize("drive", ["impulse", "pulse"])
@pytest.mark.parametrize("ns,nf", [(8, 3), (31, 32), (32, 33), (33, 1000), (128, 31), (129, 64), (700, 1),
                                   (5001, 257), (20000, 40)])
def test_admittance_matches_plain_sums(imrp, ns, nf, drive):
    nf = max(nf, 3)
    rng = np.random.default_rng(ns)
    dt, first, wmax = 0.05, 0.025, 1.7
    t = dt * np.arange(ns)
    q = rng.standard_normal(ns) + 3.0
    u = np.where(np.arange(ns) == 0, 0.7, 0.0) if drive == "impulse" else np.exp(-0.5 * (t - 0.2) ** 2)
    om, re, im = imrp.admittance(q, u, dt, first, nf, wmax)
    k = np.full(ns, dt)
    k[0] = first
    w = (np.arange(nf) + 1) * (wmax / nf)
    e = np.exp(-1j * (w * dt)[:, None] * np.arange(ns)[None, :])
    dq, ku = q - q[0], k * u
    Q, U = dt * (e @ dq), e @ ku
    np.testing.assert_allclose(om, w, rtol=1e-15)
    Y = 1j * w * Q / U
    eps = (2 * w * t[-1] + 64 + ns) * 2.0 ** -52
    tol = w * eps * (dt * np.sum(np.abs(dq)) / np.abs(U) + np.abs(Q) * np.sum(np.abs(ku)) / np.abs(U) ** 2)
    assert np.all(np.abs(re + 1j * im - Y) <= tol), np.max(np.abs(re + 1j * im - Y) / tol)
