"""Buckets of the radius sort that hold far more particles than their mean, in every form that takes them: placed
in ranges, byte passes with few equal keys and with many, a byte that all keys share. The permutation against
numpy's stable argsort of the same keys, and the time: such a bucket's work grows with its keys, not with
their square."""
import numpy as np
import pytest

from paper_2111_13072_gb300.inputs import maxwellian_shell
from test_gpu_sort import W, _check_two_steps

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def imrp():
    import torch
    assert torch.cuda.is_available()
    from paper_2111_13072_gb300 import build, imrp as m
    build.build()
    return m


def _dense(n, r_out, frac, seed):
    """Nine tenths of the particles in `frac` of the range of r^2."""
    rng = np.random.default_rng(seed)
    x = maxwellian_shell(n, r_out, 0.0, seed)[0]
    i = rng.random(n) < 0.9
    r = np.sqrt(1.0 + (r_out ** 2 - 1.0) * (0.3 + frac * rng.random(n)))
    x[i] *= (r / np.linalg.norm(x, axis=1))[i, None]
    return x.astype(np.float32).astype(np.float64)


def _shells(n, r_out, k, seed):
    """All particles on k radii, to FP32 rounding: many keys per byte value, and ties."""
    rng = np.random.default_rng(seed)
    x = maxwellian_shell(n, r_out, 0.0, seed)[0]
    x *= ((1.0 + (r_out - 1.0) * (rng.integers(0, k, n) + 0.5) / k) / np.linalg.norm(x, axis=1))[:, None]
    return x.astype(np.float32).astype(np.float64)


@pytest.mark.parametrize("n,form,arg", [(5_000, "dense", 0.01), (20_000, "dense", 0.03), (20_000, "dense", 0.001),
                                        (300_000, "dense", 0.01), (300_000, "dense", 0.003), (300_000, "dense", 0.0005),
                                        (600_000, "dense", 0.03), (600_000, "dense", 1e-5), (4_000, "shells", 3),
                                        (300_000, "shells", 30), (600_000, "shells", 1), (600_000, "shells", 500)])
@pytest.mark.parametrize("prec", [0, 1])
def test_permutation(imrp, n, form, arg, prec):
    with imrp.Sim(imrp.params_from_workload(W, N=n, precision=prec)) as sim:
        x = (_dense if form == "dense" else _shells)(n, sim.info().r_out, arg, 7)
        sim.load(x, np.zeros_like(x))
        _check_two_steps(sim, x, fp32=prec == 1, steps=1)


def test_time_grows_with_the_keys(imrp):
    """N = 3e5 with nine tenths in 0.03 of the range (some nine buckets) and in 0.003 (about one, ten times as full):
    at most ten times as long."""
    ms = []
    with imrp.Sim(imrp.params_from_workload(W, N=300_000, precision=1)) as sim:
        for frac in (0.03, 0.003):
            x = _dense(300_000, sim.info().r_out, frac, 7)
            best = np.inf
            for _ in range(4):
                sim.load(x, np.zeros_like(x))
                best = min(best, sim.profile_steps(1)[imrp.STAGES[0]])
            ms.append(best)
    assert ms[1] <= 10 * ms[0], ms
