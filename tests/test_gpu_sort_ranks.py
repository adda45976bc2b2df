"""The bucket sort's ranks within its second digit: every edge of its ranges against numpy's stable
argsort of the same keys: one CTA for everything, segments of one bucket and of several (a batch),
with ties, keys so close that a digit overflows (the byte passes), one key for all, clusters that
leave other buckets empty, and buckets that take several rounds; the largest size of the bucket sort
and the first of the global passes."""
import numpy as np
import pytest

from paper_2111_13072_gb300.inputs import maxwellian_shell
from test_gpu_sort import W, _check_two_steps, _state, _ties, radius_keys

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def imrp():
    import torch
    assert torch.cuda.is_available()
    from paper_2111_13072_gb300 import build, imrp as m
    build.build()
    return m


def _point(r):
    """A point at about radius r, its coordinates FP32 values."""
    return (r * np.array([0.42, 0.56, 0.71])).astype(np.float32).astype(np.float64)


def _positions(kind, n, r_out, seed):
    if kind in ("uniform", "narrow"):
        return _state(kind, n, r_out, seed)[0]
    if kind == "ties":
        return _ties(n, r_out, seed)
    rng = np.random.default_rng(seed)
    if kind == "equal":  # one radius exactly: the signed permutations of one point
        s = rng.choice([-1.0, 1.0], size=(n, 3))
        return s * rng.permuted(np.tile(_point(0.4 * r_out + 0.6), (n, 1)), axis=1)
    if kind == "dense":  # nine tenths of the particles in a hundredth of the range of r^2
        x = maxwellian_shell(n, r_out, 0.0, seed)[0]
        i = rng.random(n) < 0.9
        r = np.sqrt(1.0 + (r_out ** 2 - 1.0) * (0.3 + 0.01 * rng.random(n)))
        x[i] *= (r / np.linalg.norm(x, axis=1))[i, None]
        return x.astype(np.float32).astype(np.float64)
    # a cluster of 200 ties per point, three points, amid a uniform shell
    x = maxwellian_shell(n, r_out, 0.0, seed)[0]
    for k in range(3):
        i = rng.choice(n, size=min(200, n // 4), replace=False)
        x[i] = rng.choice([-1.0, 1.0], size=(i.size, 3)) * _point(1.0 + (r_out - 1.0) * (k + 1) / 4)
    return x


CASES = [(n, k, 1) for n in (2, 33, 1000, 4096) for k in ("uniform", "equal")]
CASES += [(4096, "ties", 1), (4096, "narrow", 1), (3000, "clusters", 0), (4097, "uniform", 1), (4097, "equal", 1),
          (20_000, "clusters", 1), (20_000, "narrow", 0), (20_000, "dense", 1),
          (300_000, "dense", 0), (524_289, "dense", 1), (524_288, "ties", 1), (524_289, "clusters", 1),
          (524_289, "narrow", 1), (24_000_000, "uniform", 1), (24_000_001, "uniform", 1)]


@pytest.mark.parametrize("n,kind,prec", CASES)
def test_ranks(imrp, n, kind, prec):
    with imrp.Sim(imrp.params_from_workload(W, N=n, precision=prec)) as sim:
        x = _positions(kind, n, sim.info().r_out, 3)
        sim.load(x, np.zeros_like(x))
        _check_two_steps(sim, x, fp32=prec == 1, steps=1)


def test_ranks_of_segments_of_several_buckets(imrp):
    sizes = [(4097, "equal"), (5000, "ties"), (20_000, "clusters"), (40_000, "narrow"), (60_000, "dense")]
    sims, xs = [], []
    try:
        for k, (n, kind) in enumerate(sizes):
            s = imrp.Sim(imrp.params_from_workload(W, N=n, precision=1, seed=k))
            sims.append(s)
            xs.append(_positions(kind, n, s.info().r_out, 20 + k))
            s.load(xs[-1], np.zeros_like(xs[-1]))
        b = imrp.Batch(sims)
        b.step(1)
        b.sync()
        for s, x in zip(sims, xs):
            ids = s.checkpoint()[2]
            want = np.argsort(radius_keys(x, s.info().r_out, True), kind="stable").astype(np.uint32)
            np.testing.assert_array_equal(ids, want)
        b.close()
    finally:
        for s in sims:
            s.close()
