"""Error flags stand in page-locked host memory, where atomics go over the host link one after the other. A
load with every particle in error takes about as long as a good one, and still tells what is wrong."""
import time

import pytest

from paper_2111_13072_gb300.inputs import Workload, workload_state

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def imrp():
    import torch
    assert torch.cuda.is_available()
    from paper_2111_13072_gb300 import build, imrp as m
    build.build()
    return m


def test_load_of_bad_particles_takes_no_longer(imrp):
    """With an atomic per warp a bad load of 8e6 took 2.2 times a good one. Bound: a quarter of what was added."""
    w = Workload("bad", N=8000000, l_max=4, T_e_eV=2.0, n_e_m3=1e15, precision=1, seed=1)
    x, v = workload_state(w)
    inside = 0.25 * x  # within the probe
    inside[0] = float("nan")
    with imrp.Sim(imrp.params_from_workload(w)) as sim:
        def load(pos):
            t = time.perf_counter()
            try:
                sim.load(pos, v)
                err = ""
            except imrp.IMRPError as e:
                err = str(e)
            return time.perf_counter() - t, err
        good = [load(x) for _ in range(7)]
        bad = [load(inside) for _ in range(7)]
        assert {e for _, e in good} == {""}
        assert all("non-finite" in e for _, e in bad)
        assert min(t for t, _ in bad) <= 1.3 * min(t for t, _ in good)
        inside[0] = x[0]
        inside[-1] = x[-1]
        assert "outside" in load(inside)[1]
        inside[:-1] = x[:-1]
        assert load(inside)[1] == ""
