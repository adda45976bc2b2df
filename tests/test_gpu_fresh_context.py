"""A context created on used device memory, in a worker thread, while other contexts have hundreds of steps
queued: its work areas (the sort's totals, the scans' tickets) are in order before its first step, so its
samples and state equal, bit for bit, those of the same instance alone on the GPU."""
import threading

import numpy as np
import pytest

from paper_2111_13072_gb300.inputs import Workload, workload_state

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def mods():
    import torch
    assert torch.cuda.is_available()
    from paper_2111_13072_gb300 import build, imrp
    build.build()
    return torch, imrp


def _soil(torch):
    """Free device memory full of ones, in large blocks and in small ones."""
    blocks = [torch.full((1 << 28,), -1, dtype=torch.int32, device="cuda")]
    blocks += [torch.full((1 << 18,), -1, dtype=torch.int32, device="cuda") for _ in range(64)]
    torch.cuda.synchronize()
    del blocks
    torch.cuda.empty_cache()


def _run(imrp, w, ions, steps):
    x, v = workload_state(w)
    with imrp.Sim(imrp.params_from_workload(w)) as sim:
        if ions:
            n_e = w.N - w.N // 3
            sim.set_species(n_e, 1.0, 50.0, float(2 * n_e - w.N))
        sim.load(x, v)
        q, _ = sim.step(steps)
        return (q, *sim.particles())


@pytest.mark.parametrize("n,prec,ions", [(4097, 1, 0), (100_003, 1, 1), (600_001, 1, 0), (30_001, 0, 1)])
def test_created_beside_queued_work(mods, n, prec, ions):
    torch, imrp = mods
    new = Workload("new", N=n, l_max=4, T_e_eV=2.0, n_e_m3=1e16, precision=prec, seed=n)
    alone = _run(imrp, new, ions, 5)
    busy = []
    try:
        for k in range(16):
            w = Workload(f"busy{k}", N=150_000 + 1000 * k, l_max=8, T_e_eV=3.0, n_e_m3=1e16, precision=1, seed=k)
            s = imrp.Sim(imrp.params_from_workload(w))
            busy.append(s)
            s.load(*workload_state(w))
            s.step(2)
        _soil(torch)
        for s in busy:
            s.step_async(300)
        got = []
        t = threading.Thread(target=lambda: got.extend(_run(imrp, new, ions, 5) for _ in range(3)))
        t.start()
        t.join()
        assert len(got) == 3
        for s in busy:
            s.sync()
    finally:
        for s in busy:
            s.close()
    for out in got:
        for a, b in zip(out, alone):
            np.testing.assert_array_equal(a, b)
