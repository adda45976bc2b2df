"""A tuned launch shape belongs to the field kernel and size it was measured for: loads that another
kernel or shape serves run in the shape of an untuned context. Shapes are read from a trace of the
launches (blocks of the field kernels)."""
import json

import pytest

from paper_2111_13072_gb300.inputs import Workload, workload_state

pytestmark = pytest.mark.gpu

N_PAIR = 1 << 19  # the smallest of the pair kernel


@pytest.fixture(scope="module")
def imrp():
    import torch
    assert torch.cuda.is_available()
    from paper_2111_13072_gb300 import build, imrp as m
    build.build()
    from torch.profiler import ProfilerActivity, profile
    with profile(activities=[ProfilerActivity.CUDA]):  # a process' first trace can miss its first launches
        torch.ones(8, device="cuda").sum().item()
    return m


def work(n, precision=1):
    return Workload("tuned", N=n, l_max=12, T_e_eV=2.0, n_e_m3=1e15, seed=7, precision=precision)


def load(sim, n):
    w = work(n)
    sim.load(*workload_state(w))


def field_blocks(call, tmp_path):
    """{kernel: threads per block} of the field kernels that call() launches."""
    from torch.profiler import ProfilerActivity, profile
    with profile(activities=[ProfilerActivity.CUDA]) as prof:
        call()
    path = tmp_path / "trace.json"
    prof.export_chrome_trace(str(path))
    out = {}
    for e in json.loads(path.read_text())["traceEvents"]:
        if e.get("cat") == "kernel" and "k_field" in e["name"]:
            name = e["name"].split("k_field")[1].split("<")[0]
            out.setdefault("k_field" + name, set()).add(e["args"]["block"][0])
    return out


@pytest.mark.parametrize("n", [100003, 20000])
def test_load_for_another_kernel_takes_its_own_shape(imrp, tmp_path, n):
    p = imrp.params_from_workload(work(N_PAIR))
    with imrp.Sim(p) as plain, imrp.Sim(p) as tuned:
        load(plain, n)
        want = field_blocks(lambda: plain.step(1), tmp_path)
        assert set(want) == {"k_field"}
        load(tuned, N_PAIR)
        wpb, _ = tuned.autotune()
        assert field_blocks(lambda: tuned.step(1), tmp_path) == {"k_field_pair": {32 * wpb}}
        load(tuned, n)
        assert field_blocks(lambda: tuned.step(1), tmp_path) == want
        load(tuned, N_PAIR)  # the tuned load again
        assert field_blocks(lambda: tuned.step(1), tmp_path) == {"k_field_pair": {32 * wpb}}


def test_fp64_kernel_has_one_shape(imrp, tmp_path):
    w = work(3001, precision=0)
    with imrp.Sim(imrp.params_from_workload(w)) as sim:
        sim.load(*workload_state(w))
        assert [sim.autotune()[0] for _ in range(4)] == [4] * 4
        assert field_blocks(lambda: sim.step(1), tmp_path) == {"k_field_team": {128}}


def test_batch_without_the_one_tile_kernel_tunes_nothing(imrp, tmp_path):
    """Two instances of the pair kernel leave no shape to choose; when one takes fewer particles, its
    batched launch has the shape of an untuned batch."""
    n = 100003
    p = imrp.params_from_workload(work(N_PAIR))
    with imrp.Sim(p) as a, imrp.Sim(p) as b, imrp.Sim(p) as c, imrp.Sim(p) as d:
        for s in (a, b, c):
            load(s, N_PAIR)
        load(d, n)
        a.autotune()
        blocks = []
        with imrp.Batch([c, d]) as plain, imrp.Batch([a, b]) as tuned:
            tuned.autotune()
            load(b, n)
            for batch in (plain, tuned):
                def two():
                    batch.step(2)
                    batch.sync()
                blocks.append(field_blocks(two, tmp_path))
        assert set(blocks[0]) == {"k_field_pair_batch", "k_field_batch"}
        assert blocks[1] == blocks[0]
