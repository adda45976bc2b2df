"""FP32 instances of at most 1024 particles sum the image pairs of their own tile directly, in a field
kernel of their own: every particle's field against the oracle at the edges of the tile and of the rule,
with both image rules and in the m = 0 truncation; alone and in a batch (whose kernel takes the pairs one
at a time) the same bits."""
import numpy as np
import pytest

import oracle
from paper_2111_13072_gb300.inputs import WORKLOADS, workload_state
from parity_metrics import check_field

pytestmark = pytest.mark.gpu

W = WORKLOADS["fp64_n2e4_l8"]


@pytest.fixture(scope="module")
def imrp():
    import torch
    assert torch.cuda.is_available()
    from paper_2111_13072_gb300 import build, imrp as m
    build.build()
    return m


@pytest.mark.parametrize("L,m0", [(1, 1), (2, 0), (8, 0), (8, 1), (16, 0), (24, 0)])
@pytest.mark.parametrize("n,si", [(1, 0), (2, 1), (33, 0), (991, 1), (1024, 0), (1025, 1)])
def test_field_against_the_oracle(imrp, L, m0, n, si):
    x, v = workload_state(W, N=n)
    p = imrp.params_from_workload(W, N=n, precision=1, l_max=L, self_image=si, m0_only=m0, drive_kind=1, V_volts=50.0)
    with imrp.Sim(p) as sim:
        sim.load(x, v)
        E = sim.field()
    op = oracle.from_physical(W.R_E_m, W.R_D_m, W.eps_D, W.R_out_m, W.n_e_m3, W.T_e_eV, n, L, W.dt, drive_kind=1,
                              V_volts=50.0, width_wpe=W.width_wpe, self_image=si, m0_only=m0)
    check_field(E, oracle.field_scan(op, x, u=oracle.drive(op, 0)), 1, f"N={n} L={L} m0={m0} si={si}")


def test_alone_and_in_a_batch(imrp):
    sizes = [(991, 0), (1024, 1), (40, 0), (3001, 0)]
    out = []
    for batched in (False, True):
        sims = [imrp.Sim(imrp.params_from_workload(W, N=n, precision=1, l_max=8, self_image=si)) for n, si in sizes]
        try:
            for s, (n, _) in zip(sims, sizes):
                s.load(*workload_state(W, N=n))
            if batched:
                b = imrp.Batch(sims)
                b.step(2)
                b.sync()
                b.close()
            else:
                for s in sims:
                    s.step(2)
            out.append([s.particles() for s in sims])
        finally:
            for s in sims:
                s.close()
    for (xa, va), (xb, vb) in zip(*out):
        np.testing.assert_array_equal(xa, xb)
        np.testing.assert_array_equal(va, vb)
