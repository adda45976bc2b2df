"""The moments kernel's column ranges (small instances) and particles per thread, and the field
kernel's CTA shapes: every particle's field against the oracle at sizes around which the choices
change, and a context whose particle count changes keeps giving what a fresh one gives."""
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


def _field(imrp, n, L, prec):
    x, v = workload_state(W, N=n)
    p = imrp.params_from_workload(W, N=n, precision=prec, l_max=L)
    with imrp.Sim(p) as sim:
        sim.load(x, v)
        return x, sim.field()


# one column per range and fewer ranges than columns; 16 and 4 FP64 particles per thread (100 blocks);
# several, two and one range per block
@pytest.mark.parametrize("n,L,prec", [(257, 24, 0), (257, 24, 1), (5000, 1, 0), (5000, 1, 1), (20000, 12, 0),
                                      (101376, 4, 0), (101377, 4, 0), (93185, 8, 1), (310273, 2, 1),
                                      (466944, 2, 1), (466945, 2, 1)])
def test_field_at_the_edges_of_the_launch_shapes(imrp, n, L, prec):
    x, E = _field(imrp, n, L, prec)
    op = oracle.from_physical(W.R_E_m, W.R_D_m, W.eps_D, W.R_out_m, W.n_e_m3, W.T_e_eV, n, L, W.dt,
                              drive_kind=W.drive_kind, V_volts=W.V_volts, width_wpe=W.width_wpe, seed=W.seed)
    check_field(E, oracle.field_scan(op, x, u=oracle.drive(op, 0)), prec, f"n={n} L={L}")


@pytest.mark.parametrize("prec", [0, 1])
def test_reloads_of_other_sizes(imrp, prec):
    sizes = (20001, 300, 5000)
    p = imrp.params_from_workload(W, N=max(sizes), precision=prec, l_max=8)
    with imrp.Sim(p) as sim:
        for n in sizes:
            x, v = workload_state(W, N=n)
            sim.load(x, v)
            sim.step(3)
            got = sim.particles()
            with imrp.Sim(imrp.params_from_workload(W, N=n, precision=prec, l_max=8)) as fresh:
                fresh.load(x, v)
                fresh.step(3)
                for a, b in zip(got, fresh.particles()):
                    np.testing.assert_array_equal(a, b)


@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("n", [1, 257, 393215, 393216, 500001])
def test_read_back_in_id_order(imrp, prec, n):
    """imrp_get_particles (scattering small states, gathering large ones) against the checkpoint's
    storage order and ids, exactly, after steps that permuted the storage."""
    x, v = workload_state(W, N=n)
    with imrp.Sim(imrp.params_from_workload(W, N=n, precision=prec, l_max=1)) as sim:
        sim.load(x, v)
        sim.step(2)
        xs, vs = sim.particles()
        xc, vc, ids, _ = sim.checkpoint()
    np.testing.assert_array_equal(xs[ids], xc)
    np.testing.assert_array_equal(vs[ids], vc)
