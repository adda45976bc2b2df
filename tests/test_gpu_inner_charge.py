"""The inner charge of the l = 0 term (ions inside minus electrons inside plus Q_S), which the mixed
path forms in FP32 pairs: the difference of two counts of size N must keep FP32 accuracy, in narrow
and wide shells, with and without a surface charge. At l_max = 1 it dominates the field."""
import numpy as np
import pytest

import oracle
from paper_2111_13072_gb300.inputs import Workload, workload_state

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def imrp():
    import torch
    assert torch.cuda.is_available()
    from paper_2111_13072_gb300 import build, imrp as m
    build.build()
    return m


@pytest.mark.parametrize("outer_R,n", [(1.3, 33), (2.0, 5000), (10.0, 40000), (30.0, 3001)])
@pytest.mark.parametrize("q_s", [0.0, -12345.678])
def test_radial_field_of_the_inner_charge(imrp, outer_R, n, q_s):
    """Tolerance: the oracle's FP64 field, FP32 rounding of the inner charge and of its scale
    (a few 2^-24) on top of the mixed path's error of the l = 1 terms: 1e-5 of the rms field."""
    w = Workload("inner", N=n, l_max=1, T_e_eV=2.0, n_e_m3=1e15, outer_R=outer_R, drive_kind=2, precision=1, seed=n)
    x, v = workload_state(w)
    p = imrp.params_from_workload(w, q_s=q_s)
    with imrp.Sim(p) as sim:
        sim.load(x, v)
        E = sim.field()
    op = oracle.from_physical(w.R_E_m, w.R_D_m, w.eps_D, w.R_out_m, w.n_e_m3, w.T_e_eV, n, 1, w.dt, drive_kind=2,
                              seed=w.seed)
    op.q_s = q_s
    Eo = oracle.field_scan(op, x)
    assert np.linalg.norm(E - Eo) <= 1e-5 * np.linalg.norm(Eo)
    assert np.max(np.abs(E - Eo)) <= 1e-4 * np.max(np.abs(Eo))
