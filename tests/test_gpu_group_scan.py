"""The group scan in one kernel and in two: fields, Q_diff and (with mobile ions) the inner charge against
the oracle at the edges of a run of 4 groups, of a segment of 32 and of the rule's 320 groups of 1024.
Particles whose 32-bit radius key another one shares (a few of 3e5) are left out: the library orders those
by slot, the oracle by radius, and the charge inside differs by one of them."""
import numpy as np
import pytest

import oracle
from paper_2111_13072_gb300.inputs import WORKLOADS, workload_state
from test_gpu_sort import radius_keys

pytestmark = pytest.mark.gpu

W = WORKLOADS["fp64_n2e4_l8"]


@pytest.fixture(scope="module")
def imrp():
    import torch
    assert torch.cuda.is_available()
    from paper_2111_13072_gb300 import build, imrp as m
    build.build()
    return m


@pytest.mark.parametrize("n", [1024, 4097, 32 * 1024, 32 * 1024 + 1, 36 * 1024 + 5, 65 * 1024, 320 * 1024, 320 * 1024 + 1])
@pytest.mark.parametrize("ions", [0, 1])
def test_against_the_oracle(imrp, n, ions):
    L, n_e = 4, n - n // 3 if ions else n
    x, v = workload_state(W, N=n)
    p = imrp.params_from_workload(W, N=n, precision=0, l_max=L, drive_kind=1, V_volts=50.0)
    op = oracle.from_physical(W.R_E_m, W.R_D_m, W.eps_D, W.R_out_m, W.n_e_m3, W.T_e_eV, n, L, W.dt, drive_kind=1,
                              V_volts=50.0, width_wpe=W.width_wpe)
    if ions:
        op.n_tilde, op.n_ion = n_e / (4 * np.pi / 3 * (op.r_out ** 3 - 1)), float(2 * n_e - n)
        op.charge = np.concatenate([-np.ones(n_e), np.ones(n - n_e)])
        op.mass = np.concatenate([np.ones(n_e), np.full(n - n_e, 50.0)])
    with imrp.Sim(p) as sim:
        if ions:
            sim.set_species(n_e, 1.0, 50.0, float(2 * n_e - n))
        sim.load(x, v)
        E = sim.field()
        keys = radius_keys(x, sim.info().r_out, False)
    Eo = oracle.field_scan(op, x, u=oracle.drive(op, 0))
    _, where, count = np.unique(keys, return_inverse=True, return_counts=True)
    alone = count[where] == 1
    assert np.count_nonzero(~alone) <= 4 + n * n / 2.0 ** 31
    E, Eo = E[alone], Eo[alone]
    # FP64 sums of FP32-rounded ladder factors (2^-24 each): as in the tests of the FP64 field kernel
    assert np.linalg.norm(E - Eo) <= 1e-6 * np.linalg.norm(Eo)
    np.testing.assert_allclose(E, Eo, rtol=0, atol=1e-5 * np.max(np.abs(Eo)))
