"""The FP64 field kernel of four warps per tile: every particle's field against the oracle at every
degree, at single particles, ragged tiles and sizes around the tile, with both image rules, surface
charge, mobile ions; and against the m = 0 truncation's kernel where the two coincide."""
import numpy as np
import pytest

import oracle
from paper_2111_13072_gb300.inputs import WORKLOADS, workload_state
from parity_metrics import TOL, check_field

pytestmark = pytest.mark.gpu

W = WORKLOADS["fp64_n2e4_l8"]


@pytest.fixture(scope="module")
def imrp():
    import torch
    assert torch.cuda.is_available()
    from paper_2111_13072_gb300 import build, imrp as m
    build.build()
    return m


@pytest.mark.parametrize("L", [1, 2, 4, 8, 12, 16, 24])
@pytest.mark.parametrize("n,si", [(1, 0), (2, 1), (31, 0), (33, 1), (1057, 0)])
def test_every_degree_against_the_oracle(imrp, L, n, si):
    x, v = workload_state(W, N=n)
    p = imrp.params_from_workload(W, N=n, precision=0, l_max=L, self_image=si, drive_kind=1, V_volts=50.0, q_s=3.5)
    with imrp.Sim(p) as sim:
        sim.load(x, v)
        E = sim.field()
    op = oracle.from_physical(W.R_E_m, W.R_D_m, W.eps_D, W.R_out_m, W.n_e_m3, W.T_e_eV, n, L, W.dt, drive_kind=1,
                              V_volts=50.0, width_wpe=W.width_wpe, self_image=si)
    op.q_s = 3.5
    Eo = oracle.field_scan(op, x, u=oracle.drive(op, 0))
    # the ladder factors are rounded to FP32 (2^-24 each): the method's FP64 bound holds with room
    np.testing.assert_allclose(E, Eo, rtol=0, atol=TOL[0] * np.max(np.abs(Eo)))
    assert np.linalg.norm(E - Eo) <= 1e-6 * np.linalg.norm(Eo)


@pytest.mark.parametrize("L", [4, 16])
def test_mobile_ions(imrp, L):
    n, n_e = 2001, 1400
    x, v = workload_state(W, N=n)
    p = imrp.params_from_workload(W, N=n, precision=0, l_max=L)
    with imrp.Sim(p) as sim:
        sim.set_species(n_e, 2.0, 50.0, 200.0)
        sim.load(x, v)
        E = sim.field()
    op = oracle.from_physical(W.R_E_m, W.R_D_m, W.eps_D, W.R_out_m, W.n_e_m3, W.T_e_eV, n, L, W.dt,
                              drive_kind=W.drive_kind, V_volts=W.V_volts, width_wpe=W.width_wpe)
    op.n_tilde, op.n_ion = n_e / (4 * np.pi / 3 * (op.r_out ** 3 - 1)), 200.0
    op.charge = np.concatenate([-np.ones(n_e), np.full(n - n_e, 2.0)])
    op.mass = np.concatenate([np.ones(n_e), np.full(n - n_e, 50.0)])
    check_field(E, oracle.field_scan(op, x, u=oracle.drive(op, 0)), 0, f"ions L={L}")


def test_particles_on_the_axis_match_the_m0_kernel(imrp):
    """On the polar axis only the m = 0 terms act: the full FP64 kernel (diagonal powers of a zero
    direction) gives the truncated kernel's axial field."""
    r = np.linspace(1.05, W.r_out - 0.05, 70)
    x = np.zeros((70, 3))
    x[:, 2] = r * np.where(np.arange(70) % 2 == 0, 1.0, -1.0)
    x = x.astype(np.float32).astype(np.float64)
    E = []
    for m0 in (0, 1):
        p = imrp.params_from_workload(W, N=70, precision=0, l_max=8, m0_only=m0)
        with imrp.Sim(p) as sim:
            sim.load(x, np.zeros_like(x))
            E.append(sim.field())
    np.testing.assert_allclose(E[0][:, 2], E[1][:, 2], rtol=0, atol=1e-6 * np.max(np.abs(E[1])))
