"""The field kernel of two tiles per warp (FP32, degree 12 and up, at least 2^19 particles): every
particle's field against the oracle at its smallest sizes, with whole and ragged last tiles, even
and odd tile counts; mobile ions against the same instance's electron path; a batch that mixes it
with the one-tile kernel; one step against the field it used."""
import numpy as np
import pytest

import oracle
from paper_2111_13072_gb300.inputs import WORKLOADS, Workload, workload_state
from parity_metrics import check_field

pytestmark = pytest.mark.gpu

W = WORKLOADS["fp64_n2e4_l8"]
N0 = 1 << 19


@pytest.fixture(scope="module")
def imrp():
    import torch
    assert torch.cuda.is_available()
    from paper_2111_13072_gb300 import build, imrp as m
    build.build()
    return m


@pytest.mark.parametrize("n,L,si", [(N0 - 1, 12, 0), (N0, 12, 0), (N0 + 1, 16, 0), (N0 + 33, 12, 1), (N0 + 1000, 24, 0)])
def test_every_particle_against_the_oracle(imrp, n, L, si):
    x, v = workload_state(W, N=n)
    p = imrp.params_from_workload(W, N=n, precision=1, l_max=L, drive_kind=1, V_volts=50.0, self_image=si)
    with imrp.Sim(p) as sim:
        sim.load(x, v)
        E = sim.field()
        sim.step(1)
        _, v1 = sim.particles()
    op = oracle.from_physical(W.R_E_m, W.R_D_m, W.eps_D, W.R_out_m, W.n_e_m3, W.T_e_eV, n, L, W.dt, drive_kind=1,
                              V_volts=50.0, width_wpe=W.width_wpe, self_image=si)
    check_field(E, oracle.field_scan(op, x, u=oracle.drive(op, 0)), 1, f"n={n} L={L}")
    # the push used this field: v - (dt / 2) E but for wall hits (rounded once per operation)
    dv = np.linalg.norm(v1 - (v - 0.5 * W.dt * E), axis=1)
    assert np.mean(dv > 1e-6 * np.linalg.norm(v, axis=1).max()) < 0.05


def test_species_flags_without_ions(imrp):
    n = N0 + 77
    x, v = workload_state(W, N=n)
    p = imrp.params_from_workload(W, N=n, precision=1, l_max=12)
    with imrp.Sim(p) as a, imrp.Sim(p) as b:
        a.load(x, v)
        b.set_species(n, 1.0, 100.0, float(n))
        b.load(x, v)
        np.testing.assert_array_equal(a.field(), b.field())


def test_mobile_ions_against_the_oracle(imrp):
    n = N0 + 5
    n_e = n - n // 3
    x, v = workload_state(W, N=n)
    p = imrp.params_from_workload(W, N=n, precision=1, l_max=12)
    with imrp.Sim(p) as sim:
        sim.set_species(n_e, 1.0, 100.0, float(2 * n_e - n))
        sim.load(x, v)
        E = sim.field()
    op = oracle.from_physical(W.R_E_m, W.R_D_m, W.eps_D, W.R_out_m, W.n_e_m3, W.T_e_eV, n, 12, W.dt,
                              drive_kind=W.drive_kind, V_volts=W.V_volts, width_wpe=W.width_wpe)
    op.n_tilde, op.n_ion = n_e / (4 * np.pi / 3 * (op.r_out ** 3 - 1)), float(2 * n_e - n)
    op.charge = np.concatenate([-np.ones(n_e), np.ones(n - n_e)])
    op.mass = np.concatenate([np.ones(n_e), np.full(n - n_e, 100.0)])
    check_field(E, oracle.field_scan(op, x, u=oracle.drive(op, 0)), 1, "ions")


def test_batch_and_autotune_equal_alone(imrp):
    cases = [(N0 + 100, 12), (30000, 12), (N0, 16), (2000, 16)]

    def make(n, L, k):
        w = Workload("p", N=n, l_max=L, T_e_eV=2.0, n_e_m3=1e15, precision=1, seed=k)
        s = imrp.Sim(imrp.params_from_workload(w))
        s.load(*workload_state(w))
        return s

    alone = []
    for k, (n, L) in enumerate(cases):
        with make(n, L, k) as s:
            s.autotune()
            q, _ = s.step(4)
            alone.append((q, s.particles()))
    sims = [make(n, L, k) for k, (n, L) in enumerate(cases)]
    with imrp.Batch(sims) as b:
        b.step(2)
        b.autotune()
        b.step(2)
        b.sync()
    for s, (q0, (x0, v0)) in zip(sims, alone):
        np.testing.assert_array_equal(s.qdiff()[0], q0)
        x, v = s.particles()
        np.testing.assert_array_equal(x, x0)
        np.testing.assert_array_equal(v, v0)
        s.close()
