"""The calls of this library that its speed is measured on.

Each case is a call (or a short run of calls) that a program using the library makes, through the
public entry points of ``include/imrp.h`` and their ctypes binding: stepping loaded instances of the
sizes, degrees, precisions and wall rules that the library is used with, the field evaluation
without allocation, a batch of uneven instances, a streamed load with the steps on it, and the
transform of a recorded run into its admittance. ``exact`` holds the same mathematics in plain
FP64 torch operations, written from the definitions alone.

A step case's pass takes the next `steps` steps of a loaded run and reads back what a program keeps
of them: the Q_diff and drive samples and the state. The entry points hand all numbers over as FP64;
a mixed-precision run holds its state in FP32, so its results are kept as FP32 snapshots (the values
themselves for the state). A pass has few steps, so that one rounding seldom puts a particle on the
other side of a wall (many particles) or of a neighbour's radius (few particles of much charge).
"""
import ctypes
import math

import numpy as np
import torch

from paper_2111_13072_gb300 import imrp
from paper_2111_13072_gb300.inputs import Workload

# --------------------------------------------------------------------------- cases


def listed():
    return [
        # a host program that owns all device memory asks for the field of a small particle set:
        # the smallest call, bound by launches
        dict(name="noalloc_mixed_n1000_l8", kind="noalloc", precision=1, N=1000, l_max=8),
        # a small run (a ragged number of tiles) next to others or in a parameter scan
        dict(name="steps_mixed_n3001_l8", kind="steps", precision=1, N=3001, l_max=8, steps=4),
        # the small FP64 workload: the reference precision at its usual size
        dict(name="steps_fp64_n20000_l8", kind="steps", precision=0, N=20000, l_max=8, steps=20),
        # the smallest request of the serving workload
        dict(name="steps_mixed_n100003_l16", kind="steps", precision=1, N=100003, l_max=16, steps=8),
        # the headline workload
        dict(name="steps_mixed_n2000000_l16", kind="steps", precision=1, N=2000000, l_max=16, steps=4),
        # the largest workload (40 Debye lengths of plasma, l_max = 24)
        dict(name="steps_mixed_n16000000_l24", kind="steps", precision=1, N=16000000, l_max=24, steps=4),
        # FP64 at the headline degree: what the mixed path is compared with
        dict(name="steps_fp64_n250001_l16", kind="steps", precision=0, N=250001, l_max=16, steps=3),
        # the paper's own truncation and geometry (l <= 1, m = 0, 1 < r < 10, one kick, dt = 0.01)
        dict(name="paper_mixed_n500000_l1", kind="paper", precision=1, N=500000, l_max=1, steps=20),
        # mobile ions as super-particles beside the electrons
        dict(name="ions_mixed_n300001_l8", kind="ions", precision=1, N=300001, l_max=8, steps=8),
        # an ensemble of uneven instances stepped as one batch
        dict(name="batch_mixed_16", kind="batch", precision=1, instances=16, n_lo=10000, n_hi=1000000, draw_seed=3,
             steps=4),
        # a program that feeds a new particle set, steps it and reads it back (absorbing wall, collisions)
        dict(name="stream_mixed_n700001_l12", kind="stream", precision=1, N=700001, l_max=12, steps=4),
        # the spectrum of a long run: the transform of its series at 1000 frequencies
        dict(name="spectrum_ns20000_nf1000", kind="spectrum", ns=20000, nf=1000),
    ]


DEGREES = (1, 2, 4, 8, 12, 16, 24)


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _steps_of(n):
    return 4 if n >= 700000 or n < 10000 else 8


def draw(rng):
    kind = rng.choice(["steps"] * 5 + ["fp64"] * 2 + ["noalloc", "paper", "ions", "batch", "stream", "spectrum"])
    if kind == "noalloc":
        return dict(kind=kind, precision=rng.choice((0, 1)), N=_log(rng, 200, 16384), l_max=rng.choice((4, 8, 12, 16)))
    if kind == "spectrum":
        return dict(kind=kind, ns=_log(rng, 2000, 20000), nf=rng.choice((500, 800, 1000)))
    if kind == "batch":
        return dict(kind=kind, precision=1, instances=rng.randint(4, 16), n_lo=10000, n_hi=1000000,
                    draw_seed=rng.randint(10, 9999), steps=4)
    if kind == "fp64":
        n = _log(rng, 1000, 300000)
        return dict(kind="steps", precision=0, N=n, l_max=rng.choice((4, 8, 12, 16)), steps=5 if n > 50000 else 20)
    if kind == "paper":
        return dict(kind=kind, precision=1, N=_log(rng, 100000, 1000000), l_max=1, steps=20)
    n = _log(rng, 1000, 4000000) if kind == "steps" else _log(rng, 50000, 1000000)
    return dict(kind=kind, precision=1, N=n, l_max=rng.choice((8, 12, 16, 24) if kind == "steps" else (4, 8, 12)),
                steps=_steps_of(n))


# --------------------------------------------------------------------------- inputs

ION_MASS = 100.0


def _workload(case, seed):
    """Physical configuration of a single-instance case."""
    kind, n, L = case["kind"], case["N"], case["l_max"]
    kw = dict(N=n, l_max=L, precision=case["precision"], seed=seed)
    if kind == "paper":
        return Workload("paper", T_e_eV=3.0, n_e_m3=1e15, R_E_m=3e-3, R_D_m=4e-3, outer_R=10.0, dt=0.01, drive_kind=1,
                        V_volts=289.0, m0_only=1, **kw)
    if kind == "ions":
        return Workload("ions", T_e_eV=5.0, n_e_m3=1e15, drive_kind=1, V_volts=50.0, **kw)
    if kind == "stream":
        return Workload("stream", T_e_eV=3.0, n_e_m3=1e16, wall_rule=2, drive_kind=1, V_volts=10.0, **kw)
    if L == 24:
        return Workload("large", T_e_eV=2.0, n_e_m3=1e16, outer_debye=40.0, **kw)
    if case["precision"] == 0 or n < 50000:
        return Workload("small", T_e_eV=2.0, n_e_m3=1e15, **kw)
    return Workload("mixed", T_e_eV=3.0, n_e_m3=1e16, **kw)


def _nu(case):
    return 0.1 if case["kind"] == "stream" else 0.0


def _electrons(case):
    return case["N"] - case["N"] // 3 if case["kind"] == "ions" else case["N"]


def _shell(n, r_out, sigma_v, seed, n_slow=0):
    """Uniform Maxwellian shell, FP32-representable, on the current CUDA device: x, v [n, 3] FP64.
    The last n_slow particles are ions as hot as the electrons."""
    g = torch.Generator(device="cuda").manual_seed(int(seed))
    lo, hi = 1.0 + 1e-6, r_out * (1.0 - 1e-6)
    r = (lo ** 3 + torch.rand(n, generator=g, device="cuda", dtype=torch.float64) * (hi ** 3 - lo ** 3)) ** (1.0 / 3.0)
    d = torch.randn((n, 3), generator=g, device="cuda", dtype=torch.float64)
    d /= torch.linalg.norm(d, dim=1, keepdim=True)
    x = (d * r[:, None]).float().double()
    rr = torch.linalg.norm(x, dim=1)
    x = torch.where(((rr < lo) | (rr > hi))[:, None], (x / rr[:, None] * rr.clamp(lo, hi)[:, None]).float().double(), x)
    v = torch.randn((n, 3), generator=g, device="cuda", dtype=torch.float64) * sigma_v
    if n_slow:
        v[n - n_slow:] /= math.sqrt(ION_MASS)
    return x.contiguous(), v.float().double().contiguous()


def _inputs(case, seed):
    w = _workload(case, seed)
    return (w,) + _shell(w.N, w.r_out, w.sigma_v, seed, case["N"] - _electrons(case))


def _batch_cases(case):
    """The instances of a batch: N log-uniform, l_max of 8, 12 and 16."""
    rng = np.random.default_rng(case["draw_seed"])
    return [dict(kind="steps", precision=case["precision"], steps=case["steps"], l_max=int(rng.choice((8, 12, 16))),
                 N=int(round(math.exp(rng.uniform(math.log(case["n_lo"]), math.log(case["n_hi"]))))))
            for _ in range(case["instances"])]


def _series(case, seed):
    """A recorded run: the drive of the Gaussian pulse, a damped response with noise, dt = 0.05."""
    rng = np.random.default_rng(seed)
    t = 0.05 * np.arange(case["ns"])
    u = 2e-4 * np.exp(-0.5 * ((t - 8.0) / 2.0) ** 2)
    b, c = rng.uniform(0.04, 0.1), rng.uniform(0.4, 0.7)
    tau = np.maximum(t - 8.0, 0.0)
    q = 1e-4 * np.exp(-b * tau) * np.sin(c * tau) + 1e-6 * rng.standard_normal(t.size) + rng.uniform(-1e-4, 1e-4)
    return q, u


# --------------------------------------------------------------------------- passes


def _pinned(t):
    return torch.empty(t.shape, dtype=t.dtype, pin_memory=True).copy_(t)


def _new_sim(case, w):
    sim = imrp.Sim(imrp.params_from_workload(w, nu_coll=_nu(case)))
    if case["kind"] == "ions":
        n_e = _electrons(case)
        sim.set_species(n_e, 1.0, ION_MASS, float(2 * n_e - w.N))
    return sim


class _Run:
    """A loaded instance with the buffers that a program reads its state back into."""

    def __init__(self, case, seed, load=True):
        self.w, x, v = _inputs(case, seed)
        self.case, self.mixed = case, case["precision"] == 1
        self.sim = _new_sim(case, self.w)
        self.x, self.v = _pinned(x), _pinned(v)
        torch.cuda.synchronize()
        if load:
            self.sim.load_ptr(self.x.data_ptr(), self.v.data_ptr(), self.w.N)
        if not load or not self.mixed:
            self.xo, self.vo = torch.empty_like(self.x, pin_memory=True), torch.empty_like(self.v, pin_memory=True)
        else:
            self.xo, self.vo = self.x, self.v  # the inputs are loaded: their buffers take the state
        if self.mixed:
            self.x32 = torch.empty(self.x.shape, dtype=torch.float32)
            self.v32 = torch.empty(self.v.shape, dtype=torch.float32)
        self.q = torch.zeros(case["steps"], dtype=torch.float64, pin_memory=True)

    def state(self):
        pd = ctypes.POINTER(ctypes.c_double)
        rc = imrp.load_library().imrp_get_particles(self.sim._h, ctypes.cast(self.xo.data_ptr(), pd),
                                                    ctypes.cast(self.vo.data_ptr(), pd))
        if rc != 0:
            raise imrp.IMRPError(rc, "imrp_get_particles")
        return (self.x32.copy_(self.xo), self.v32.copy_(self.vo)) if self.mixed else (self.xo, self.vo)

    def samples(self, q):
        return q.astype(np.float32) if self.mixed else q


class _Batch:
    def __init__(self, case, seed):
        self.runs = [_Run(c, 1000 * seed + k) for k, c in enumerate(_batch_cases(case))]
        self.batch = imrp.Batch([r.sim for r in self.runs])

    def __del__(self):  # the batch goes before the instances that it steps
        self.batch.close()


def prepare(case, seed):
    kind = case["kind"]
    if kind == "spectrum":
        return dict(case=case, series=_series(case, seed))
    if kind == "batch":
        return dict(case=case, batch=_Batch(case, seed))
    if kind == "noalloc":
        w, x, _ = _inputs(case, seed)
        return dict(case=case, n=w.N, x=x, E=torch.zeros_like(x), params=imrp.params_from_workload(w))
    return dict(case=case, run=_Run(case, seed, load=kind != "stream"))


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "spectrum":
        q, u = state["series"]
        return imrp.admittance(q, u, 0.05, 0.025, case["nf"], 2.0)
    if kind == "noalloc":
        s = torch.cuda.current_stream().cuda_stream
        imrp.field_noalloc(state["params"], state["x"].data_ptr(), state["n"], 0, state["E"].data_ptr(), s)
        return state["E"].float() if case["precision"] == 1 else state["E"]
    if kind == "batch":
        b = state["batch"]
        b.batch.step(case["steps"])
        b.batch.sync()
        out = []
        for r in b.runs:
            done = r.sim.info().step
            out.append((r.samples(r.sim.qdiff(done - case["steps"], case["steps"])[0]),) + r.state())
        return out
    r = state["run"]
    if kind == "stream":
        r.sim.load_async_ptr(r.x.data_ptr(), r.v.data_ptr(), r.w.N)
        r.sim.step_async(case["steps"])
        r.sim.copy_qdiff_async(0, case["steps"], r.q.data_ptr())
        x, v = r.state()  # waits for the work above
        return r.samples(r.q.numpy()), x, v
    q, u = r.sim.step(case["steps"])
    return (r.samples(q), u) + r.state()


# --------------------------------------------------------------------------- work


def _step_work(case):
    n, L, es = case["N"], case["l_max"], 4 if case["precision"] == 1 else 8
    k = 3 * L if case["kind"] == "paper" else (L + 1) ** 2  # harmonics per particle
    return 2 * 6 * es * n, 24 * k * n


def work(case):
    """Bytes: the particle state read and written once per step, the host copies once per pass. Flops: 24 per
    harmonic (of both families and the gradient) and particle, the count of the mathematics."""
    kind = case["kind"]
    if kind == "spectrum":
        return dict(bytes=16.0 * case["ns"] + 24.0 * case["nf"], flops=12.0 * case["ns"] * case["nf"])
    if kind == "batch":
        parts = [work(c) for c in _batch_cases(case)]
        return dict(bytes=sum(p["bytes"] for p in parts), flops=sum(p["flops"] for p in parts))
    if kind == "noalloc":
        return dict(bytes=48.0 * case["N"], flops=float(_step_work(case)[1]))
    b, f = _step_work(case)
    io = 48.0 * case["N"] * (2 if kind == "stream" else 1)
    return dict(bytes=float(b * case["steps"]) + io, flops=float(f * case["steps"]))


# --------------------------------------------------------------------------- 64-bit values


def _coefficients(w, L):
    """f_l of the image term and the coefficient of r^-(l+1) P_l in Psi_anti (odd l)."""
    d, eps = 1.0 - w.R_E_m / w.R_D_m, w.eps_D
    f, psi = [0.0] * (L + 1), [0.0] * (L + 1)
    for l in range(1, L + 1):
        x = (1.0 - d) ** (2 * l + 1)
        f[l] = (l * (eps - 1) + (l + eps + l * eps) * x) / ((l + 1 + l * eps) + (l + 1) * (eps - 1) * x)
        if l % 2:
            k = (l + 1) // 2
            c = (-1.0) ** (k + 1) * 0.5 ** (k + 1) * (4 * k - 1) / math.factorial(k)
            for j in range(2 * k - 3, 1, -2):
                c *= j
            psi[l] = c * (2 * l + 1) * eps * (1 - d) ** (l + 1) / ((l + 1) * (eps - 1) * x + l * eps + l + 1)
    return f, psi


def _before(t):
    """Exclusive prefix sums."""
    return torch.cumsum(t, 0) - t


def _after(t):
    """Exclusive suffix sums."""
    return torch.flip(_before(torch.flip(t, (0,))), (0,))


def _field(w, x, charge, n_tilde, n_ion, q_s, u):
    """E at every particle, and sum_i q_i Psi_anti(x_i): in radius order, the pairs' terms
    r_<^l / r_>^(l+1) P_l(cos g) - f_l P_l(cos g) / (r r')^(l+1) separate into sums over the inner, the outer
    and the other particles of q times the solid harmonics (l <= l_max; m = 0 alone with m0_only)."""
    L, r_out = w.l_max, w.r_out
    f, psi = _coefficients(w, L)
    r = torch.linalg.norm(x, dim=1)
    order = torch.argsort(r, stable=True)
    r, q = r[order], charge[order]
    xs = x[order]
    X, Y, Z = xs[:, 0], xs[:, 1], xs[:, 2]
    rho = torch.sqrt(X * X + Y * Y)
    ct, st = Z / r, rho / r
    cp, sp = X / rho, Y / rho
    rs = r / r_out  # regular harmonics in r / r_out: no overflow at any degree
    g_r, g_t, g_p = torch.zeros_like(r), torch.zeros_like(r), torch.zeros_like(r)  # gradient of the pair potential
    tally = torch.zeros((), dtype=torch.float64, device=x.device)
    pmm = torch.ones_like(r)  # sqrt((l-m)!/(l+m)!) P_l^m at l = m, without the sign (it cancels)
    cm, sm = torch.ones_like(r), torch.zeros_like(r)  # cos and sin of m phi
    for m in range(0, 1 if w.m0_only else L + 1):
        if m > 0:
            pmm = pmm * st * math.sqrt((2 * m - 1) / (2 * m))
            cm, sm = cm * cp - sm * sp, sm * cp + cm * sp
        p1, p0 = pmm, torch.zeros_like(r)
        for l in range(m, L + 1):
            if l > m:
                a = (2 * l - 1) / math.sqrt((l + m) * (l - m))
                b = math.sqrt((l + m - 1) * (l - m - 1) / ((l + m) * (l - m)))
                p1, p0 = a * ct * p1 - b * p0, p1
            if l == 0:
                continue
            dp = (l * ct * p1 - (math.sqrt((l + m) * (l - m)) * p0 if l > m else 0.0)) / st  # d/d theta
            reg, irr = rs ** l, r ** -(l + 1)
            scale = (2.0 if m else 1.0)
            fac = r_out ** l
            for trig, dtrig in ((cm, -sm), (sm, cm)) if m else ((cm, None),):
                y = p1 * trig
                qi = q * y * irr
                inner, outer = fac * _before(q * y * reg), fac * _after(qi)
                total = qi.sum()
                if l % 2 and m == 0:
                    tally = tally + psi[l] * total
                others = total if w.self_image else total - qi
                ci = inner - f[l] * others  # of irr y
                if m == 0 and u:
                    ci = ci + u * psi[l] * 4 * math.pi * n_tilde
                pot = scale * (ci * irr + outer * reg)  # potential per y
                g_r += scale * (l * outer * reg - (l + 1) * ci * irr) * y
                g_t += pot * dp * trig
                if m:
                    g_p += pot * p1 * (m * dtrig)
    pf = 1.0 / (4 * math.pi * n_tilde)
    qin = n_ion * (r ** 3 - 1) / (r_out ** 3 - 1) + q_s + _before(q)
    e_r = pf * (qin / (r * r) - g_r / r)
    e_t = -pf * g_t / r
    e_p = -pf * g_p / rho
    E = torch.empty_like(x)
    h = e_r * st + e_t * ct
    E[order] = torch.stack((h * cp - e_p * sp, h * sp + e_p * cp, e_r * ct - e_t * st), 1)
    return E, tally


def _philox(c0, c1, ids, tag, seed):
    """Philox4x32-10 (Salmon et al., SC 2011): four words in int64, counter (c0, c1, ids, tag), key seed."""
    M = 0xFFFFFFFF
    c = [torch.full_like(ids, c0), torch.full_like(ids, c1), ids, torch.full_like(ids, tag)]
    k0, k1 = seed & M, (seed >> 32) & M
    for _ in range(10):
        a, b = c[0] * 0xD2511F53, c[2] * 0xCD9E8D57  # 64-bit products, wrapped
        c = [((b >> 32) & M) ^ c[1] ^ k0, b & M, ((a >> 32) & M) ^ c[3] ^ k1, a & M]
        k0, k1 = (k0 + 0x9E3779B9) & M, (k1 + 0xBB67AE85) & M
    return c


def _frame(n):
    """Two unit vectors normal to n (Duff et al., JCGT 2017)."""
    sg = torch.where(n[:, 2] >= 0, 1.0, -1.0).to(n)
    a = -1.0 / (sg + n[:, 2])
    b = n[:, 0] * n[:, 1] * a
    return (torch.stack((1 + sg * n[:, 0] ** 2 * a, sg * b, -sg * n[:, 0]), 1),
            torch.stack((b, sg + n[:, 1] ** 2 * a, -n[:, 1]), 1))


def _walls(w, x, v, step, seed):
    """Diffuse reflection, or absorption with re-injection from the outer wall; returns the probe's absorptions."""
    r = torch.linalg.norm(x, dim=1)
    hit = torch.nonzero((r < 1.0) | (r > w.r_out)).flatten()
    if hit.numel() == 0:
        return 0
    lo, hi = step & 0xFFFFFFFF, step >> 32
    rh = r[hit]
    inner = rh < 1.0
    if w.wall_rule == 2:
        uni = lambda word: ((word >> 8).double() + 0.5) / 16777216.0  # noqa: E731
        a, b = _philox(lo, hi, hit, 0x494E4A30, seed), _philox(lo, hi, hit, 0x494E4A31, seed)
        u1, u2, u3, u4, u5, u6 = (uni(t) for t in (*a, b[0], b[1]))
        ct = 1 - 2 * u1
        st = torch.sqrt(1 - ct * ct)
        n = torch.stack((st * torch.cos(2 * math.pi * u2), st * torch.sin(2 * math.pi * u2), ct), 1)
        vn = w.sigma_v * torch.sqrt(-2 * torch.log(u3))
        rho = w.sigma_v * torch.sqrt(-2 * torch.log(u4))
        t1, t2 = _frame(n)
        x[hit] = (w.r_out - u6 * w.dt * vn).clamp_min(1.0)[:, None] * n
        v[hit] = (-vn[:, None] * n + (rho * torch.cos(2 * math.pi * u5))[:, None] * t1 +
                  (rho * torch.sin(2 * math.pi * u5))[:, None] * t2)
        return int(inner.sum())
    e = x[hit] / rh[:, None]
    rn = torch.where(inner, 2.0 - rh, 2.0 * w.r_out - rh).clamp(1.0, w.r_out)
    x[hit] = e * rn[:, None]
    n = torch.where(inner[:, None], e, -e)
    o = _philox(lo, hi, hit, 0x494D5250, seed)
    ca = 1.0 - (o[0] >> 8).double() / 16777216.0
    ph = 2 * math.pi * (o[1] >> 8).double() / 16777216.0
    sa = torch.sqrt(1 - ca * ca)
    t1, t2 = _frame(n)
    v[hit] = torch.linalg.norm(v[hit], dim=1)[:, None] * (
        ca[:, None] * n + sa[:, None] * (torch.cos(ph)[:, None] * t1 + torch.sin(ph)[:, None] * t2))
    return 0


def _scatter(v, nu, dt, step, seed):
    """Elastic isotropic electron-neutral collisions."""
    ids = torch.arange(v.shape[0], device=v.device)
    o = _philox(step & 0xFFFFFFFF, step >> 32, ids, 0x434F4C4C, seed)
    k = torch.nonzero((o[0] >> 8) < int(math.floor((1.0 - math.exp(-nu * dt)) * 16777216.0))).flatten()
    ct = 1 - 2 * (o[1][k] >> 8).double() / 16777216.0
    ph = 2 * math.pi * (o[2][k] >> 8).double() / 16777216.0
    st = torch.sqrt(1 - ct * ct)
    v[k] = torch.linalg.norm(v[k], dim=1)[:, None] * torch.stack((st * torch.cos(ph), st * torch.sin(ph), ct), 1)


def _drive(w, n):
    v_hat = w.V_volts * 8.8541878128e-12 / (w.n_e_m3 * 1.602176634e-19 * w.R_D_m ** 2)
    if w.drive_kind == 1:
        return v_hat if n == 0 else 0.0
    return v_hat * math.exp(-0.5 * ((n * w.dt - 4 * w.width_wpe) / w.width_wpe) ** 2)


def _setup(case, w, device):
    n_e = _electrons(case)
    charge = torch.full((w.N,), -1.0, dtype=torch.float64, device=device)
    charge[n_e:] = 1.0
    n_tilde = n_e / (4 * math.pi / 3 * (w.r_out ** 3 - 1))
    return n_e, charge, n_tilde, float(w.N if n_e == w.N else 2 * n_e - w.N)


def _exact_steps(case, w, x, v, steps):
    n_e, charge, n_tilde, n_ion = _setup(case, w, x.device)
    qm = charge.clone()
    qm[n_e:] /= ION_MASS
    absorbed, qs, us = 0, [], []
    for s in range(steps):
        u = _drive(w, s)
        E, tally = _field(w, x, charge, n_tilde, n_ion, -float(absorbed), u)
        qs.append(float(-tally / n_tilde))
        us.append(u)
        v += (0.5 * w.dt if s == 0 else w.dt) * qm[:, None] * E
        x += w.dt * v
        absorbed += _walls(w, x, v, s, w.seed)
        if _nu(case) > 0:
            _scatter(v, _nu(case), w.dt, s, w.seed)
    return np.array(qs), np.array(us), x.cpu(), v.cpu()


def exact(case, seed):
    kind = case["kind"]
    if kind == "spectrum":
        q, u = _series(case, seed)
        t = 0.05 * torch.arange(case["ns"], dtype=torch.float64, device="cuda")
        om = 2.0 / case["nf"] * torch.arange(1, case["nf"] + 1, dtype=torch.float64, device="cuda")
        ph = om[:, None] * t[None, :]
        e = torch.complex(torch.cos(ph), -torch.sin(ph))
        kick = torch.full_like(t, 0.05)
        kick[0] = 0.025
        Q = 0.05 * (e @ torch.from_numpy(q - q[0]).to("cuda", torch.complex128))
        U = e @ (kick * torch.from_numpy(u).to("cuda")).to(torch.complex128)
        y = 1j * om * Q / U
        return om.cpu().numpy(), y.real.cpu().numpy(), y.imag.cpu().numpy()
    if kind == "batch":
        out = []
        for k, c in enumerate(_batch_cases(case)):
            q, _, x, v = _exact_steps(c, *_inputs(c, 1000 * seed + k), c["steps"])
            out.append((q, x, v))
        return out
    w, x, v = _inputs(case, seed)
    if kind == "noalloc":
        _, charge, n_tilde, n_ion = _setup(case, w, x.device)
        return _field(w, x, charge, n_tilde, n_ion, 0.0, _drive(w, 0))[0]
    q, u, x, v = _exact_steps(case, w, x, v, case["steps"])
    return (q, x, v) if kind == "stream" else (q, u, x, v)
