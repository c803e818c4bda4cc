"""GPU parity: the CUDA path (through the C ABI) against the FP64 oracle.

Tolerances (max|a-b|/max|b| per field, vector norm for u, and the same over
all populations):
  FP64 storage  <= 1e-12 relative,
  FP32 storage  <= 1e-5 relative over 1000 steps.
Integer-like work (pure streaming with omega = 0, checkpoint round trips)
is compared bit for bit.
"""
import math

import numpy as np
import pytest

import oracle as O
from oracle import riemann as R
from paper_1402_5487_gb300 import build, inputs as I, plbm

from parity_util import field_errors, gpu_run, oracle_run, patch_fields, rel

pytestmark = pytest.mark.gpu

V5 = I.SET_013
TOL64 = 1e-12
TOL32 = 1e-5


@pytest.fixture(scope="module", autouse=True)
def _lib():
    build.build()
    plbm.lib()


def smooth_fields(nx, ny, seed, amp_u=0.05, amp_r=0.02, theta0=1.0):
    rng = np.random.default_rng(seed)
    x = np.arange(nx)[None, :] * 2 * np.pi / nx
    y = np.arange(ny)[:, None] * 2 * np.pi / ny
    ph = rng.uniform(0, 2 * np.pi, 4)
    rho = 1 + amp_r * np.sin(x + ph[0]) * np.cos(y + ph[1]) + 0.001 * rng.uniform(-1, 1, (ny, nx))
    ux = amp_u * np.sin(y + ph[2]) + 0.002 * rng.uniform(-1, 1, (ny, nx))
    uy = amp_u * np.cos(x + ph[3]) + 0.002 * rng.uniform(-1, 1, (ny, nx))
    th = theta0 * (1 + amp_r * np.cos(x + y + ph[0])) + 0 * rho
    return (np.ascontiguousarray(rho), np.ascontiguousarray(ux), np.ascontiguousarray(uy),
            np.ascontiguousarray(th))


@pytest.mark.parametrize("nx,ny", [(33, 17), (7, 5), (1, 1), (130, 3), (256, 2)])
def test_pure_stream_bit_exact(nx, ny):
    # omega = 0 leaves only the pull: identical FP64 inputs must give identical outputs.
    lat = O.Lattice(2, V5, 0.0, nx, ny, theta0=1.0)
    f0 = lat.init(*smooth_fields(nx, ny, 1))
    s = plbm.Solver(2, V5, 0.0, nx, ny, theta0=1.0, prec="f64")
    s.set_populations(f0)
    s.step(3)
    assert np.array_equal(s.get_populations(), lat.run(f0, 3))
    s.close()


@pytest.mark.parametrize("nx,ny", [(33, 17), (130, 3)])
def test_pure_stream_fixed_ends_bit_exact(nx, ny):
    left, right = (1.2, 0.05, 0.9), (0.8, -0.02, 1.1)
    lat = O.Lattice(2, V5, 0.0, nx, ny, bc="fixed", theta0=1.0, left_state=left, right_state=right)
    f0 = lat.init(*smooth_fields(nx, ny, 5))
    s = plbm.Solver(2, V5, 0.0, nx, ny, theta0=1.0, prec="f64", bc="fixed", left_state=left,
                    right_state=right)
    s.set_populations(f0)
    s.step(4)
    got, ref = s.get_populations(), lat.run(f0, 4)
    # ghost populations come from the library's own FP64 f^eq: equal to rounding
    assert np.max(np.abs(got - ref)) <= 1e-15
    s.close()


@pytest.mark.parametrize("nx,ny", [(33, 17), (7, 5), (1, 1), (200, 9), (34, 18), (1, 2)])
def test_parity_d2q25_f64(nx, ny):
    fields = smooth_fields(nx, ny, 2)
    (mg, fg, _) = gpu_run(2, V5, 1.3, nx, ny, fields, 100, prec="f64")
    _, fo, mo = oracle_run(2, V5, 1.3, nx, ny, fields, 100)
    assert rel(fg, fo) <= TOL64
    # tiny periodic grids damp u to a small fraction of its start within 100 steps: scale
    # the velocity error by its initial amplitude
    u0 = np.max(np.hypot(fields[1], fields[2]))
    assert np.max(np.hypot(mg[1] - mo[1], mg[2] - mo[2])) <= TOL64 * u0
    assert O.rel_err(mg[0], mo[0]) <= TOL64 and O.rel_err(mg[3], mo[3]) <= TOL64


# Even ny takes the row-paired two-nodes-per-thread kernel, odd ny the one-node kernel.
@pytest.mark.parametrize("nx,ny", [(33, 17), (7, 5), (1, 1), (130, 3), (34, 18), (8, 6), (1, 2),
                                   (130, 4), (257, 10)])
@pytest.mark.parametrize("prec,tol", [("f32", 2e-6), ("f16dev", 2e-3), ("bf16dev", 2e-2)])
def test_parity_d2q25_reduced_storage_small_grids(nx, ny, prec, tol):
    fields = smooth_fields(nx, ny, 7)
    steps = 50
    (mg, fg, _) = gpu_run(2, V5, 1.3, nx, ny, fields, steps, prec=prec)
    _, fo, mo = oracle_run(2, V5, 1.3, nx, ny, fields, steps)
    u0 = np.max(np.hypot(fields[1], fields[2]))
    assert np.max(np.hypot(mg[1] - mo[1], mg[2] - mo[2])) <= tol * u0
    assert O.rel_err(mg[0], mo[0]) <= tol * 0.1 and O.rel_err(mg[3], mo[3]) <= tol * 0.1
    assert np.max(np.abs(fg - fo)) <= tol * 0.1 * np.max(np.abs(fo))


@pytest.mark.parametrize("prec,tol", [("f64", TOL64), ("f32", 2e-6)])
@pytest.mark.parametrize("v,theta0,omega,iso", [((0, 1, -1), 0.25, 1.2, True),
                                                ((0, 1, -1), 1.0 / 3.0, 1.5, True),
                                                ((1, -1, 3, -3), 4.0 / 3.0, 1.1, True),
                                                ((0, 1, -1, 2, -2), 1 / 1.6 ** 2, 1.6, False),
                                                ((0, 2, -2, 3, -3), 1.6, 1.2, False),
                                                ((0, 2, -4), 1.0, 1.0, True),
                                                ((0, 1, -1, 2, -2, 3), 0.8, 1.3, False),
                                                ((0, 1, -1, 2, -2, 3, -3), 1.0, 1.3, False),
                                                ((0, 1, -1, 2, -2, 3, -3, 4), 1.0, 1.3, False)])
def test_parity_other_sets(v, theta0, omega, iso, prec, tol):
    nx, ny = 70, 19
    fields = smooth_fields(nx, ny, 3, amp_u=0.03, amp_r=0.01, theta0=theta0)
    (mg, fg, _) = gpu_run(2, v, omega, nx, ny, fields, 60, prec=prec, theta0=theta0, isothermal=iso)
    _, fo, mo = oracle_run(2, v, omega, nx, ny, fields, 60, theta0=theta0, isothermal=iso)
    assert rel(fg, fo) <= tol
    assert O.rel_err(mg[0], mo[0]) <= tol and O.rel_err(mg[3], mo[3]) <= tol


@pytest.mark.parametrize("prec,tol", [("f64", TOL64), ("f32", TOL32)])
def test_parity_d1q5_shock_tube(prec, tol):
    left, right = (1.1, 0.0, 0.5), (1.0, 0.0, 0.5)
    fields = I.shock_tube_fields(1000, left, right)
    (mg, fg, _) = gpu_run(1, V5, 1.5, 1000, 1, fields, 500, prec=prec, theta0=0.5, bc="fixed",
                          left=left, right=right)
    _, fo, mo = oracle_run(1, V5, 1.5, 1000, 1, fields, 500, theta0=0.5, bc="fixed", left=left,
                           right=right)
    errs = field_errors(mg, mo)
    assert max(errs.values()) <= tol, errs
    if prec == "f64":
        assert rel(fg, fo) <= tol


def test_shock_tube_gpu_vs_exact_riemann():
    left, right = (1.1, 0.0, 0.5), (1.0, 0.0, 0.5)
    fields = I.shock_tube_fields(1000, left, right)
    (mg, _, _) = gpu_run(1, V5, 1.5, 1000, 1, fields, 361, prec="f64", theta0=0.5, bc="fixed",
                         left=left, right=right)
    rho, ux, _, th = (a[0] for a in mg)
    x = np.arange(1000) + 0.5
    re, ue, pe = R.sample(R.State(1.1, 0.0, 0.55), R.State(1.0, 0.0, 0.5), 3.0, (x - 500) / 361)
    assert np.mean(np.abs(rho - re)) / np.mean(re) < 0.002
    assert np.mean(np.abs(ux - ue)) / np.max(np.abs(ue)) < 0.02
    assert np.mean(np.abs(th - pe / re)) / np.mean(pe / re) < 0.002


@pytest.mark.parametrize("L", [128])
def test_parity_kh_1000_steps(L):
    fields = I.kh_fields(L)
    _, fo, mo = oracle_run(2, V5, 1.3, L, L, fields, 1000)
    (m64, f64, _) = gpu_run(2, V5, 1.3, L, L, fields, 1000, prec="f64")
    (m32, f32, _) = gpu_run(2, V5, 1.3, L, L, fields, 1000, prec="f32")
    e64 = field_errors(m64, mo)
    e32 = field_errors(m32, mo)
    assert max(e64.values()) <= TOL64 and rel(f64, fo) <= TOL64, e64
    assert max(e32.values()) <= TOL32 and rel(f32, fo) <= TOL32, e32


@pytest.mark.slow
def test_parity_kh_512_config_1000_steps():
    # Kelvin-Helmholtz double shear layer, 512^2, D2Q25 {0,+-1,+-3}^2, theta0 = 1, omega = 1.3.
    L = 512
    fields = I.kh_fields(L)
    _, fo, mo = oracle_run(2, V5, 1.3, L, L, fields, 1000)
    (m64, f64, _) = gpu_run(2, V5, 1.3, L, L, fields, 1000, prec="f64")
    (m32, f32, _) = gpu_run(2, V5, 1.3, L, L, fields, 1000, prec="f32")
    e64 = field_errors(m64, mo)
    e32 = field_errors(m32, mo)
    assert max(e64.values()) <= TOL64 and rel(f64, fo) <= TOL64, e64
    assert max(e32.values()) <= TOL32 and rel(f32, fo) <= TOL32, e32


@pytest.mark.parametrize("L,prec,tol", [(2048, "f32", 1e-6), (2047, "f32", 1e-6), (2048, "f16dev", 2e-3),
                                         (2048, "bf16dev", 2e-2)])
def test_fullsize_2048_sampled_nodes(L, prec, tol):
    # Bench workloads (2048^2 KH in FP32 and 16-bit storage on row pairs; 2047^2, the
    # plain layout of odd sides): after k steps a node depends only on nodes within 3k
    # in each direction, so the oracle advances a (6k+1)^2 periodic window around each
    # sampled node and its centre must match the GPU.
    k, half = 4, 12
    fields = I.kh_fields(L)
    s = plbm.Solver(2, V5, 1.3, L, L, theta0=1.0, prec=prec)
    s.init(*fields)
    s.step(k)
    mg = s.moments()
    rng = np.random.default_rng(11)
    pts = [(0, 0), (L - 1, L - 1), (L // 2, L // 4), (3, L - 2)] + [
        tuple(int(a) for a in rng.integers(0, L, 2)) for _ in range(28)]
    errs = []
    for cx, cy in pts:
        pf = patch_fields(fields, cx, cy, half, L, L)
        lat, f, mo = oracle_run(2, V5, 1.3, 2 * half + 1, 2 * half + 1, pf, k)
        for gi, oi in zip(mg, mo):
            errs.append(abs(gi[cy, cx] - oi[half, half]) / max(1e-30, np.max(np.abs(fields[0]))))
    rho_g, ux_g, uy_g, _ = mg
    assert max(errs[0::4]) < tol      # rho
    assert max(errs[3::4]) < tol      # theta
    assert max(max(errs[1::4]), max(errs[2::4])) < tol  # velocity components (scale ~0.1)
    d = s.diagnostics()
    assert abs(d["mass"] - L * L) / (L * L) < max(tol, 1e-6)
    s.close()


def test_conservation_periodic_f64():
    L = 64
    fields = I.kh_fields(L)
    s = plbm.Solver(2, V5, 1.3, L, L, theta0=1.0, prec="f64")
    s.init(*fields)
    c0 = s.conserved()
    s.step(10000)
    c1 = s.conserved()
    assert np.max(np.abs(c1 - c0)) <= 1e-12 * np.max(np.abs(c0))
    lat = O.Lattice(2, V5, 1.3, L, L, theta0=1.0)
    f = lat.init(*fields)
    assert np.max(np.abs(c0 - lat.conserved(f))) <= 1e-13 * np.max(np.abs(c0))
    s.close()


def test_diagnostics_match_oracle():
    L = 48
    fields = I.kh_fields(L, seed=5)
    (mg, fg, s) = gpu_run(2, V5, 1.3, L, L, fields, 37, prec="f64")
    lat, fo, mo = oracle_run(2, V5, 1.3, L, L, fields, 37)
    d = s.diagnostics()
    co = lat.conserved(fo)
    for a, b in zip((d["mass"], d["jx"], d["jy"], d["energy"]), co):
        assert abs(a - b) <= 1e-12 * max(1.0, abs(co[0]))
    assert abs(d["rho_min"] - mo[0].min()) < 1e-13
    assert abs(d["theta_min"] - mo[3].min()) < 1e-13
    assert d["status"] == 0 and d["steps"] == 37
    s.close()


@pytest.mark.parametrize("prec", ["f64", "f32", "f16dev", "bf16dev"])
def test_checkpoint_resume_is_bit_identical(prec):
    L = 40
    fields = I.kh_fields(L, seed=3)
    a = plbm.Solver(2, V5, 1.3, L, L, theta0=1.0, prec=prec)
    a.init(*fields)
    a.step(20)
    f20 = a.get_populations()
    a.step(20)
    ref = a.get_populations()
    b = plbm.Solver(2, V5, 1.3, L, L, theta0=1.0, prec=prec)
    b.set_populations(f20, step=20)
    b.step(20)
    assert np.array_equal(b.get_populations(), ref)
    assert b.diagnostics()["steps"] == 40
    a.close()
    b.close()


def test_device_pointers_and_streams():
    import torch
    L = 64
    fields = I.kh_fields(L, seed=4)
    st = torch.cuda.Stream()
    s = plbm.Solver(2, V5, 1.3, L, L, theta0=1.0, prec="f32", stream=st)
    dev = [torch.from_numpy(a).to("cuda") for a in fields]
    torch.cuda.synchronize()
    s.init(*dev)
    s.step(10)
    md = s.moments(on_device=True)
    st.synchronize()
    mh = s.moments()
    for a, b in zip(md, mh):
        assert np.array_equal(a.cpu().numpy(), b)
    (mg, _, _) = gpu_run(2, V5, 1.3, L, L, fields, 10, prec="f32")
    for a, b in zip(mg, mh):
        assert np.array_equal(a, b)
    s.close()


@pytest.mark.parametrize("prec,tol", [("f16dev", 2e-2), ("bf16dev", 1e-1)])
def test_reduced_precision_error_is_bounded(prec, tol):
    L = 128
    fields = I.kh_fields(L)
    _, _, mo = oracle_run(2, V5, 1.3, L, L, fields, 1000)
    (mg, _, s) = gpu_run(2, V5, 1.3, L, L, fields, 1000, prec=prec)
    errs = field_errors(mg, mo)
    assert errs["u"] <= tol and errs["rho"] <= tol * 0.1 and errs["theta"] <= tol * 0.1, errs
    assert s.check() == plbm.PLBM_OK


def test_literal_shock_tube_reports_divergence():
    # rho 1 / 0.125, theta 0.5 / 0.4 on {0,+-1,+-3}: leaves the positivity region (theta <= 0).
    left, right = (1.0, 0.0, 0.5), (0.125, 0.0, 0.4)
    s = plbm.Solver(1, V5, 1.5, 1000, 1, theta0=0.5, prec="f64", bc="fixed", left_state=left,
                    right_state=right, check_every=5)
    s.init(*I.shock_tube_fields(1000, left, right))
    st = s.step_status(500)
    assert st == plbm.PLBM_E_DIVERGED
    assert "diverged" in plbm.last_error(s.h)
    # sticky: further steps are refused, diagnostics still readable
    assert s.step_status(1) == plbm.PLBM_E_DIVERGED
    assert s.diagnostics()["status"] != 0
    s.close()


def test_literal_kh_omega_reports_divergence():
    L = 64
    s = plbm.Solver(2, V5, 1.8, L, L, theta0=1.0, prec="f32", check_every=50)
    s.init(*I.kh_fields(L))
    assert s.step_status(3000) == plbm.PLBM_E_DIVERGED
    s.close()


def test_stable_kh_stays_healthy():
    L = 64
    s = plbm.Solver(2, V5, 1.3, L, L, theta0=1.0, prec="f32", check_every=100)
    s.init(*I.kh_fields(L))
    assert s.step_status(3000) == plbm.PLBM_OK
    rho, ux, uy, th = s.moments()
    assert abs(rho - 1).max() < 0.01 and abs(th - 1).max() < 0.01
    assert np.hypot(ux, uy).max() < 0.12
    s.close()


# --------------------------------------------------------------------------
# The paper's own parameters (Sec. 4): {0, +-1, +-2} = {0, +-a, +-2a} sqrt(theta0),
# theta0 = 1 / a^2, omega = 1.9.
# --------------------------------------------------------------------------
SET_012 = (0, 1, -1, 2, -2)


def _exact_rounded_coefficients(v):
    """V^{-1} in exact rational arithmetic, each entry rounded once to FP64."""
    from fractions import Fraction
    q = len(v)
    A = [[Fraction(vk) ** n for vk in v] + [Fraction(int(n == k)) for k in range(q)] for n in range(q)]
    for c in range(q):
        p = next(r for r in range(c, q) if A[r][c] != 0)
        A[c], A[p] = A[p], A[c]
        d = A[c][c]
        A[c] = [x / d for x in A[c]]
        for r in range(q):
            if r != c and A[r][c] != 0:
                m = A[r][c]
                A[r] = [a_ - m * b_ for a_, b_ in zip(A[r], A[c])]
    return np.array([[float(A[i][q + n]) for n in range(q)] for i in range(q)])


def coefficient_sensitivity(dim, v, omega, nx, ny, fields, steps, **kw):
    """Oracle fields after `steps` and the oracle's own drift against a copy of
    itself whose c_ij are the exact rationals rounded once (a few ulps of each
    row's scale from its Gauss-Jordan values): the part of an FP64 difference
    that the last bits of the coefficients explain."""
    lat = O.Lattice(dim, v, omega, nx, ny, **kw)
    alt = O.Lattice(dim, v, omega, nx, ny, **kw)
    cex = _exact_rounded_coefficients(v)
    row = np.max(np.abs(cex), axis=1, keepdims=True)
    assert np.max(np.abs(cex - lat.C) / (np.finfo(float).eps * row)) <= 8.0
    for i, c in enumerate(cex.ravel()):
        alt.struct.C[i] = c
    m0 = lat.moments(lat.run(lat.init(*fields), steps))
    m1 = alt.moments(alt.run(alt.init(*fields), steps))
    return m0, field_errors(m1, m0)


def test_paper_shear_layer_f64_within_the_coefficient_rounding_sensitivity():
    # At omega = 1.9 the BGK step hardly damps the momentum error that a one-ulp
    # difference in the c_ij injects every step, so two correct FP64
    # implementations whose coefficients differ in the last bit drift apart
    # linearly (the library builds c_ij by Lagrange expansion, the oracle by
    # Gauss-Jordan elimination).  The bound is the oracle's own drift against a
    # copy of itself with correctly rounded coefficients (at most one ulp away).
    fields, theta0 = I.paper_kh_fields()
    steps = 1000
    lat = O.Lattice(2, SET_012, 1.9, 128, 128, theta0=theta0)
    alt = O.Lattice(2, SET_012, 1.9, 128, 128, theta0=theta0)
    cex = _exact_rounded_coefficients(SET_012)
    assert np.max(np.abs(cex - lat.C) / np.spacing(np.abs(cex) + 1e-300)) <= 1.0
    for i, c in enumerate(cex.ravel()):
        alt.struct.C[i] = c
    m0 = lat.moments(lat.run(lat.init(*fields), steps))
    m1 = alt.moments(alt.run(alt.init(*fields), steps))
    (mg, _, _) = gpu_run(2, SET_012, 1.9, 128, 128, fields, steps, prec="f64", theta0=theta0)
    sens = field_errors(m1, m0)
    errs = field_errors(mg, m0)
    assert errs["rho"] <= TOL64 and errs["theta"] <= TOL64, errs
    assert errs["u"] <= max(TOL64, 2.0 * sens["u"]), (errs, sens)


@pytest.mark.parametrize("steps,tol", [(100, TOL32), (1000, 1e-4)])
def test_paper_shear_layer_f32_matches_oracle(steps, tol):
    # The FP32 bar (1e-5) at 100 steps.  With the paper's slow flow (u0 = 0.043)
    # and omega = 1.9, which hardly damps the momentum error of the FP32 storage
    # rounding (a few 1e-9 per population per step), the relative u error walks to
    # 1.05e-5 at 200 steps and 4.4e-5 at 1000 steps (a regression bound there).
    fields, theta0 = I.paper_kh_fields()
    (mg, fg, _) = gpu_run(2, SET_012, 1.9, 128, 128, fields, steps, prec="f32", theta0=theta0)
    _, fo, mo = oracle_run(2, SET_012, 1.9, 128, 128, fields, steps, theta0=theta0)
    errs = field_errors(mg, mo)
    assert max(errs.values()) <= tol, errs


def test_paper_shear_layer_stays_stable_to_the_last_printed_step_in_f64():
    # The paper shows the 25-velocity shear layer up to step 3695 at omega = 1.9.
    from paper_1402_5487_gb300 import plbm
    fields, theta0 = I.paper_kh_fields()
    s = plbm.Solver(2, SET_012, 1.9, 128, 128, theta0=theta0, prec="f64")
    s.init(*fields)
    s.step(3695)
    assert s.check() == plbm.PLBM_OK
    rho, ux, uy, th = s.moments()
    s.close()
    assert 0.995 < rho.min() and rho.max() < 1.005
    assert 0.995 < th.min() / theta0 and th.max() / theta0 < 1.005
    assert np.max(np.hypot(ux, uy)) < 0.06


def test_paper_shear_layer_in_f32_follows_f64_then_diverges_and_is_reported():
    # FP32 rounding (~1e-7) seeds the mode that the oracle shows growing from a
    # 1e-7 perturbation of the FP64 initial state (tests/test_oracle_paper_params.py):
    # the FP32 run follows FP64 for 1500 steps, then departs and the status word
    # reports the divergence before the paper's last printed step.
    from paper_1402_5487_gb300 import plbm
    fields, theta0 = I.paper_kh_fields()
    a = plbm.Solver(2, SET_012, 1.9, 128, 128, theta0=theta0, prec="f32")
    b = plbm.Solver(2, SET_012, 1.9, 128, 128, theta0=theta0, prec="f64")
    for s in (a, b):
        s.init(*fields)
        s.step(1500)
    ea = field_errors(a.moments(), b.moments())
    assert max(ea.values()) < 1e-3, ea
    statuses = []
    for _ in range(9):                       # up to step 3750
        a.step(250)
        statuses.append(a.check())
        if statuses[-1] != plbm.PLBM_OK:
            break
    a.close()
    b.close()
    assert statuses[-1] == plbm.PLBM_E_DIVERGED, statuses


@pytest.mark.parametrize("prec", ["f64", "f32"])
def test_d1q7_thermal_shock_tube_matches_oracle(prec):
    # The conventional seven-velocity on-lattice thermal set {0, +-1, +-2, +-3}
    # (q1 = 7, n* = 6) through the general-q1 kernels.  FP64: rho, theta within
    # 1e-12 and u within twice the oracle's own sensitivity to the last bit of
    # its c_ij (denominators up to 720 here); FP32 within 1e-5.
    v = (0, 1, -1, 2, -2, 3, -3)
    left, right = (1.1, 0.0, 1.0), (1.0, 0.0, 1.0)
    fields = I.shock_tube_fields(1000, left, right)
    (mg, fg, _) = gpu_run(1, v, 1.5, 1000, 1, fields, 300, prec=prec, theta0=1.0, bc="fixed", left=left,
                          right=right)
    m0, sens = coefficient_sensitivity(1, v, 1.5, 1000, 1, fields, 300, bc="fixed", theta0=1.0,
                                       left_state=left, right_state=right)
    errs = field_errors(mg, m0)
    if prec == "f64":
        assert errs["rho"] <= TOL64 and errs["theta"] <= TOL64, errs
        assert errs["u"] <= max(TOL64, 2.0 * sens["u"]), (errs, sens)
    else:
        assert max(errs.values()) <= TOL32, errs


def test_paper_d1q5_shock_tube_f64_within_the_coefficient_rounding_sensitivity():
    # Same bound as the shear layer: at omega = 1.9 the one-ulp differences of the
    # c_ij between the library and the oracle drift the slow post-shock flow apart.
    theta = 1 / 1.96
    left, right = (1.1, 0.0, theta), (1.0, 0.0, theta)
    fields = I.shock_tube_fields(1000, left, right)
    m0, sens = coefficient_sensitivity(1, SET_012, 1.9, 1000, 1, fields, 346, bc="fixed", theta0=theta,
                                       left_state=left, right_state=right)
    (mg, _, _) = gpu_run(1, SET_012, 1.9, 1000, 1, fields, 346, prec="f64", theta0=theta, bc="fixed",
                         left=left, right=right)
    errs = field_errors(mg, m0)
    assert errs["rho"] <= TOL64 and errs["theta"] <= TOL64, errs
    assert errs["u"] <= max(TOL64, 2.0 * sens["u"]), (errs, sens)


def test_paper_d1q5_shock_tube_f32_matches_oracle():
    # A regression bound: at omega = 1.9 the shock leaves acoustic oscillations of
    # a third of the post-shock velocity that the collision barely damps, and the
    # FP32 rounding of the stored populations walks the slow flow (u ~ 0.02) away
    # from FP64 by ~2.5e-5 in u after 346 steps (the 1e-5 bar holds for the
    # omega = 1.5 shock tube, test_parity_d1q5_shock_tube).
    theta = 1 / 1.96
    left, right = (1.1, 0.0, theta), (1.0, 0.0, theta)
    fields = I.shock_tube_fields(1000, left, right)
    (mg, fg, _) = gpu_run(1, SET_012, 1.9, 1000, 1, fields, 346, prec="f32", theta0=theta, bc="fixed",
                          left=left, right=right)
    _, fo, mo = oracle_run(1, SET_012, 1.9, 1000, 1, fields, 346, theta0=theta, bc="fixed", left=left,
                           right=right)
    errs = field_errors(mg, mo)
    assert errs["u"] <= 5e-5 and errs["rho"] <= 5e-6 and errs["theta"] <= 5e-6, errs


# --------------------------------------------------------------------------
# The three-velocity models of Sec. 4 (isothermal, D2Q9 tensor products):
# LBGK (zeta = 3) and the parametric zeta = 4 model on the paper's shear layer,
# and second-order convergence on the GPU path.
# --------------------------------------------------------------------------
@pytest.mark.parametrize("zeta", [3, 4])
def test_zeta_shear_layer_matches_oracle_and_the_papers_stability_pattern(zeta):
    from paper_1402_5487_gb300 import plbm
    theta0 = 1.0 / zeta
    omega = {3: 1.99880, 4: 1.99862}[zeta]
    fields, _ = I.paper_kh_fields(theta0=theta0)
    early, late = {3: (500, 1800), 4: (577, 2078)}[zeta]
    (mg, fg, s) = gpu_run(2, (0, 1, -1), omega, 128, 128, fields, early, prec="f64", theta0=theta0,
                          isothermal=True)
    _, fo, mo = oracle_run(2, (0, 1, -1), omega, 128, 128, fields, early, theta0=theta0, isothermal=True)
    assert max(field_errors(mg, mo).values()) <= TOL64
    s.step(late - early)
    status = s.check()
    s.close()
    # LBGK is gone before its step 1800; zeta = 4 is still running at 2078
    assert status == (plbm.PLBM_E_DIVERGED if zeta == 3 else plbm.PLBM_OK), status


@pytest.mark.parametrize("prec", ["f64", "f32"])
@pytest.mark.parametrize("v,theta0,iso,omega", [((0, 1, -1), 0.25, True, 1.2),
                                                ((0, 1, -1, 3, -3), 1.0, False, 1.3)],
                         ids=["zeta4", "d2q25"])
def test_taylor_green_converges_at_second_order_on_gpu(v, theta0, iso, omega, prec):
    from test_oracle_paper_params import taylor_green_errors

    def runner(v, theta0, iso, omega, N, fields, steps):
        (m, _, s) = gpu_run(2, v, omega, N, N, fields, steps, prec=prec, theta0=theta0, isothermal=iso)
        s.close()
        return m

    errs = taylor_green_errors(v, theta0, iso, omega, runner=runner)
    orders = [math.log2(errs[i] / errs[i + 1]) for i in range(len(errs) - 1)]
    assert all(o > 1.8 for o in orders), (errs, orders)


@pytest.mark.parametrize("prec,dim", [("f64", 1), ("f32", 2), ("f16dev", 2)])
def test_graph_replayed_steps_equal_single_launches(prec, dim):
    # Small lattices advance by replays of a captured 32-step graph; the result must
    # equal the same steps launched one call at a time, bit for bit.
    nx, ny = (1000, 1) if dim == 1 else (64, 48)
    fields = I.kh_fields(nx, ny=ny) if dim == 2 else I.shock_tube_fields(nx)
    out = []
    for chunks in ([150], [1] * 150):
        if dim == 1:
            s = plbm.Solver(1, I.SET_013, 1.5, nx, 1, theta0=0.5, prec=prec, bc="fixed",
                            left_state=(1.1, 0.0, 0.5), right_state=(1.0, 0.0, 0.5))
            s.init(fields[0], fields[1], None, fields[3])
        else:
            s = plbm.Solver(2, I.SET_013, 1.3, nx, ny, theta0=1.0, prec=prec)
            s.init(*fields)
        for c in chunks:
            s.step(c)
        out.append(s.get_populations())
        assert s.check() == 0
        s.close()
    assert np.array_equal(out[0], out[1])


@pytest.mark.parametrize("prec", ["f32", "bf16dev", "f64"])
def test_banded_host_transfers_equal_device_pointers(prec):
    # Lattices of 2^18 nodes or more move host fields in eight row bands on a copy
    # stream overlapped with the kernels; the result must equal the device-pointer
    # calls bit for bit (640 x 512 = 327,680 nodes in bands of 64 rows; 520 x 517
    # in uneven bands).
    import torch
    for nx, ny in ((640, 512), (520, 517)):
        fields = I.kh_fields(nx, ny=ny, seed=6)
        st = torch.cuda.Stream()
        a = plbm.Solver(2, V5, 1.3, nx, ny, theta0=1.0, prec=prec, stream=st)
        b = plbm.Solver(2, V5, 1.3, nx, ny, theta0=1.0, prec=prec, stream=st)
        a.init(*fields)                                          # host pointers, banded
        b.init(*[torch.from_numpy(f).to("cuda") for f in fields])  # device pointers
        st.synchronize()
        assert np.array_equal(a.get_populations(), b.get_populations())
        a.step(3)
        b.step(3)
        mh = a.moments()                                         # host pointers, banded
        md = b.moments(on_device=True)
        st.synchronize()
        for x, y in zip(mh, md):
            assert np.array_equal(x, y.cpu().numpy())
        a.close()
        b.close()


@pytest.mark.parametrize("prec,dim", [("f64", 2), ("f32", 2), ("f16dev", 2), ("f64", 1), ("f32", 1)])
def test_fused_step_diagnostics_match_separate_reduction(prec, dim):
    # The last step of plbm_step_diagnostics forms the FP64 sums in the step kernel;
    # they must equal plbm_diagnostics of the same state (FP64: to rounding; 16/32-bit:
    # the fused sums use the kernel's FP32 moments, so to FP32 rounding), and the
    # populations must be those of plain stepping.
    if dim == 2:
        nx, ny = 96, 64
        fields = I.kh_fields(nx, ny=ny, seed=8)
        make = lambda: plbm.Solver(2, V5, 1.3, nx, ny, theta0=1.0, prec=prec)
        init = lambda s: s.init(*fields)
    else:
        nx, ny = 1000, 1
        left, right = (1.1, 0.0, 0.5), (1.0, 0.0, 0.5)
        fields = I.shock_tube_fields(nx, left, right)
        make = lambda: plbm.Solver(1, V5, 1.5, nx, 1, theta0=0.5, prec=prec, bc="fixed", left_state=left,
                                   right_state=right)
        init = lambda s: s.init(fields[0], fields[1], None, fields[3])
    a, b = make(), make()
    init(a)
    init(b)
    da = a.step_diagnostics(37)
    b.step(37)
    db = b.diagnostics()
    assert np.array_equal(a.get_populations(), b.get_populations())
    assert da["steps"] == db["steps"] == 37 and da["status"] == db["status"] == 0
    # 16-bit: the stored state carries the storage rounding of the deviations (~5e-6 each)
    tol = {"f64": 1e-12, "f32": 2e-6, "f16dev": 3e-5}[prec]
    scale = max(abs(db["mass"]), 1.0)
    for k in ("mass", "jx", "jy", "energy"):
        assert abs(da[k] - db[k]) <= tol * max(scale, abs(db["energy"])), (k, da[k], db[k])
    for k in ("rho_min", "theta_min"):
        assert abs(da[k] - db[k]) <= tol * abs(db[k]), (k, da[k], db[k])
    a.close()
    b.close()


# --------------------------------------------------------------------------
# The isothermal three-velocity shock tubes of Sec. 3.2 on the GPU path: the
# 6:1 tube's printed front and post-shock velocity, and the 1.1:1 comparison of
# the zeta = 4 model with LBGK under nu and nu_hat viscosity matching.
# --------------------------------------------------------------------------
def _gpu_tube(prec):
    def tube(v, omega, theta0, left, right, steps):
        fields = I.shock_tube_fields(1000, left, right)
        (m, _, s) = gpu_run(1, v, omega, 1000, 1, fields, steps, prec=prec, theta0=theta0, bc="fixed",
                            left=left, right=right, isothermal=True)
        s.close()
        return m
    return tube


@pytest.mark.parametrize("prec,tol", [("f64", 1e-12), ("f32", 2e-6)])
def test_zeta4_vs_lbgk_small_ratio_on_gpu(prec, tol):
    from test_oracle_riemann import zeta4_vs_lbgk_small_ratio
    ref, _, _ = zeta4_vs_lbgk_small_ratio()
    got, _, _ = zeta4_vs_lbgk_small_ratio(tube=_gpu_tube(prec))
    for k in ref:
        for a, b in zip(got[k], ref[k]):
            assert abs(a - b) <= tol, (k, got, ref)
    assert got["nu_hat"][0] < got["nu"][0] / 10


@pytest.mark.parametrize("prec", ["f64", "f32"])
def test_zeta4_shock_tube_printed_front_on_gpu(prec):
    from conftest import read_printed_values
    vals = read_printed_values()
    theta0 = 0.25
    omega = 4 * math.sqrt(3) - 6
    steps = int(vals["shock6_iterations_param"])
    left, right = (6.0, 0.0, theta0), (1.0, 0.0, theta0)
    mg = _gpu_tube(prec)((0, 1, -1), omega, theta0, left, right, steps)
    _, _, mo = oracle_run(1, (0, 1, -1), omega, 1000, 1, I.shock_tube_fields(1000, left, right), steps,
                          theta0=theta0, bc="fixed", left=left, right=right, isothermal=True)
    errs = field_errors(mg, mo)
    assert max(errs.values()) <= (TOL64 if prec == "f64" else TOL32), errs
    rho, ux = mg[0][0], mg[1][0] / math.sqrt(theta0)
    assert abs(np.mean(ux[650:750]) - vals["shock6_u_post"]) < 0.005
    plateau = np.mean(rho[650:750])
    half = 0.5 * (plateau + 1.0)
    i = int(np.nonzero(rho > half)[0].max())
    front = (i + 1) + (rho[i] - half) / (rho[i] - rho[i + 1])
    assert abs(front - vals["shock6_front_x"]) < 2.5


# --------------------------------------------------------------------------
# Degenerate calls and states: no steps, a negative count, the rest state.
# --------------------------------------------------------------------------
@pytest.mark.parametrize("prec", ["f64", "f32", "f16dev", "bf16dev"])
def test_zero_steps_change_nothing_and_negative_counts_are_refused(prec):
    s = plbm.Solver(2, V5, 1.3, 34, 18, theta0=1.0, prec=prec)
    s.init(*smooth_fields(34, 18, 3))
    s.step(5)
    f0 = s.get_populations()
    n0 = s.diagnostics()["steps"]
    s.step(0)
    assert np.array_equal(s.get_populations(), f0) and s.diagnostics()["steps"] == n0 == 5
    assert s.step_status(-1) == plbm.PLBM_E_ARG
    assert np.array_equal(s.get_populations(), f0) and s.diagnostics()["steps"] == n0
    s.close()


@pytest.mark.parametrize("prec", ["f64", "f32", "f16dev", "bf16dev"])
@pytest.mark.parametrize("dim", [1, 2])
def test_rest_state_is_a_fixed_point(prec, dim):
    # rho = 1, u = 0, theta = theta0: f = w0, which streaming and the collision
    # (Eq. eq:srt with f^eq = w0) leave in place; the 16/32-bit kernels store the
    # deviation from w0, which stays exactly zero.  FP64 stores f itself and
    # recomputes f^eq from the rounded moments each step: the state stays uniform
    # bit for bit (every node does the same arithmetic) and moves by at most a few
    # roundings per step.
    nx, ny = 130, (18 if dim == 2 else 1)
    one, zero = np.ones((ny, nx)), np.zeros((ny, nx))
    s = plbm.Solver(dim, V5, 1.3, nx, ny, theta0=1.0, prec=prec)
    s.init(one, zero, zero if dim == 2 else None, one)
    f0 = s.get_populations()
    s.step(200)
    f = s.get_populations()
    assert s.check() == plbm.PLBM_OK
    if prec == "f64":
        assert np.all(f == f[:, :1, :1])
        assert np.max(np.abs(f - f0)) <= 200 * 16 * np.finfo(float).eps * np.max(f0)
    else:
        assert np.array_equal(f, f0)
    s.close()


@pytest.mark.parametrize("prec,ny,nx", [("f32", 48, 70), ("f16dev", 48, 70), ("bf16dev", 48, 70), ("f16dev", 12, 70),
                                        ("bf16dev", 16, 70), ("f16dev", 20, 70), ("f16dev", 14, 50),
                                        ("f16dev", 22, 200), ("f16dev", 2, 1)])
def test_plain_and_row_paired_layouts_give_the_same_state(prec, ny, nx):
    # The plain-layout kernel (one node per thread: odd ny, PLBM_FLAG_PLAIN_LAYOUT)
    # runs the single-lane forms of the row-paired kernel's packed operations,
    # each correctly rounded, so both layouts give every node the same bits.
    # ny = 12, 16, 20: most pair rows pull across the pair boundary (swapped lanes).
    # FP16 steps take two node pairs per thread (tiles of 64 pairs): nx = 50, ny = 14
    # gives an odd tile count (the last thread block has one tile), nx = 200 a ragged
    # last tile, and 1 x 2 a single node pair.
    fields = I.kh_fields(nx, ny=ny)
    out = []
    for plain in (False, True):
        s = plbm.Solver(2, V5, 1.3, nx, ny, theta0=1.0, prec=prec, plain_layout=plain)
        s.init(*fields)
        s.step(25)
        d = s.step_diagnostics(1)
        out.append((s.get_populations(), d))
        s.close()
    for o in out[1:]:
        assert np.array_equal(out[0][0], o[0])
        for k in ("mass", "jx", "jy", "energy", "rho_min", "theta_min"):
            assert abs(out[0][1][k] - o[1][k]) <= 1e-12 * max(1.0, abs(out[0][1][k])), k


# Sets whose factors 1/(2a) and 1/(2a^2) are no powers of two: a product fused into a sum would show.
@pytest.mark.parametrize("prec", ["f32", "f16dev", "bf16dev"])
@pytest.mark.parametrize("v", [(0, 3, -3, 1, -1), (0, 3, -3, 2, -2), (0, 5, -5, 1, -1)])
def test_layouts_give_the_same_state_for_factors_that_are_no_powers_of_two(prec, v):
    nx, ny = 131, 48
    fields = I.kh_fields(nx, ny=ny)
    out = []
    for plain in (False, True):
        s = plbm.Solver(2, v, 1.1, nx, ny, theta0=1.0, prec=prec, plain_layout=plain, skip_admissibility=True)
        s.init(*fields)
        pops = [s.get_populations()]
        for _ in range(3):
            s.step(1)
            pops.append(s.get_populations())
        out.append(pops)
        s.close()
    for k, (a, b) in enumerate(zip(*out)):
        assert bool(np.isfinite(a).all()) and bool(np.array_equal(a, b)), (k, np.mean(a != b))


# Blocks of 64 and 128 threads of the plain layout, by the columns of a row's last block, against the paired layout.
@pytest.mark.parametrize("prec", ["f32", "f16dev", "bf16dev"])
@pytest.mark.parametrize("nx", [20, 32, 33, 64, 65, 128, 130, 192, 193])
def test_plain_layout_blocks_give_the_paired_state(prec, nx):
    ny = 512
    fields = I.kh_fields(nx, ny=ny)
    out = []
    for plain in (False, True):
        s = plbm.Solver(2, V5, 1.3, nx, ny, theta0=1.0, prec=prec, plain_layout=plain)
        s.init(*fields)
        s.step(5)
        out.append(s.get_populations())
        s.close()
    assert bool(np.array_equal(out[0], out[1]))


# Steps queued back to back (large grids overlap one step's start with the end of the
# step before; small ones do not) equal steps awaited one by one, bit for bit: every
# step kernel, on both sides of the size from which its launches overlap.
@pytest.mark.parametrize("dim,v,shape,prec,kw", [
    (2, I.SET_013, (256, 256), "f32", {}), (2, I.SET_013, (512, 300), "f32", {}), (2, I.SET_013, (1024, 258), "f16dev", {}),
    (2, I.SET_013, (1024, 258), "bf16dev", {}), (2, I.SET_013, (513, 257), "f32", {}), (2, I.SET_D1Q3, (520, 300), "f32",
                                                                                       {"theta0": 1 / 3, "isothermal": True}),
    (2, I.SET_013, (300, 280), "f64", {}), (1, I.SET_013, (70000, 1), "f64", {}), (3, I.SET_013, (64, 40, 30), "f32", {}),
    (3, I.SET_013, (64, 64, 34), "f16dev", {}), (3, I.SET_013, (64, 64, 33), "bf16dev", {}), (3, I.SET_013, (64, 40, 30), "f64", {}),
])
def test_queued_steps_equal_awaited_steps(dim, v, shape, prec, kw):
    import torch
    from paper_1402_5487_gb300 import plbm
    nx, ny, nz = (tuple(shape) + (1,))[:3]
    rng = np.random.default_rng(5)
    shp = (ny, nx) if dim < 3 else (nz, ny, nx)
    one = np.ones(shp)
    u = [0.05 * rng.uniform(-1, 1, shp) for _ in range(3)]
    th = kw.get("theta0", 1.0) * one
    got = []
    for await_each in (False, True):
        s = plbm.Solver(dim, v, 1.1, nx, ny, nz=nz, prec=prec, **kw)
        if dim == 3:
            s.init(one, u[0], u[1], theta=th, uz=u[2])
        else:
            s.init(one, u[0], u[1] if dim == 2 else None, th)
        for _ in range(7 if await_each else 1):
            s.step(1 if await_each else 7)
            if await_each:
                torch.cuda.synchronize()
        got.append(s.get_populations())
        s.close()
    assert np.array_equal(got[0], got[1])


# Small 16/32-bit lattices let the next grid start after their arithmetic (kernels of their own, in both layouts).
@pytest.mark.parametrize("prec", ["f32", "f16dev", "bf16dev"])
@pytest.mark.parametrize("shape", [(101, 97), (128, 128), (33, 5), (255, 255), (256, 254)])
def test_queued_steps_of_small_lattices_equal_awaited_steps(prec, shape):
    test_queued_steps_equal_awaited_steps(2, I.SET_013, shape, prec, {})


# Lattices between the sizes at which one step's start overlaps the step before: launched plainly, with a row's
# last block nearly empty, and FP64 grids of one and three waves.
@pytest.mark.parametrize("dim,v,shape,prec,kw", [
    (2, I.SET_013, (360, 360), "f32", {}), (2, I.SET_013, (360, 360), "f16dev", {}), (2, I.SET_013, (360, 360), "bf16dev", {}),
    (2, I.SET_013, (430, 377), "bf16dev", {}), (2, I.SET_013, (38, 2152), "bf16dev", {}), (2, I.SET_013, (300, 301), "f32", {}),
    (2, I.SET_D1Q3, (405, 134), "f16dev", {"theta0": 1 / 3, "isothermal": True}), (2, I.SET_013, (119, 456), "f64", {}),
    (2, (0, 1, -1, 2, -2, 3, -3), (60, 50), "f64", {"theta0": 0.8}), (3, I.SET_013, (32, 32, 32), "f64", {}), (3, I.SET_013, (64, 64, 64), "f64", {})])
def test_queued_steps_between_the_launch_rules_equal_awaited_steps(dim, v, shape, prec, kw):
    test_queued_steps_equal_awaited_steps(dim, v, shape, prec, kw)


# FP64 sums of five-velocity sets on the integer pipe: fields of given populations against exact
# rational sums, over the exponent range and past both of its ends (there in FP64), with zeros,
# negative values, a spread of 1e-9 and equal values.  A term is held to 2^-57 of the largest, a
# sum and each operation after it round once: 25 2^-57 + 4 2^-53 of the sum of magnitudes.
@pytest.mark.parametrize("kind", ["spread", "mixed", "equal", "zeros"])
@pytest.mark.parametrize("scale", [1.0, 2.0**-958, 2.0**-961, 1e-300, 1e200, 2.0**876, 2.0**879, 1e300])
def test_f64_sums_on_the_integer_pipe(kind, scale):
    from fractions import Fraction as F
    from paper_1402_5487_gb300 import plbm
    nx, ny, v = 5, 4, I.SET_013
    rng = np.random.default_rng(11)
    f = rng.uniform(0.5, 1.0, (25, ny, nx))
    if kind == "spread":
        f *= 10.0 ** rng.uniform(-9, 0, f.shape)
    elif kind == "mixed":
        f *= np.where(rng.uniform(size=f.shape) < 0.2, -0.1, 1.0)
    elif kind == "equal":
        f[:] = 1.0
    else:
        f[rng.uniform(size=f.shape) < 0.5] = 0.0
    f *= scale
    s = plbm.Solver(2, v, 1.1, nx, ny, prec="f64")
    s.set_populations(f)
    rho, ux, uy, th = s.moments()
    s.close()
    for y in range(ny):
        for x in range(nx):
            g = [F(float(a)) for a in f[:, y, x]]
            vx, vy = [v[p // 5] for p in range(25)], [v[p % 5] for p in range(25)]
            m, size = sum(g), sum(abs(a) for a in g)
            jx, jy = sum(a * b for a, b in zip(vx, g)), sum(a * b for a, b in zip(vy, g))
            e = sum((a * a + b * b) * c for a, b, c in zip(vx, vy, g))
            tol = F(25, 2**57) + F(4, 2**53)
            assert abs(F(float(rho[y, x])) - m) <= tol * size
            amp = size / m   # how much the sums cancel
            assert abs(F(float(ux[y, x])) - jx / m) <= 2 * 3 * tol * amp * amp
            assert abs(F(float(uy[y, x])) - jy / m) <= 2 * 3 * tol * amp * amp
            assert abs(F(float(th[y, x])) - (e / m - (jx / m) ** 2 - (jy / m) ** 2) / 2) <= 40 * tol * amp * amp * amp


# The FP64 rule in fixed point, on both sides of the range it is taken in (|u| < 1/2, theta < 3/2, |v| <= 3):
# initial state and one step against the oracle.  Its C mu rule sums five terms of at most 30 (mu_4), 2^-53
# of each; two axes; f' adds omega times that: 1e-12 of the largest population.
@pytest.mark.parametrize("dim", [1, 2])
@pytest.mark.parametrize("iso", [False, True])
@pytest.mark.parametrize("v", [I.SET_013, I.SET_012, (0, 2, -2, 1, -1), (0, 3, -3, 1, -1), (0, 2, -2, 3, -3), (0, 1, -1, 4, -4)])
def test_f64_rule_in_and_out_of_the_fixed_point_range(dim, iso, v):
    rng = np.random.default_rng(13)
    nx, ny = 40, 9 if dim == 2 else 1
    edge = [0.5, np.nextafter(0.5, 0), -0.5, -np.nextafter(0.5, 0), 0.0, -0.0, 1e-300, 2.0**-9, 2.0**-30]
    u = rng.uniform(-0.7, 0.7, (2, ny, nx))
    u[0, 0, :9], u[1, 0, 9:18] = edge, edge
    th = rng.uniform(0.2, 2.0, (ny, nx))
    th[0, :4] = [1.5, np.nextafter(1.5, 0), 1e-12, 1e-300]
    rho = rng.uniform(0.5, 2.0, (ny, nx))
    s = plbm.Solver(dim, v, 1.2, nx, ny, theta0=1.0, prec="f64", isothermal=iso, skip_admissibility=True)
    s.init(rho, u[0], u[1] if dim == 2 else None, None if iso else th)
    lat = O.Lattice(dim, v, 1.2, nx, ny, theta0=1.0, isothermal=iso)
    fo = lat.init(rho, u[0], u[1] if dim == 2 else 0 * u[1], 0 * th + 1.0 if iso else th)
    for k in range(2):
        g = s.get_populations()
        o = np.asarray(fo).reshape(g.shape)
        assert np.max(np.abs(g - o)) <= 1e-12 * np.max(np.abs(o)), k
        if k == 0:
            s.step(1)
            fo = lat.run(fo, 1)
    s.close()


# Fields of FP16 pairs from exact 32-bit sums below 1/4 and in float-float from there on: as the 3D test of
# the same; 25 roundings of 2^-53 of the sum of magnitudes.
# The reciprocal of the FP64 steps and fields, through the velocity of nodes whose momentum is a power of two: within
# half a unit of the last place and 2^-59 over the normal range, the division's value at and beyond its ends.
def test_f64_reciprocal():
    from fractions import Fraction
    rng = np.random.default_rng(6)
    rho = np.concatenate([rng.uniform(1, 2, 3000), -rng.uniform(1, 2, 200), 10.0 ** rng.uniform(-300, 300, 1000),
                          [1.0, np.nextafter(1, 2), np.nextafter(1, 0), np.nextafter(2, 1), 1.5, 4 / 3],
                          2.0 ** np.arange(-1021, -1015), 2.0 ** np.arange(1015, 1023),
                          np.nextafter(2.0**-1021, 0) * np.ones(1), np.nextafter(2.0**1021, 0) * np.ones(1)])
    odd = np.array([0.0, 5e-324, 2.0**-1030, -2.0**-1040, np.inf, -np.inf, np.nan, 1.7e308])
    n = len(rho) + len(odd)
    f = np.zeros((5, n))
    with np.errstate(all="ignore"):
        k = np.floor(np.log2(np.abs(rho))) - 20
        f[1, :len(rho)] = 2.0 ** np.maximum(k, -1074)
        f[0, :len(rho)] = rho - f[1, :len(rho)]
        f[0, len(rho):] = odd
        f[1, len(rho):] = 1.0 / 1024
    s = plbm.Solver(1, I.SET_013, 1.1, n, 1, theta0=1.0, prec="f64")
    s.init(np.ones((1, n)), np.zeros((1, n)), np.zeros((1, n)), np.ones((1, n)))
    s.set_populations(f.reshape(5, 1, n))
    m, u = (np.asarray(a).reshape(-1) for a in s.moments()[:2])
    s.close()
    with np.errstate(all="ignore"):
        total = f[0] + f[1]
        assert np.array_equal(m, total, equal_nan=True)
        assert np.array_equal(u[len(rho):], f[1, len(rho):] * (1.0 / total[len(rho):]), equal_nan=True)
    for r, j, v in zip(total[:len(rho)], f[1], u):
        exact = Fraction(float(j)) / Fraction(float(r))
        if abs(exact) < Fraction(2) ** -1000:
            continue
        err = abs(Fraction(float(v)) - exact)
        assert err <= Fraction(float(np.spacing(abs(float(exact))))) / 2 + abs(exact) / 2**59, (r, j, v)


# The FP64 rule of the symmetric sets in and out of the range of its fixed point: a fluid at rest stays exactly at
# rest, and the mirrored flow is the flow, mirrored, bit for bit.  Sizes on both sides of the number of threads from
# which the conversions are made by integer instructions.
SETS_F64 = [I.SET_013, I.SET_012, (0, 3, -3, 1, -1), (0, 2, -2, 3, -3), (0, 1, -1, 4, -4)]


@pytest.mark.parametrize("v", SETS_F64)
@pytest.mark.parametrize("dim,nx,ny", [(1, 64, 1), (2, 40, 36), (2, 300, 260)])
def test_f64_rest_is_exact(v, dim, nx, ny):
    for th in np.random.default_rng(3).uniform(0.3, 1.6, 12 if nx < 100 else 3):
        s = plbm.Solver(dim, v, 1.1, nx, ny, theta0=float(th), prec="f64", skip_admissibility=True)
        one = np.ones((ny, nx))
        s.init(one, 0 * one, 0 * one, th * one)
        for _ in range(3):
            _, ux, uy, _ = s.moments()
            assert not ux.any() and not uy.any(), (th, np.abs(ux).max())
            s.step(2)
        s.close()


@pytest.mark.parametrize("v", SETS_F64)
@pytest.mark.parametrize("n,speed", [(48, 0.02), (48, 0.6), (264, 0.02)])
def test_f64_steps_commute_with_mirrors(v, n, speed):
    rng = np.random.default_rng(4)
    rho, th = 1.0 + 0.01 * rng.uniform(-1, 1, (2, n, n))
    ux, uy = speed * rng.uniform(-1, 1, (2, n, n))
    ux[3, 5] = uy[7, 2] = 0.0

    def run(f):
        s = plbm.Solver(2, v, 1.0, n, n, theta0=1.0, prec="f64", skip_admissibility=True)
        s.init(*[np.ascontiguousarray(a) for a in f])
        s.step(3)
        out = s.moments()
        s.close()
        return out

    back = -np.arange(n) % n
    ref = run((rho, ux, uy, th))
    for index, sign in ((np.ix_(np.arange(n), back), (1, -1, 1, 1)), (np.ix_(back, np.arange(n)), (1, 1, -1, 1))):
        got = run([g * a[index] for g, a in zip(sign, (rho, ux, uy, th))])
        for g, a, b in zip(sign, got, ref):
            assert bool(np.array_equal(a, g * b[index])), np.abs(a - g * b[index]).max()


@pytest.mark.parametrize("v", [I.SET_013, I.SET_012])
@pytest.mark.parametrize("extra", [None, 0.25, -0.25, 0.2498779296875, -0.2498779296875, 2.0**-24, 7.5, -300.0, np.inf, np.nan])
def test_fp16_fields_from_exact_sums(extra, v):
    nx, ny = 133, 8
    rng = np.random.default_rng(19)
    s = plbm.Solver(2, v, 1.1, nx, ny, theta0=0.7 if max(v) == 2 else 1.0, prec="f16dev")
    one = np.ones((ny, nx))
    s.init(one, 0 * one, 0 * one, (0.7 if max(v) == 2 else 1.0) * one)
    f = s.get_populations()
    g = (0.05 * rng.uniform(-1, 1, f.shape) * 10.0 ** rng.uniform(-5, 0, f.shape)).astype(np.float16).astype(np.float64)
    if extra is not None:
        g[7, 1, 5] = g[20, 6, 132] = extra
    s.set_populations(f + g)
    p = s.get_populations()
    rho, ux, uy, th = s.moments()
    s.close()
    c = np.array([(v[k // 5], v[k % 5]) for k in range(25)], float)
    ok = np.isfinite(p).all(axis=0)
    assert ok.sum() == ok.size - (2 if extra is not None and not np.isfinite(extra) else 0)
    p = np.where(ok, p, 1.0)
    m, size = p.sum(0), np.abs(p).sum(0)
    j = np.einsum("ka,kyx->ayx", c, p)
    e = np.einsum("k,kyx->yx", (c ** 2).sum(1), p)
    tol = 25 * 2.0**-53 * size / np.abs(m)
    assert np.all((np.abs(rho - m) <= tol * np.abs(m))[ok])
    for a, b in zip((ux, uy), j):
        assert np.all((np.abs(a - b / m) <= 2 * 3 * tol * size / np.abs(m))[ok])
    t = (e / m - ((j / m) ** 2).sum(0)) / 2
    assert np.all((np.abs(th - t) <= 2 * 18 * tol * (size / m) ** 2)[ok])
    assert not np.isfinite(rho[~ok]).any()


# The final pass of the reductions (a cluster of blocks over one record per block of a step):
# fewer records than blocks, one per thread, one more, several per thread.  The sums of the
# populations themselves within 1e-13 of the sum of magnitudes, minima those of the fields.
@pytest.mark.parametrize("prec", ["f64", "f32", "bf16dev"])
@pytest.mark.parametrize("shape", [(5, 2), (100, 14), (128, 510), (129, 512), (128, 2049), (130, 4098), (1500, 900)])
def test_final_pass_of_the_reductions(prec, shape):
    from paper_1402_5487_gb300 import plbm
    nx, ny = shape
    rng = np.random.default_rng(7)
    s = plbm.Solver(2, I.SET_013, 1.1, nx, ny, prec=prec)
    one = np.ones((ny, nx))
    s.init(one + 0.01 * rng.uniform(-1, 1, (ny, nx)), *(0.02 * rng.uniform(-1, 1, (2, ny, nx))), one)
    s.step(2)
    # 16/32-bit steps take their sums in FP32 arithmetic before the state is rounded to storage
    for d in ([s.step_diagnostics(3)] if prec == "f64" else []) + [s.diagnostics()]:
        f = s.get_populations().reshape(5, 5, -1)
        v = np.array(I.SET_013, float)
        e2 = v[:, None] ** 2 + v[None, :] ** 2
        for key, w in (("mass", np.ones((5, 5))), ("jx", v[:, None] + 0 * v), ("jy", v[None, :] + 0 * v[:, None]), ("energy", e2)):
            w = np.broadcast_to(w, (5, 5))
            exact = math.fsum((w[:, :, None] * f).ravel())
            assert abs(d[key] - exact) <= 1e-13 * np.sum(np.abs(w[:, :, None] * f)), (key, d[key], exact)
        rho, _, _, th = s.moments()
        assert abs(d["rho_min"] - rho.min()) <= 1e-13 and abs(d["theta_min"] - th.min()) <= 1e-12
        assert d["status"] == 0
    s.close()
    bad = plbm.Solver(2, I.SET_013, 1.1, nx, ny, prec=prec)
    bad.init(one, 0 * one, 0 * one, one)
    g = bad.get_populations()
    g[0, ny - 1, nx - 1] = np.nan
    bad.set_populations(g)
    d = bad.diagnostics()
    assert d["status"] & 1 and np.isnan(d["mass"]) and abs(d["rho_min"] - 1.0) <= 0.02
    bad.close()


# Large lattices advance two steps per launch (strips of columns, segments of rows): the
# state must be that of single steps bit for bit, in both layouts, for odd and even step counts,
# status reads between, a captured stream and a set in either order; strips one column apart in
# width, a last wave with few blocks, few rows and few columns.
@pytest.mark.parametrize("prec,v,shape,plain", [("f32", *c) for c in [
    (I.SET_013, (1024, 1024), False), (I.SET_013, (1009, 1030), False), (I.SET_013, (901, 901), False),
    (I.SET_013, (1200, 902), True), (I.SET_012, (1021, 1026), False), (I.SET_012, (1011, 1021), False),
    ((0, 3, -3, 1, -1), (960, 1026), False), ((0, 2, -2, 1, -1), (1031, 957), False), ((0, 2, -2, 3, -3), (1500, 800), False),
    (I.SET_013, (40000, 100), False), (I.SET_013, (90, 40000), False), (I.SET_013, (40000, 101), False),
    (I.SET_012, (400000, 8), False), (I.SET_013, (700, 1000), False), ((0, 1, -1, 4, -4), (1024, 1024), False)]] + [
    ("f16dev", I.SET_013, (2051, 2050), False), ("f16dev", (0, 3, -3, 1, -1), (2051, 2050), False), ("f16dev", (0, 2, -2, 3, -3), (2050, 2052), False),
    ("f16dev", I.SET_012, (1900, 1726), False),
    ("bf16dev", I.SET_013, (2301, 2204), False), ("bf16dev", (0, 3, -3, 1, -1), (1150, 4412), False),
    ("f16dev", I.SET_013, (2500, 2501), False), ("bf16dev", (0, 2, -2, 1, -1), (2611, 2444), True), ("f16dev", I.SET_013, (1500, 900), False)])
def test_two_steps_of_one_launch_equal_single_steps(prec, v, shape, plain):
    import torch
    from paper_1402_5487_gb300 import plbm
    nx, ny = shape
    g = torch.Generator(device="cuda").manual_seed(3)
    one = torch.ones(ny, nx, dtype=torch.float64, device="cuda")
    u = [0.02 * (torch.rand(ny, nx, dtype=torch.float64, device="cuda", generator=g) - 0.5) for _ in range(2)]
    th0 = 0.7 if max(v) == 2 else 1.0
    side = torch.cuda.Stream()

    def run(parts, ce=0, how="step"):
        s = plbm.Solver(2, v, 1.1, nx, ny, theta0=th0, prec=prec, plain_layout=plain, check_every=ce,
                        skip_admissibility=True, stream=side)
        torch.cuda.synchronize()
        s.init(one, u[0], u[1], th0 * one)
        for k in parts:
            if how == "graph":
                side.synchronize()
                gr = torch.cuda.CUDAGraph()
                with torch.cuda.graph(gr, stream=side):
                    s.step(k)
                with torch.cuda.stream(side):
                    gr.replay()
            elif how == "diag":
                s.step_diagnostics(k)
            else:
                s.step(k)
        side.synchronize()
        out = s.moments(on_device=True)
        side.synchronize()
        pop = s.get_populations() if nx * ny < 1 << 21 else None
        s.close()
        return out, pop

    ref = run((1,) * 11)
    for parts, kw in (((11,), {}), ((2, 3, 6), {}), ((4, 7), {"ce": 5}), ((11,), {"how": "graph"}), ((6, 5), {"how": "diag"})):
        out, pop = run(parts, **kw)
        assert all(torch.equal(a, b) for a, b in zip(ref[0], out)), (parts, kw)
        assert pop is None or np.array_equal(ref[1], pop)


# The same where the library says that it launched once per two steps: shapes well inside the rule on any
# number of SMs, and the flattest ones that it takes (15 and 8 rows of pairs for w = 3 and 2: nearly every
# row pulls across the wrap; the strips fill the resident CTAs exactly).
@pytest.mark.parametrize("prec,v,shape,plain", [
    ("f32", I.SET_013, (2048, 1100), False), ("f32", I.SET_013, (2047, 1101), False), ("f32", I.SET_012, (1700, 1500), True),
    ("f32", (0, 3, -3, 1, -1), (2048, 1100), False), ("f32", I.SET_013, (90 * 2, 32), False), ("f32", I.SET_012, (60 * 8, 16), False),
    ("f16dev", I.SET_013, (2700, 2704), False), ("f16dev", I.SET_012, (2701, 2703), False), ("bf16dev", I.SET_013, (3000, 3002), False)])
def test_lattices_that_take_two_steps_of_one_launch(prec, v, shape, plain):
    import torch
    from paper_1402_5487_gb300 import plbm
    nx, ny = shape
    if nx < 1000:
        nx *= torch.cuda.get_device_properties(0).multi_processor_count
    g = torch.Generator(device="cuda").manual_seed(5)
    one = torch.ones(ny, nx, dtype=torch.float64, device="cuda")
    u = [0.02 * (torch.rand(ny, nx, dtype=torch.float64, device="cuda", generator=g) - 0.5) for _ in range(2)]
    th0 = 0.7 if max(v) == 2 else 1.0
    out = []
    for parts, launches in (((1,) * 8, 8), ((8,), 4), ((3, 5), 3 + 3)):   # as many launches as steps, modulo 2
        s = plbm.Solver(2, v, 1.1, nx, ny, theta0=th0, prec=prec, plain_layout=plain)
        s.init(one, u[0], u[1], th0 * one)
        for k in parts:
            s.step(k)
        assert s.step_launches == launches, (parts, s.step_launches)
        out.append([f.clone() for f in s.moments(on_device=True)])
        s.close()
    for o in out[1:]:
        assert all(torch.equal(a, b) for a, b in zip(out[0], o))


def test_step_launches_counts_what_was_launched():
    from paper_1402_5487_gb300 import plbm
    one = np.ones((64, 64))
    s = plbm.Solver(2, I.SET_013, 1.1, 64, 64, prec="f32")
    s.init(one, 0 * one, 0 * one, one)
    s.step(70)                # two replays of 32 and six single steps
    s.step_diagnostics(3)
    assert s.step_launches == 73
    s.close()
    t = plbm.Solver(1, I.SET_013, 1.1, 1000, 1, prec="f32")
    t.init(np.ones(1000), np.zeros(1000), None, np.ones(1000))
    t.step(64)
    assert 0 < t.step_launches < 64
    t.close()
    assert plbm.lib().plbm_step_launches(None, None) == plbm.PLBM_E_ARG


# Several steps per launch of a 1D lattice cost more arithmetic, the more the wider the velocities: long lattices with
# |v| = 4 and more take single steps, short ones never do.
@pytest.mark.parametrize("prec", ["f32", "bf16dev"])
@pytest.mark.parametrize("v,n,single", [((0, 1, -1, 2, -4), 2000000, True), ((1, -1, 2, -2, 3, -3, 4, -4), 2000000, True),
                                        ((0, 1, -1), 2000000, False), ((1, -1, 2, -2, 3, -3, 4, -4), 1000, False), (I.SET_013, 1000, False)])
def test_1d_steps_per_launch_by_velocities(prec, v, n, single):
    from paper_1402_5487_gb300 import plbm
    one = np.ones((1, n))
    s = plbm.Solver(1, v, 1.1, n, 1, theta0=1.0, prec=prec, skip_admissibility=True)
    s.init(one, 0 * one, 0 * one, one)
    s.step(16)
    assert (s.step_launches == 16) == single
    s.close()


# Two lattices whose rings differ in size (w = 2 and 3), stepped by two threads on streams of their own.
@pytest.mark.parametrize("prec", ["f32", "f16dev"])
def test_two_steps_of_one_launch_from_two_threads(prec):
    import threading
    import torch
    from paper_1402_5487_gb300 import plbm
    L = 2048
    one = torch.ones(L, L, dtype=torch.float64, device="cuda")
    x = torch.arange(L, dtype=torch.float64, device="cuda")
    u = 0.01 * torch.sin(2 * math.pi * x / L)[None, :] * one

    def make(v):
        s = plbm.Solver(2, v, 1.1, L, L, theta0=0.7 if max(v) == 2 else 1.0, prec=prec, stream=torch.cuda.Stream())
        torch.cuda.synchronize()
        s.init(one, u, -u, (0.7 if max(v) == 2 else 1.0) * one)
        return s

    got = []
    for threads in (False, True):
        sols = [make(v) for v in (I.SET_012, I.SET_013)]
        work = [threading.Thread(target=lambda s=s: [s.step(4) for _ in range(30)]) for s in sols]
        for w in work:
            w.start()
            if not threads:
                w.join()
        for w in work:
            w.join()
        torch.cuda.synchronize()
        assert all(s.check() == plbm.PLBM_OK for s in sols)
        out = [s.moments(on_device=True) for s in sols]
        torch.cuda.synchronize()
        got.append(out)
        for s in sols:
            s.close()
    for a, b in zip(*got):
        assert all(torch.equal(p, q) for p, q in zip(a, b))


# FP64 steps of five-velocity sets: the symmetric ones in either order of a and b,
# thermal and isothermal, with fixed ends, on one row, at another density scale, and a
# set in an order the symmetric core does not take; 60 steps within 1e-12 of the oracle.
@pytest.mark.parametrize("dim,v,theta0,omega,iso,fixed,shape,scale", [
    (2, (0, 3, -3, 1, -1), 1.0, 1.3, False, False, (70, 19), 1.0),
    (2, (0, 1, -1, 2, -2), 0.7, 1.1, True, False, (33, 8), 1.0),
    (2, (0, 1, -1, 3, -3), 1.0, 1.2, False, True, (65, 5), 1.0),
    (2, (0, 1, -1, 3, -3), 1.0, 1.2, False, False, (1, 9), 1.0),
    (2, (0, 1, -1, 3, -3), 1.0, 1.2, False, False, (40, 12), 1e3),
    (2, (1, 0, -1, 3, -3), 1.0, 1.2, False, False, (40, 12), 1.0),
    (1, (0, 3, -3, 1, -1), 1.0, 1.3, False, True, (257, 1), 1.0),
    (1, (0, 1, -1, 2, -2), 0.7, 1.1, True, False, (64, 1), 1.0),
])
def test_f64_five_velocity_steps_match_oracle(dim, v, theta0, omega, iso, fixed, shape, scale):
    nx, ny = shape
    rho, ux, uy, th = smooth_fields(nx, ny, 7, amp_u=0.03, amp_r=0.01, theta0=theta0)
    fields = (scale * rho, ux, uy if dim == 2 else 0 * uy, th)
    ends = {"bc": "fixed", "left": (1.02 * scale, 0.01, theta0), "right": (0.99 * scale, 0.0, theta0)} if fixed else {}
    mg, fg, _ = gpu_run(dim, v, omega, nx, ny, fields, 60, theta0=theta0, isothermal=iso, **ends)
    _, fo, mo = oracle_run(dim, v, omega, nx, ny, fields, 60, theta0=theta0, isothermal=iso, **ends)
    assert rel(fg, fo) <= TOL64
    assert O.rel_err(mg[0], mo[0]) <= TOL64 and O.rel_err(mg[3], mo[3]) <= TOL64


# Several 1D steps per launch (a warp steps the 32 nodes around its outputs) equal the
# oracle and, for every split of the same number of steps, each other bit for bit: every
# q1, periodic and fixed ends, thermal and isothermal, lattices shorter than a warp,
# of one tile more or less, and long ones that take one step per launch.  (The
# six-velocity set is linearly unstable, |lambda| = 1.17: any rounding grows 8e4-fold in
# 71 steps, so it is held to the bitwise comparison alone.)
@pytest.mark.parametrize("v,theta0,iso,tol32", [((0, 1, -1), 1 / 3, True, 2e-6), ((1, -1, 3, -3), 4 / 3, True, 2e-6),
                                                ((0, 1, -1, 3, -3), 1.0, False, 1e-5), ((0, 3, -3, 1, -1), 1.0, False, 1e-5),
                                                ((1, 0, -1, 3, -3), 1.0, False, 1e-5), ((0, 1, -1, 2, -2, 3), 0.8, False, 1e-5),
                                                ((0, 1, -1, 2, -2, 3, -3), 1.0, False, 1e-5),
                                                ((0, 1, -1, 2, -2, 3, -3, 4), 1.0, False, 1e-5)])
@pytest.mark.parametrize("n,bc", [(5, "periodic"), (31, "fixed"), (96, "periodic"), (97, "fixed"), (1000, "fixed"),
                                  (40000, "periodic")])
def test_steps_of_one_launch_match_oracle_and_single_steps(v, theta0, iso, tol32, n, bc):
    x = np.arange(n)
    rho = (1 + 0.01 * np.sin(2 * np.pi * x / n))[None]
    ux = (0.01 * np.cos(2 * np.pi * x / n))[None]
    th = np.full((1, n), theta0)
    ends = {"left_state": (1.0, 0.01, theta0), "right_state": (1.0, 0.01, theta0)} if bc == "fixed" else {}
    lat = O.Lattice(1, v, 1.1, n, 1, bc=bc, theta0=theta0, isothermal=iso, **ends)
    fo = lat.run(lat.init(rho, ux, 0 * ux, th), 71)
    stable = plbm.linear_stability(1, v, 1.1, theta0, 0.01, isothermal=iso) <= 1 + 1e-9
    for prec, tol in (("f64", TOL64), ("f32", tol32), ("f16dev", 2e-2), ("bf16dev", 1e-1)):
        got = []
        for parts in ((71,), (64, 7), (1,) * 71, (3, 2, 5, 61)):
            s = plbm.Solver(1, v, 1.1, n, 1, theta0=theta0, prec=prec, bc=bc, isothermal=iso, **ends)
            s.init(rho, ux, None, None if iso else th)
            for k in parts:
                s.step(k)
            assert s.check() == plbm.PLBM_OK or not stable
            got.append(s.get_populations())
            s.close()
        assert rel(got[0], np.asarray(fo).reshape(got[0].shape)) <= tol or not stable
        for g in got[1:]:
            assert np.array_equal(got[0], g, equal_nan=True)
