"""Batched runner on the GPU: the four launch schemes agree bit for bit, agree
with single-lattice handles, and match the FP64 oracle per instance.  The
instances of the sweep have odd and even sides (reading R10: any integer side),
so a batch holds row-paired lattices and plain-layout ones; a mixed batch adds
FP64, FP16, isothermal D2Q9 and D2Q16 lattices."""
import numpy as np
import pytest

import oracle as O
from paper_1402_5487_gb300 import batch as B, build, inputs as I, plbm

from parity_util import field_errors, oracle_run

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    build.build()
    plbm.lib()


@pytest.fixture(scope="module")
def small_instances():
    inst, _ = B.draw_instances(10, seed=4242, size_lo=16, size_hi=150)
    assert any(i.L % 2 for i in inst) and any(i.L % 2 == 0 for i in inst)
    return inst


def _mixed():
    """Lattices of every group kind: row-paired FP32 and FP16, plain-layout FP32 (odd
    side), FP64, FP16 (odd side), isothermal D2Q9 and isothermal D2Q16."""
    mk = lambda k, L, v, om, th, kind, prec=None, iso=False: I.Instance(
        index=k, L=L, v=v, omega=om, theta0=th, kind=kind, seed=700 + k, prec=prec, isothermal=iso)
    return [mk(0, 37, I.SET_013, 1.3, 1.0, "kh"), mk(1, 40, I.SET_012, 1.2, 0.7, "kh"),
            mk(2, 33, I.SET_013, 1.1, 0.9, "shear", prec="f64"), mk(3, 36, I.SET_013, 1.25, 1.0, "kh", prec="f16dev"),
            mk(4, 35, I.SET_012, 1.0, 0.8, "shear", prec="f16dev"),
            mk(5, 30, (0, 1, -1), 1.2, 1.0 / 3.0, "shear", iso=True),
            mk(6, 25, (1, -1, 3, -3), 1.1, 4.0 / 3.0, "shear", iso=True),
            mk(7, 64, I.SET_013, 1.3, 1.0, "kh", prec="f64")]


def _run(instances, mode, steps, prec="f32", config=None, order=None):
    b = B.Batch(instances, prec=prec)
    if config:
        b.set_config(*config)
    if order:
        b.set_order(order)
    b.init()
    b.step(steps, mode)
    pops = [s.get_populations() for s in b.solvers]
    st = b.check()
    b.close()
    return pops, st


def test_launch_schemes_bit_identical(small_instances):
    ref, st = _run(small_instances, "persistent", 7)
    assert st[0] == plbm.PLBM_OK
    for mode in ("persistent_graph", "per_instance", "per_instance_graph"):
        got, _ = _run(small_instances, mode, 7)
        for a, b in zip(got, ref):
            assert np.array_equal(a, b), mode
    for cfg in ((64, 1), (256, 2), (128, 0)):
        for order in ("contiguous", "interleaved"):
            got, _ = _run(small_instances, "persistent_graph", 7, config=cfg, order=order)
            for a, b in zip(got, ref):
                assert np.array_equal(a, b), (cfg, order)


def test_batch_equals_single_handles(small_instances):
    got, _ = _run(small_instances, "persistent_graph", 12)
    for inst, g in zip(small_instances, got):
        s = plbm.Solver(2, inst.v, inst.omega, inst.L, inst.L, theta0=inst.theta0, prec="f32")
        s.init(*I.instance_fields(inst))
        s.step(12)
        assert np.array_equal(s.get_populations(), g)
        s.close()


@pytest.mark.parametrize("prec,tol", [("f32", 1e-5), ("f16dev", 5e-3)])
def test_batch_instances_vs_oracle_100_steps(small_instances, prec, tol):
    b = B.Batch(small_instances, prec=prec)
    b.init()
    b.step(100, "persistent_graph")
    for inst, s in zip(small_instances, b.solvers):
        _, _, mo = oracle_run(2, inst.v, inst.omega, inst.L, inst.L, I.instance_fields(inst), 100,
                              theta0=inst.theta0)
        mg = s.moments()
        e = field_errors(mg, mo)
        # velocity error on the scale of the sweep's largest flow (0.1): 16-bit storage
        # resolves a 1e-3 shear wave only to about 1 % of its own amplitude
        du = np.max(np.hypot(mg[1] - mo[1], mg[2] - mo[2])) / 0.1
        assert e["rho"] <= tol and e["theta"] <= tol and du <= tol, (inst, e, du)
    assert b.check()[0] == plbm.PLBM_OK
    b.close()


def test_autotune_and_cache(tmp_path, small_instances):
    b = B.Batch(small_instances)
    b.init()
    cache = str(tmp_path / "tune.json")
    c1 = b.autotune(steps_per_trial=2, cache_path=cache)
    assert c1["block_x"] in (64, 128, 256) and c1["ctas_per_sm"] >= 1 and not c1["cached"]
    info = b.info()
    assert info["block_x"] == c1["block_x"] and info["ctas"] >= 1
    c2 = b.autotune(cache_path=cache)
    assert c2["cached"] and c2["block_x"] == c1["block_x"]
    with pytest.raises(plbm.PlbmError):
        b.set_config(96, 1)
    b.close()


def test_unstable_instance_is_reported():
    inst, _ = B.draw_instances(3, seed=99, size_lo=32, size_hi=64)
    bad = I.Instance(index=3, L=48, v=I.SET_013, omega=1.8, theta0=1.0, kind="kh", seed=5)
    b = B.Batch(inst + [bad])
    b.init()
    b.step(400, "persistent_graph")
    st, first = b.check()
    assert st == plbm.PLBM_E_DIVERGED and first == 3
    b.close()


def test_instance_handles_are_owned_by_the_batch(small_instances):
    b = B.Batch(small_instances[:2])
    h = b.solvers[0].h
    assert plbm.lib().plbm_destroy(h) == plbm.PLBM_E_STATE
    b.close()


def test_mixed_batch_groups_schemes_and_single_handles():
    inst = _mixed()
    b = B.Batch(inst, prec="f32")
    paired, plain, launches = b.groups()
    # five-velocity thermal 16/32-bit groups (f32: 37 odd, 40 even; f16: 36 even, 35 odd) and
    # one-node-per-thread groups (f64 q5 x2, isothermal f32 q3, isothermal f32 q4)
    assert (paired, plain) == (4, 4) and launches == 5
    b.close()
    ref, st = _run(inst, "persistent", 9)
    assert st[0] == plbm.PLBM_OK
    for mode in ("persistent_graph", "per_instance", "per_instance_graph"):
        got, _ = _run(inst, mode, 9)
        for a, c in zip(got, ref):
            assert np.array_equal(a, c), mode
    for i, g in zip(inst, ref):
        s = plbm.Solver(2, i.v, i.omega, i.L, i.L, theta0=i.theta0, prec=i.prec or "f32", isothermal=i.isothermal)
        rho, ux, uy, th = I.instance_fields(i)
        s.init(rho, ux, uy, None if i.isothermal else th)
        s.step(9)
        assert np.array_equal(s.get_populations(), g), i
        s.close()


def test_mixed_batch_instances_vs_oracle_100_steps():
    inst = _mixed()
    b = B.Batch(inst, prec="f32")
    b.init()
    b.step(100, "persistent_graph")
    tol = {"f64": 1e-12, "f32": 1e-5, "f16dev": 5e-3}
    for i, s in zip(inst, b.solvers):
        _, _, mo = oracle_run(2, i.v, i.omega, i.L, i.L, I.instance_fields(i), 100, theta0=i.theta0,
                              isothermal=i.isothermal)
        mg = s.moments()
        e = field_errors(mg, mo)
        du = np.max(np.hypot(mg[1] - mo[1], mg[2] - mo[2])) / 0.1
        t = tol[i.prec or "f32"]
        assert e["rho"] <= t and e["theta"] <= t and du <= t, (i, e, du)
    assert b.check()[0] == plbm.PLBM_OK
    b.close()


# FP32 lattices beyond the second-level cache take two steps per launch in runs of four: both layouts,
# sets with w = 2 and 3 in either order, strips of one column more or less, a thin lattice, beside
# groups that take single steps; every scheme, and instances stepped alone between (an even number).
def test_two_steps_per_launch_of_a_batch_equal_single_steps():
    mk = lambda k, L, v, om, th, prec=None: I.Instance(index=k, L=L, v=v, omega=om, theta0=th, kind="kh", seed=900 + k, prec=prec)
    v2, v3 = I.SET_012, I.SET_013
    inst = [mk(0, 514, v3, 1.3, 1.0), mk(1, 513, v2, 1.2, 0.7), mk(2, 181, v3, 1.1, 1.0), mk(3, 98, v3, 1.2, 0.9),
            mk(4, 60, v2, 1.1, 0.8), mk(5, 640, (0, 3, -3, 1, -1), 1.2, 1.0), mk(6, 187, (0, 2, -2, 1, -1), 1.1, 0.7),
            mk(7, 12, v3, 1.2, 1.0), mk(8, 9, v2, 1.2, 0.7), mk(9, 72, v3, 1.3, 1.0, "f64"), mk(10, 66, v3, 1.2, 1.0, "f16dev")]
    got = []
    for parts, mode in (((11,), "per_instance"), ((11,), "persistent"), ((11,), "persistent_graph"), ((4, 6, 1), "persistent_graph"),
                        ((1, 10), "persistent"), ((5, -2, 4), "persistent_graph")):
        b = B.Batch(inst, prec="f32")
        b.init()
        for k in parts:
            if k > 0:
                b.step(k, mode)
            else:
                for s in b.solvers:
                    s.step(-k)
        assert b.check()[0] == plbm.PLBM_OK
        got.append([s.get_populations() for s in b.solvers])
        b.close()
    for g in got[1:]:
        assert all(np.array_equal(x, y) for x, y in zip(got[0], g))


# A group large enough for its pieces to be chosen (the test above stays below that): pieces of every width, both
# layouts, thin lattices down to the fewest rows (2w), sets with w = 2 and 3 in either order, beside groups
# that take single steps.  Against one launch per instance and step, bit for bit, and by the number of launches.
def _beyond_the_cache(more=()):
    v2, v3 = I.SET_012, I.SET_013
    mem = [(1100, v3), (1001, v2), (1003, v3), (514, v3), (513, v2), (181, v3), (98, v3), (60, v2), (640, (0, 3, -3, 1, -1)),
           (187, (0, 2, -2, 1, -1)), (12, v3), (9, v2), (7, v3), (8, v2), (5, v2), (97, v3), (90, v3), (91, v3), *more]
    inst = [I.Instance(index=k, L=L, v=v, omega=1.1 + 0.01 * k, theta0=1.6 if {2, 3} <= set(v) else 0.7 if max(v) == 2 else 1.0, kind="kh",
                       seed=950 + k)
            for k, (L, v) in enumerate(mem)]
    n = len(inst)
    return inst + [I.Instance(index=n, L=72, v=v3, omega=1.3, theta0=1.0, kind="kh", seed=7, prec="f64"),
                   I.Instance(index=n + 1, L=66, v=v3, omega=1.2, theta0=1.0, kind="kh", seed=8, prec="f16dev")]


def _runs_equal_single_launches(inst):
    fields = [I.instance_fields(x) for x in inst]
    ref = None
    # parts of a run (negative: each instance stepped on its own), scheme, step kernels launched for the FP32 group
    for parts, mode, launches in (((11,), "per_instance", None), ((11,), "persistent", 2 * 2 + 3), ((11,), "persistent_graph", 2 * 2 + 3),
                                  ((4, 6, 1), "persistent_graph", 2 + (2 + 2) + 1), ((1, 10), "persistent", 1 + (2 * 2 + 2)),
                                  ((5, -2, 4), "persistent_graph", (2 + 1) + 2)):
        b = B.Batch(inst, prec="f32")
        for s, f in zip(b.solvers, fields):
            s.init(*f)
        for k in parts:
            if k > 0:
                b.step(k, mode)
            else:
                for s in b.solvers:
                    s.step(-k)
        assert b.check()[0] == plbm.PLBM_OK
        if launches is not None:   # the other two groups take one launch a step
            assert b.step_launches == launches + 2 * sum(k for k in parts if k > 0)
        got = [s.get_populations() for s in b.solvers]
        b.close()
        ref = ref or got
        for x, a, c in zip(inst, ref, got):
            assert np.array_equal(a, c), (x.L, x.v, parts, mode)


def test_batches_beyond_the_cache_take_two_steps_per_launch():
    _runs_equal_single_launches(_beyond_the_cache())


# Odd sides (plain layout, packed arithmetic over two columns in the fused kernel) with sets whose factors 1/(2a)
# and 1/(2a^2) are no powers of two.
def test_batches_of_two_steps_per_launch_with_factors_that_are_no_powers_of_two():
    _runs_equal_single_launches(_beyond_the_cache([(371, (0, 3, -3, 1, -1)), (229, (0, 3, -3, 2, -2)), (370, (0, 3, -3, 2, -2)),
                                                   (13, (0, 3, -3, 1, -1))]))


def test_autotune_times_the_kernel_whose_shape_it_chooses():
    # the shape and order are those of the single-step kernel; a group that takes two steps per launch in runs of four
    # has to be timed by single steps all the same
    b = B.Batch(_beyond_the_cache()[:-2], prec="f32")
    b.init()
    shapes = 0
    for bx in (64, 128, 256):
        b.set_config(bx, 0)
        shapes += b.info()["max_ctas_per_sm"]
    b.step(4, "persistent")
    assert b.step_launches == 2
    b.autotune(steps_per_trial=6)
    assert b.step_launches == 2 + 2 * shapes * (2 + 6)   # two orders; two steps before each trial
    b.step(4, "persistent")
    assert b.step_launches == 4 + 2 * shapes * (2 + 6)
    assert b.check()[0] == plbm.PLBM_OK
    b.close()


def test_full_sweep_sampled_nodes():
    # The bench's sweep (256 instances drawn by the R8 gates, sides over every
    # integer of [64, 1024], 1.0e8 nodes) in its timed launch scheme: after k steps a
    # node depends only on nodes within 3k, so the oracle advances a (6k+1)^2
    # periodic window of the instance's own fields around sampled nodes.
    from parity_util import patch_fields
    inst, _ = B.draw_instances(256)
    b = B.Batch(inst, prec="f32")
    b.init()
    k, half = 4, 12
    b.step(k, "persistent_graph")
    assert b.check()[0] == plbm.PLBM_OK
    odd = [i for i, x in enumerate(inst) if x.L % 2][:4]
    even = [i for i, x in enumerate(inst) if x.L % 2 == 0][:4]
    rng = np.random.default_rng(21)
    for idx in odd + even:
        x = inst[idx]
        fields = I.instance_fields(x)
        mg = b.solvers[idx].moments()
        for _ in range(3):
            cx, cy = (int(a) for a in rng.integers(0, x.L, 2))
            pf = patch_fields(fields, cx, cy, half, x.L, x.L)
            _, _, mo = oracle_run(2, x.v, x.omega, 2 * half + 1, 2 * half + 1, pf, k, theta0=x.theta0)
            for f_g, f_o, scale in zip(mg, mo, (1.0, 0.1, 0.1, x.theta0)):
                assert abs(f_g[cy, cx] - f_o[half, half]) <= 1e-6 * scale, (idx, x.L, cx, cy)
    b.close()
