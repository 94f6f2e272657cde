"""The engine's host side on the CPU: the library linked against a fake CUDA runtime (host_engine.py)."""
import ctypes
import gc
import os
import subprocess
import sys

import pytest

import host_engine
import paper_0906_5170_gb300 as pk
import workloads as W

TESTS = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def lib_path():
    return host_engine.build()


@pytest.fixture
def fake(lib_path):
    old = pk.capi._lib
    L = host_engine.load(lib_path)
    L.fake_reset()
    yield L
    gc.collect()             # handles of the fake library are released by it
    pk.capi._lib = old


TICKET_AFTER_PLAN = """
import ctypes, sys
sys.path[:0] = [{root!r}, {tests!r}]
import host_engine, workloads as W
import paper_0906_5170_gb300 as pk
L = host_engine.load({lib!r})
c = pk.Context(0)
for cancel in (False, True):
    pl = c.plan(W.piston_small(n_steps=60, precision="fp32"))
    updates = pl.info()["cell_updates"]
    t = pl.submit()
    pl.close()                     # returns once the request has finished
    if cancel:
        t.cancel()                 # of a finished request: no effect
    F, err, st = t.force(-1)
    assert st["cell_updates"] == updates, st
c.close()
"""


def test_ticket_outlives_its_plan(lib_path):
    # a plan has to live until its requests have finished, and its tickets are collected after that:
    # casimir_force and casimir_cancel read nothing of the plan (freed memory is overwritten here)
    script = TICKET_AFTER_PLAN.format(root=os.path.dirname(TESTS), tests=TESTS, lib=lib_path)
    r = subprocess.run([sys.executable, "-c", script], env=dict(os.environ, MALLOC_PERTURB_="165"),
                       capture_output=True, text=True, timeout=120)
    assert r.returncode == 0, (r.returncode, r.stderr[-2000:])


def test_result_buffer_of_a_failed_run_is_not_reused(fake):
    # its copies may still be in flight: only a request whose results have landed leaves its pinned buffer
    # to the next one
    c = pk.Context(0)
    pl = c.plan(W.piston_small(n_steps=60, precision="fp32"))
    pl.run()
    assert fake.fake_host_frees() == 0          # kept
    fake.fake_fail_late(1)
    with pytest.raises(pk.CasimirError):
        pl.run()
    fake.fake_fail_late(0)
    assert fake.fake_host_frees() == 1
    pl.run()
    c.close()


EXIT_WITH_OPEN_HANDLES = """
import sys
sys.path[:0] = [{root!r}, {tests!r}]
import host_engine, workloads as W
import paper_0906_5170_gb300 as pk
L = host_engine.load({lib!r})
c = pk.Context(0)
pl = c.plan(W.piston_small(n_steps=60, precision="fp32"))
t = pl.submit()
t.force(-1)
def hold():
    return c, pl, t
{end}
"""


@pytest.mark.parametrize("end", ["", "hold.cycle = [c, pl, hold]; del c, pl, t, hold; import gc; gc.collect()"])
def test_context_and_plans_are_released_in_any_order(lib_path, end):
    # the garbage collector finalises a context and its plans in no set order, weak references cleared first
    script = EXIT_WITH_OPEN_HANDLES.format(root=os.path.dirname(TESTS), tests=TESTS, lib=lib_path, end=end)
    r = subprocess.run([sys.executable, "-c", script], env=dict(os.environ, MALLOC_PERTURB_="165"),
                       capture_output=True, text=True, timeout=120)
    assert r.returncode == 0, (r.returncode, r.stderr[-2000:])


def test_planning_leaves_the_callers_device_current(fake):
    c = pk.Context(1)
    fake.fake_device(0)
    for p in (W.piston_small(n_steps=60, precision="fp32"), W.cylinder_piston(10, [0, 1], t_max=2.0)):
        with_resident = c.plan(p)
        assert fake.fake_device(-1) == 0
        with_resident.close()
    c.close()


SHAPE_SIZES = [(60, 20, 96), (3, 12, 4), (400, 166, 640), (400, 80, 64), (512, 512, 64), (128, 128, 320), (37, 901, 7), (251, 93, 40)]


@pytest.mark.parametrize("cyl,fp64", [(0, 0), (0, 1), (1, 0), (1, 1)])
@pytest.mark.parametrize("nx,ny,nsims", SHAPE_SIZES)
def test_resident_shapes_come_best_first_and_are_looked_up_as_needed(fake, cyl, fp64, nx, ny, nsims):
    # the order is that of the model over every shape that fits, ties in the order of rows and cluster size
    def first(most):
        shapes, clocks = (ctypes.c_int * 64)(), (ctypes.c_double * 64)()
        n = fake.fake_res_shapes(cyl, fp64, nx, ny, nsims, most, shapes, clocks)
        return [(clocks[i], shapes[i]) for i in range(n)]
    every = first(64)
    assert every == sorted(every) and len(set(every)) == len(every)
    queries = fake.fake_queries()
    fake.fake_reset()
    assert first(1) == every[:1]
    assert fake.fake_queries() <= max(4, 2 * queries // 3)


@pytest.mark.parametrize("steps,per_launch", [(90, 3), (301, 3), (64, 1), (77, 2)])
def test_kernel_launches_are_counted(fake, steps, per_launch):
    c = pk.Context(0)
    pl = c.plan(W.piston_small(n_steps=steps, precision="fp32"), options={"steps_per_launch": per_launch})
    fake.fake_reset()
    st = pl.run()[2]
    assert st["kernel_launches"] == fake.fake_launches(b"") - fake.fake_launches(b"inject")
    c.close()


@pytest.mark.parametrize("limit_ms", [50.0, 200.0, 1000.0])
def test_a_watched_run_takes_few_more_launches(fake, limit_ms):
    # 64 simulations of 400 x 80: 0.5 ms a launch of 192 steps; a watched chunk still ends well inside the limit
    p = W.config2_piston(W.config2_heights()[0], n_harm=4, n_steps=20000)
    c = pk.Context(0)
    pl = c.plan(p)
    fake.fake_reset()
    fake.fake_cost(b"k_res2d", 0.5)
    pl.run()
    plain = fake.fake_launches(b"k_res2d")
    c.set_watchdog(limit_ms)
    fake.fake_reset()
    fake.fake_cost(b"k_res2d", 0.5)
    pl.run()
    assert plain <= fake.fake_launches(b"k_res2d") <= 1.05 * plain + 2
    c.close()


@pytest.mark.parametrize("how", ["run", "submit"])
def test_a_failed_resident_run_stops_at_its_chunk(fake, how):
    # a wait that ran out is seen after the chunk it happened in, not at the end of the run's 20000 steps
    c = pk.Context(0)
    pl = c.plan(W.config2_piston(W.config2_heights()[0], n_harm=4, n_steps=20000))
    fake.fake_reset()
    fake.fake_fail_resident(1)
    with pytest.raises(pk.CasimirError) as e:
        pl.run() if how == "run" else pl.submit().force(-1)
    assert e.value.code == pk.capi.ECUDA and "ran out" in str(e.value)
    assert fake.fake_launches(b"k_res2d") == 1
    fake.fake_fail_resident(0)
    pl.run()                    # the next run's status is its own
    c.close()


@pytest.mark.parametrize("make", [lambda: W.piston_small(n_steps=60, precision="fp32"), lambda: W.piston_small(n_steps=60, precision="fp64"),
                                  lambda: W.cylinder_piston(20, [0, 1, 2], t_max=3.0, n_harm=20, precision="fp64")])
def test_harmonics_of_a_face_share_their_resident_tables(fake, make):
    # the tables of a simulation's layout are one per lattice, face and source component, not one per harmonic
    c = pk.Context(0)
    resident = c.plan(make()).info()
    other = c.plan(make(), options={"steps_per_launch": 2}).info()
    assert resident["device_bytes"] <= 1.005 * other["device_bytes"]
    c.close()


@pytest.mark.parametrize("p,kernel,other", [
    (W.piston_small(n_steps=60, precision="fp32"), b"k_res2d", b"k_step2d"),
    (W.piston_small(n_steps=60, precision="fp64"), b"k_res2d", b"k_step2d"),
    (W.cylinder_piston(10, [0, 1], t_max=2.0), b"k_rescyl", b"k_cyl")])
def test_options_of_a_plan_give_the_same_plan(fake, p, kernel, other):
    c = pk.Context(0)
    o = c.plan(p).options()
    assert o["resident"] == 1
    pl = c.plan(p, options=o)
    assert pl.options() == o
    fake.fake_reset()
    pl.run()
    assert fake.fake_launches(kernel) > 0 and fake.fake_launches(other) == 0
    # a number of steps per launch alone still names a kernel of that many
    o.pop("resident")
    pl = c.plan(p, options=o)
    assert pl.options() == o
    fake.fake_reset()
    pl.run()
    assert fake.fake_launches(kernel) == 0 and fake.fake_launches(other) > 0
    # asked for where it does not fit: the kernel of that many steps
    big = W.config2_piston(W.config2_heights()[0], n_harm=1, n_steps=12)
    big["n"] = [400, 1000, 1]
    o = c.plan(big, options={"steps_per_launch": 3, "resident": 1}).options()
    assert o["steps_per_launch"] == 3 and "resident" not in o
    c.close()


def _cell(nx, ny, steps=200):
    p = W._base(2, (nx, ny, 1), 10.0, steps)
    p["faces"] = W.box_faces([3.0, 3.0], [6.0, 5.0], 2)
    p.update(n_harm=1, polarization="TE+TM", precision="fp32", force_axis=0)
    return p


def test_autotuning_knows_the_resident_marches(fake):
    c = pk.Context(0)
    c.set_autotune(True)
    cyl = W.cylinder_piston(10, [0, 1], t_max=2.0)
    # a class keeps the default unless another candidate is clearly faster
    fake.fake_cost(b"k_rescyl", 64 * 0.010)
    fake.fake_cost(b"k_march6", 0.0099)
    fake.fake_cost(b"k_cyl2", 0.0099)
    pl = c.plan(cyl)
    assert pl.options()["resident"] == 1
    fake.fake_reset()
    pl.run()
    assert fake.fake_launches(b"k_rescyl") > 0
    assert c.plan(W.cylinder_piston(10, [0, 1], t_max=2.0, below=0.4)).options()["resident"] == 1
    # a grid too large for a cluster and a smaller one of the same class (size to a factor of two)
    fake.fake_reset()
    fake.fake_cost(b"k_step2d_tk", 0.0101)
    fake.fake_cost(b"k_step2d", 0.010)
    assert "resident" not in c.plan(_cell(400, 500)).options()
    # each kernel tried once: 43 launches of three steps, 64 of two, 128 of one
    assert fake.fake_launches(b"k_step2d_tk") == 43
    pl = c.plan(_cell(400, 280))
    assert pl.options()["resident"] == 1
    c.close()
    # clearly faster: it is kept, for both
    c = pk.Context(0)
    c.set_autotune(True)
    fake.fake_reset()
    fake.fake_cost(b"k_rescyl", 64 * 0.010)
    fake.fake_cost(b"k_march6", 0.010)
    fake.fake_cost(b"k_cyl2", 0.002)
    for below in (0.5, 0.4):
        o = c.plan(W.cylinder_piston(10, [0, 1], t_max=2.0, below=below)).options()
        assert "resident" not in o and o["steps_per_launch"] in (1, 2)
    c.close()


def test_a_budget_that_held_the_multi_step_plan_still_does(fake):
    p = W.piston_small(n_steps=60, precision="fp64")
    c = pk.Context(0)
    resident, other = c.plan(p).info()["device_bytes"], c.plan(p, options={"steps_per_launch": 2}).info()["device_bytes"]
    c.close()
    assert resident > other
    for autotune in (False, True):
        c = pk.Context(0, hbm_budget_bytes=other)
        c.set_autotune(autotune)
        pl = c.plan(p)
        assert "resident" not in pl.options()
        pl.run()
        pl.close()
        c.close()
    c = pk.Context(0, hbm_budget_bytes=other - 1)
    with pytest.raises(pk.CasimirError) as e:
        c.plan(p)
    assert e.value.code == pk.capi.ENOMEM
    c.close()
