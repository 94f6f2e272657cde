"""Which kernel a plan takes, and each against another: resident marches at sizes that do take them (grids
narrower than a thread's columns, one row high, as wide as a CTA has threads, as large as a cluster holds),
the multi-step kernels where they do not or where the options name them.

Fields are equal bit for bit, so contributions differ only by the order of FP64 sums of T weighted samples:
16 u sqrt(T) of the largest contribution."""
import numpy as np
import pytest

import workloads as W
from test_gpu_parity import _check, _tiny_2d, ctx, pk  # noqa: F401  (fixtures)
from test_gpu_resident import _box, _cylinder

pytestmark = pytest.mark.gpu


def _line(nx, ny, prec, steps):
    """A periodic cell with a dielectric block and one short line through its middle."""
    d = 0.1
    p = W._base(2, (nx, ny, 1), 10.0, steps)
    p["bc"] = ["periodic", "periodic", "pec"]
    p["objects"] = [{"shape": "box", "lo": [0.3 * nx * d, 0.35 * ny * d, 0], "hi": [0.55 * nx * d, 0.7 * ny * d, 0],
                     "kind": "dielectric", "eps": 3.0, "mu": 1.0}]
    i0 = int(0.2 * nx)
    i1 = min(nx, i0 + max(1, min(nx // 2, 40)))
    p["faces"] = [{"axis": 1, "sign": 1, "pos": 0.5 * ny * d, "lo": [i0 * d, 0.5 * ny * d, 0.0], "hi": [i1 * d, 0.5 * ny * d, 0.0]}]
    p["force_axis"] = 1
    p.update(n_harm=2, polarization="TE+TM", precision=prec)
    return p


def _against(ctx, p, options, resident):
    pl = ctx.plan(p)
    assert pl.options().get("resident", 0) == resident
    _, per, _ = pl.run(per_sim=True)
    _, ref, _ = ctx.plan(p, options=options).run(per_sim=True)
    lim = 16 * 2.0 ** -53 * np.sqrt(p["n_steps"]) * np.max(np.abs(ref))
    assert np.max(np.abs(per - ref)) <= lim, (p["n"], np.max(np.abs(per - ref)) / lim)
    return per


@pytest.mark.parametrize("nx,ny,precs", [
    (1, 200, "both"), (2, 90, "both"), (3, 60, "both"), (4, 35, "both"), (5, 30, "both"), (7, 19, "both"), (140, 1, "both"),
    (71, 3, "fp64"), (2, 1000, "both"), (16, 512, "both"), (500, 127, "both"), (512, 128, "both"), (1023, 61, "both"),
    (256, 255, "both"), (2047, 31, "fp32"), (400, 320, "fp32"), (512, 254, "fp32")])
@pytest.mark.parametrize("prec", ["fp32", "fp64"])
def test_resident_at_the_edges_of_its_layout(ctx, prec, nx, ny, precs):
    if precs not in (prec, "both"):
        pytest.skip("does not fit in this precision")
    _against(ctx, _line(nx, ny, prec, 200), {"steps_per_launch": 3}, 1)


@pytest.mark.parametrize("prec", ["fp32", "fp64"])
@pytest.mark.parametrize("nx,ny", [(33, 13), (64, 64), (83, 45), (130, 7), (400, 83), (251, 93), (127, 201)])
def test_resident_takes_closed_contours(ctx, prec, nx, ny):
    _against(ctx, _box(nx, ny, prec, 100), {"steps_per_launch": 3}, 1)


@pytest.mark.parametrize("prec,nx,ny", [("fp32", 512, 300), ("fp64", 500, 201), ("fp64", 512, 130)])
def test_larger_grids_take_the_multi_step_kernels(ctx, prec, nx, ny):
    _against(ctx, _box(nx, ny, prec, 100), {"steps_per_launch": 1}, 0)


@pytest.mark.parametrize("prec", ["fp32", "fp64"])
def test_resident_takes_cylinders(ctx, prec):
    _against(ctx, _cylinder(18, 1.0, (0, 2), prec, 256), {"steps_per_launch": 2}, 1)


def test_two_steps_per_launch_against_the_oracle(ctx):
    # the FP64 kernel of grids too large for a cluster: ragged tiles, PMC walls, the point basis, a periodic axis
    k2 = {"steps_per_launch": 2}
    p = W._base(2, (83, 45, 1), 10.0, 500)
    p["objects"] = [{"shape": "box", "lo": [3.0, 1.0, 0], "hi": [4.5, 2.9, 0], "kind": "pec"},
                    {"shape": "box", "lo": [5.5, 0.5, 0], "hi": [6.0, 3.5, 0], "kind": "dielectric", "eps": 3.0, "mu": 1.0}]
    p["faces"] = W.box_faces([2.8, 0.8], [4.8, 3.3], 2)
    p.update(n_harm=5, polarization="TE+TM", force_axis=0, precision="fp64")
    _check(ctx, p, "ragged", True, k2)
    p = W.piston_small(n_steps=400, precision="fp64")
    height = p["n"][1] / p["resolution"]
    p["objects"] = p["objects"] + [{"shape": "box", "lo": [0.0, 0.0, 0.0], "hi": [6.0, 0.05, 0.0], "kind": "pmc"},
                                   {"shape": "box", "lo": [0.0, height - 0.05, 0.0], "hi": [6.0, height, 0.0], "kind": "pmc"}]
    _check(ctx, p, "pmc", True, k2)
    _check(ctx, dict(p, basis="point", n_steps=200), "point", True, k2)
    p = W.piston_small(n_steps=400, precision="fp64")
    p["bc"] = ["periodic", "pec", "pec"]
    _check(ctx, p, "periodic", True, k2)
    for nx, ny in ((7, 40), (40, 1), (3, 2)):
        _check(ctx, _tiny_2d(nx, ny, "TE+TM"), ("tiny2d", nx, ny), True, k2)


def test_plan_teardown_overlapping_graph_capture_of_step_kernels(ctx, pk):
    # runs of the multi-step kernels, which capture graphs (resident runs capture none)
    p = W.piston_small(n_steps=120)
    k = {"steps_per_launch": 2}
    ref = ctx.plan(p, options=k).run()[0]
    prev = ctx.plan(p, options=k)
    prev.run()
    for it in range(12):
        pl = ctx.plan(p, options=k)
        t = pl.submit()
        if it % 2:
            t.cancel()
        prev.close()                            # overlaps the worker's admission and capture
        prev = pl
        try:
            F = t.force(-1)[0]
        except pk.CasimirError as e:
            assert it % 2 and e.code == -6, (it, e)
            continue
        assert F == pytest.approx(ref, rel=1e-9, abs=0)
    prev.close()


def test_resident_runs_in_waves(ctx):
    probs = [_box(83, 45, "fp32", 200), _cylinder(10, 0.5, (0, 1), "fp64", 120)]
    whole = [ctx.plan(p).run(per_sim=True)[1] for p in probs]
    try:
        ctx.set_wave_bytes(100_000)
        for p, w in zip(probs, whole):
            pl = ctx.plan(p)
            assert pl.options()["resident"] == 1
            assert np.array_equal(pl.run(per_sim=True)[1], w)
    finally:
        ctx.set_wave_bytes(0)


def test_resident_run_with_a_callers_allocator(ctx, pk):
    torch = pytest.importorskip("torch")
    p = _box(83, 45, "fp32", 200)
    ref = ctx.plan(p).run(per_sim=True)[1]
    held = {}

    def alloc(n):
        t = torch.empty(n, dtype=torch.uint8, device="cuda")
        held[t.data_ptr()] = t
        return t.data_ptr()
    c = pk.Context(0)
    try:
        c.set_allocator(alloc, lambda a: held.pop(a, None))
        pl = c.plan(p)
        assert pl.options()["resident"] == 1
        assert np.array_equal(pl.run(per_sim=True)[1], ref)
        assert held
    finally:
        c.close()
    assert not held


def test_autotuned_plans_give_the_same_results(ctx, pk):
    probs = [_box(83, 45, "fp32", 200), _cylinder(18, 1.0, (0, 2), "fp32", 256), _box(512, 300, "fp32", 60)]
    c = pk.Context(0)
    try:
        c.set_autotune(True)
        for p in probs:
            per = c.plan(p).run(per_sim=True)[1]
            ref = ctx.plan(p).run(per_sim=True)[1]
            assert np.max(np.abs(per - ref)) <= 16 * 2.0 ** -53 * np.sqrt(p["n_steps"]) * np.max(np.abs(ref))
    finally:
        c.close()
