"""The resident march of 2D TM/TE runs (fields in registers, one cluster per simulation) against the
oracle and against the three-step kernel, at the sizes where its layout can go wrong: grids narrower
than a thread's columns, one or two rows, ragged last columns, bands one row short, several row bands per
CTA and several CTAs per simulation, periodic and PMC walls, dielectric (mixed-material) warps, runs whose
last chunk is short.

The fields are the three-step kernel's bit for bit (the same operations on the same values), so the
contributions differ only by the order of the FP64 sums of T weighted samples: 16 u sqrt(T) of the
largest contribution, the rounding floor the oracle comparison uses."""
import numpy as np
import pytest

import oracle
import workloads as W
from parity_bounds import assert_parity

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    from paper_0906_5170_gb300 import build
    build.build()
    import paper_0906_5170_gb300 as pk
    c = pk.Context(0)
    yield c
    c.close()


def _box(nx, ny, prec, steps, n_harm=2, bc=("pec", "pec", "pec"), pol="TE+TM", objects=None):
    """A cell of nx x ny with a small dielectric block off the grid lines' symmetry and a rectangular
    contour (or a line through a cell one or two rows high)."""
    res = 10.0
    d = 1.0 / res
    p = W._base(2, (nx, ny, 1), res, steps)
    p["bc"] = list(bc)
    if objects is None:
        objects = [{"shape": "box", "lo": [0.3 * nx * d, 0.35 * ny * d, 0], "hi": [0.55 * nx * d, 0.7 * ny * d, 0],
                    "kind": "dielectric", "eps": 3.0, "mu": 1.0}]
    p["objects"] = objects
    i0, i1 = int(0.2 * nx), max(int(0.7 * nx), int(0.2 * nx) + 1)
    if ny >= 6:
        j0, j1 = int(0.2 * ny), int(0.8 * ny)
        p["faces"] = W.box_faces([i0 * d, j0 * d], [i1 * d, j1 * d], 2)
    else:
        p["faces"] = [{"axis": 1, "sign": 1, "pos": 0.5 * ny * d, "lo": [i0 * d, 0.5 * ny * d, 0.0], "hi": [i1 * d, 0.5 * ny * d, 0.0]}]
        p["force_axis"] = 1
    p.update(n_harm=n_harm, polarization=pol, precision=prec)
    return p


def _compare(ctx, p):
    F, per, st = ctx.plan(p).run(per_sim=True)
    assert st["kernel_launches"] > 0
    _, per3, _ = ctx.plan(p, options={"steps_per_launch": 3}).run(per_sim=True)
    lim = 16 * 2.0 ** -53 * np.sqrt(p["n_steps"]) * np.max(np.abs(per3))
    assert np.max(np.abs(per - per3)) <= lim, (p["n"], np.max(np.abs(per - per3)) / lim)
    return F, per


SIZES = [(2, 7), (3, 12), (5, 1), (9, 2), (33, 13), (64, 64), (61, 29), (83, 45), (130, 7), (400, 83), (251, 93), (127, 201), (512, 130), (500, 201)]


@pytest.mark.parametrize("prec", ["fp32", "fp64"])
@pytest.mark.parametrize("nx,ny", SIZES)
def test_resident_equals_three_step_kernel(ctx, prec, nx, ny):
    _compare(ctx, _box(nx, ny, prec, 200))


@pytest.mark.parametrize("prec", ["fp32", "fp64"])
@pytest.mark.parametrize("nx,ny", [(3, 12), (33, 13), (83, 45), (61, 29)])
def test_resident_against_oracle(ctx, prec, nx, ny):
    p = _box(nx, ny, prec, 150)
    F, per = _compare(ctx, p)
    Fo, parts, _ = oracle.force(p, return_parts=True)
    assert_parity(per, F[p["force_axis"]], np.array(parts), Fo, p["n_steps"], prec == "fp64", str((nx, ny)))


@pytest.mark.parametrize("steps", [1, 2, 3, 191, 192, 193, 385])
def test_resident_chunk_boundaries(ctx, steps):
    _compare(ctx, _box(66, 50, "fp32", steps))


@pytest.mark.parametrize("bc", [("periodic", "pec", "pec"), ("pec", "periodic", "pec"), ("periodic", "periodic", "pec")])
def test_resident_periodic(ctx, bc):
    _compare(ctx, _box(83, 45, "fp32", 300, bc=bc))


def test_resident_pmc_and_many_materials(ctx):
    rng = np.random.default_rng(5)
    objs = [{"shape": "box", "lo": [0, 0, 0], "hi": [9.0, 0.05, 0], "kind": "pmc"}]
    for _ in range(40):
        x, y = rng.uniform(0.2, 8.0), rng.uniform(0.2, 4.0)
        objs.append({"shape": "box", "lo": [x, y, 0], "hi": [x + 0.4, y + 0.3, 0], "kind": "dielectric",
                     "eps": float(rng.uniform(1, 9)), "mu": float(rng.uniform(1, 2))})
    _compare(ctx, _box(90, 47, "fp32", 250, objects=objs))
    _compare(ctx, _box(90, 47, "fp64", 250, objects=objs))


def _cylinder(resolution, h, m_list, prec, steps):
    p = W.cylinder_blocks(h, resolution=resolution, m_list=m_list, n_harm=2, precision=prec)
    p["n_steps"] = steps
    return p


@pytest.mark.parametrize("prec", ["fp32", "fp64"])
@pytest.mark.parametrize("resolution,h,m_list,steps", [(10, 0.5, (0, 1), 150), (14, 0.5, (1, 2), 129), (18, 1.0, (0, 2), 256),
                                                        (24, 2.0, (0, 1, 2), 130), (40, 1.0, (1,), 65)])
def test_resident_cylinder_equals_two_step_march(ctx, prec, resolution, h, m_list, steps):
    p = _cylinder(resolution, h, m_list, prec, steps)
    _, per, st = ctx.plan(p).run(per_sim=True)
    _, per2, _ = ctx.plan(p, options={"steps_per_launch": 2}).run(per_sim=True)
    lim = 16 * 2.0 ** -53 * np.sqrt(steps) * np.max(np.abs(per2))
    assert np.max(np.abs(per - per2)) <= lim, np.max(np.abs(per - per2)) / lim


@pytest.mark.parametrize("prec", ["fp32", "fp64"])
def test_resident_cylinder_against_oracle(ctx, prec):
    p = _cylinder(10, 0.5, (0, 1, 2), prec, 120)
    F, per, _ = ctx.plan(p).run(per_sim=True)
    Fo, parts, _ = oracle.force(p, return_parts=True)
    assert_parity(per, F[p["force_axis"]], np.array(parts), Fo, p["n_steps"], prec == "fp64", "cylinder")


def test_resident_results_do_not_depend_on_the_batch(ctx):
    probs = [_box(66, 50, "fp32", 301), _box(83, 45, "fp64", 250), _box(66, 50, "fp32", 500), _box(130, 40, "fp32", 333)]
    alone = [ctx.plan(p).run()[0] for p in probs]
    plans = [ctx.plan(p) for p in probs]
    got = [t.force(-1)[0] for t in [pl.submit(tag=i) for i, pl in enumerate(plans)]]
    for x, y in zip(alone, got):
        assert np.array_equal(x, y)
