"""The coupled uniform step at the edges of its launch: boundary cells found from the segments' numbers (boxes of up to
524,288 cells) and from the list (larger ones), boxes that span a periodic axis or exceed a walled one, grids of a few
cells, rows that begin inside a warp.  Tolerances of test_gpu_uniform.py: FP64 1e-10, FP16 5e-3 of max|g|."""
import numpy as np
import pytest

from test_gpu_uniform import assert_links_equal, assert_pops_close, lib, make_pair  # noqa: F401

pytestmark = pytest.mark.gpu
P, N = "periodic", "noslip"


@pytest.mark.parametrize("precision,shape,d,bc,steps", [
    ("fp64", (53, 52, 51), 41.0, (P, P, P), 6),     # 50^3 box cells, 489 segments: a prefix in one pass
    ("fp64", (82, 84, 83), 72.0, (P, P, P), 3),     # 80^3 box cells, 2,000 segments: the largest prefixes
    ("fp64", (85, 86, 84), 74.0, (P, P, P), 3),     # 82^3 box cells: the list
    ("fp64", (9, 9, 9), 5.0, (P, P, P), 40),        # the box spans every axis
    ("fp64", (7, 40, 9), 3.0, (N, P, N), 40),       # the box exceeds two walled axes
    ("fp64", (8, 8, 257), 4.0, (P, N, P), 40),
    ("fp16", (22, 9, 11), 5.0, (P, N, P), 60),      # pairs of several rows in one warp
    ("fp16", (10, 13, 9), 5.0, (N, P, P), 60),
    ("fp16", (56, 57, 54), 46.0, (P, P, P), 6),
])
def test_step_edges(orc, lib, precision, shape, d, bc, steps):  # noqa: F811
    pos = np.array(shape, dtype=float) / 2 + np.array([0.23, -0.31, 0.17])
    u = np.array([0.03, -0.04, 0.05]) * (0.2 if min(shape) < 10 else 1.0)
    o, g = make_pair(orc, lib, shape, precision=precision, tau=0.7, bc=bc, sphere=(pos, d, 0.6, 0.5),
                     gravity=(0, 0, -2e-5), velocity=(u, (0.001, -0.002, 0.0005)))
    o.step(steps)
    g.step(steps)
    assert_pops_close(o, g, 1e-10 if precision == "fp64" else 5e-3)
    if precision == "fp64":
        assert np.array_equal(o.flags(), g.flags())
        assert_links_equal(o, g)


@pytest.mark.parametrize("edges", [
    (16,), (32,) * 15, (32,) * 30, (16, 48, 32) * 24,
], ids=["four CTAs a segment", "two", "one", "two segments a CTA"])
def test_batch_step_splits(lib, edges):  # noqa: F811
    """Boundary CTAs of a batch: a segment of a box shared by several, or several segments each (here with an odd last
    one); first, middle and last simulation against a run of its own (FP64 1e-10)."""
    sims = [dict(edge=e, pos=np.full(3, e / 2) + 0.01 * i * np.array([1, -1, 0.5]), diameter=max(5.0, e / 6), tau=0.7,
                 density_ratio=0.6, cv=0.5, gravity=(0.0, 0.0, -2e-5)) for i, e in enumerate(edges)]
    b = lib.BatchSimulation(sims, precision="fp64")
    b.step(12)
    for i in sorted({0, len(sims) // 2, len(sims) - 1}):
        s = sims[i]
        g = lib.Simulation((s["edge"],) * 3, precision="fp64", tau=s["tau"])
        g.add_sphere(s["pos"], s["diameter"], s["density_ratio"], cv=s["cv"])
        g.set_gravity(s["gravity"])
        g.init_fluid()
        g.step(12)
        a, c = g.populations(), b.populations(i)
        assert np.abs(a - c).max() <= 1e-10 * np.abs(a).max()
        np.testing.assert_allclose(b.particle(i)[6:12], g.particle()[6:12], rtol=1e-10, atol=1e-12)


def test_records_read_back(lib):  # noqa: F811
    """Histories from a ring that has wrapped, whole and in part, and the particle records of a batch of more than one
    copy's 32 before and after further steps: equal to those of runs that read nothing in between."""
    def run(cap, parts):
        g = lib.Simulation((16, 16, 16), precision="fp64", tau=0.7, history_capacity=cap)
        g.add_sphere((8.2, 7.9, 8.1), 5.0, 0.6, cv=0.5)
        g.set_gravity((0, 0, -2e-5))
        g.init_fluid()
        for n in parts:
            g.step(n)
            g.particle()
        return g
    full, ring = run(32, (13,)).history(), run(8, (5, 8))
    assert full.shape == (13, 15) and np.array_equal(ring.history(), full[5:])
    assert np.array_equal(run(13, (13,)).history(), full)
    sims = [dict(edge=16, pos=(8.0, 8.0, 8.0), diameter=5.0, density_ratio=0.3 + 0.01 * i, cv=0.5, tau=0.7,
                 gravity=(0, 0, -2e-5)) for i in range(34)]
    a, b = (lib.BatchSimulation(sims, precision="fp64") for _ in range(2))
    a.step(3)
    first = [a.particle(i) for i in (0, 31, 32, 33)]
    a.step(4)
    b.step(7)
    for i, was in zip((33, 0, 31, 32), (first[3], *first[:3])):
        assert np.array_equal(a.particle(i), b.particle(i)) and not np.array_equal(a.particle(i), was)
        assert np.array_equal(a.history(i), b.history(i)) and a.history(i).shape == (7, 15)


@pytest.mark.parametrize("precision,shape", [("fp64", (10, 9, 11)), ("fp32", (33, 8, 9)), ("fp16", (10, 9, 11)),
                                             ("fp16", (66, 8, 9)), ("fp16", (4, 9, 8)), ("fp16", (9, 8, 11))])
def test_moving_walls_on_every_axis(orc, lib, precision, shape):  # noqa: F811
    """Walls on all axes, those of x and z moving, gravity-free but forced by the walls: faces, edges and corners of
    the domain, in FP16 pairs with lanes that begin a row, end one, or both.  Tolerances of test_gpu_uniform.py."""
    o, g = make_pair(orc, lib, shape, precision=precision, tau=0.7, bc=(N, N, N))
    for axis, side, u in ((0, 0, (0.0, 0.02, -0.01)), (0, 1, (0.0, -0.01, 0.03)), (2, 1, (0.03, 0.01, 0.0))):
        o.set_wall_velocity(axis, side, u)
        g.set_wall_velocity(axis, side, u)
    o.step(40)
    g.step(40)
    assert_pops_close(o, g, {"fp64": 1e-10, "fp32": 1e-5, "fp16": 5e-3}[precision])
