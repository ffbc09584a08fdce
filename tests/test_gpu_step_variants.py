"""Variants of the step that are chosen by size and type, against the oracle where others are compared in FP64 alone: the
FP32 step of five CTAs per SM (from 622,593 cells on) with a sphere, a moving wall and a body force, its boundary CTAs of 40 list
entries (from 1,556,225 cells on), the list of large spheres in FP16, and batches of both types.  Tolerances
of test_gpu_uniform.py and test_gpu_batch.py: FP32 1e-5 of max|g| (a batch against single runs 1e-6), FP16 5e-3."""
import numpy as np
import pytest

from test_gpu_uniform import assert_pops_close, lib, make_pair  # noqa: F401

pytestmark = pytest.mark.gpu
P, N = "periodic", "noslip"
TOL = {"fp32": 1e-5, "fp16": 5e-3}


@pytest.mark.parametrize("precision,shape,d,bc,force,steps", [
    ("fp32", (88, 86, 84), 12.0, (P, P, P), 0.0, 10),
    ("fp32", (88, 86, 84), 12.0, (N, P, P), 1e-6, 10),
    ("fp32", (120, 118, 112), 16.0, (P, P, P), 0.0, 6),
    ("fp16", (86, 85, 84), 74.0, (P, P, P), 0.0, 3),
], ids=["five CTAs", "five CTAs, wall and force", "40 entries a CTA", "list"])
def test_large_steps(orc, lib, precision, shape, d, bc, force, steps):  # noqa: F811
    pos = np.array(shape, dtype=float) / 2 + np.array([0.23, -0.31, 0.17])
    o, g = make_pair(orc, lib, shape, precision=precision, tau=0.7, bc=bc, body_force=(force, -2 * force, 0.0),
                     sphere=(pos, d, 0.6, 0.5), gravity=(0, 0, -2e-5),
                     velocity=((0.03, -0.04, 0.05), (0.001, -0.002, 0.0005)))
    if N in bc:
        for s in (o, g):
            s.set_wall_velocity(0, 1, (0.0, 0.02, -0.01))
    o.step(steps)
    g.step(steps)
    assert_pops_close(o, g, TOL[precision])
    np.testing.assert_allclose(g.particle()[6:9], o.particle()[6:9], rtol=0, atol=1e-5)


@pytest.mark.parametrize("precision", ["fp32", "fp16"])
@pytest.mark.parametrize("edges", [(16,), (32,) * 15, (16, 48, 32) * 24], ids=["four CTAs a segment", "two", "two segments"])
def test_batch_types_and_shapes(lib, precision, edges):  # noqa: F811
    """First and last simulation against a run of its own; the shape that the autotuner chooses changes no bit."""
    sims = [dict(edge=e, pos=np.full(3, e / 2) + 0.01 * i * np.array([1, -1, 0.5]), diameter=max(5.0, e / 6), tau=0.7,
                 density_ratio=0.6, cv=0.5, gravity=(0.0, 0.0, -2e-5)) for i, e in enumerate(edges)]
    b, tuned = (lib.BatchSimulation(sims, precision=precision) for _ in range(2))
    tuned.autotune(3)
    b.step(13)
    tuned.step(13)
    for i in sorted({0, len(sims) - 1}):
        s = sims[i]
        assert np.array_equal(b.populations(i), tuned.populations(i))
        assert np.array_equal(b.particle(i), tuned.particle(i))
        g = lib.Simulation((s["edge"],) * 3, precision=precision, tau=s["tau"])
        g.add_sphere(s["pos"], s["diameter"], s["density_ratio"], cv=s["cv"])
        g.set_gravity(s["gravity"])
        g.init_fluid()
        g.step(13)
        a, c = g.populations(), b.populations(i)
        assert np.abs(a - c).max() <= (1e-6 if precision == "fp32" else 5e-3) * np.abs(a).max()
