"""Gradients on a box of three different odd extents (the last CTA of the plain cells is not full), and around a sphere
with more cells next to it than the reverse step has warps for them (4,864).  Against the tangent oracle: FP64 1e-9,
FP32 1e-4, as in test_gpu_adjoint.py."""
import numpy as np
import pytest

from lattice_ref import C
from paper_2103_10882_gb300 import workloads
from test_gpu_adjoint import lib, make_sim, run  # noqa: F401

pytestmark = pytest.mark.gpu


def near_cells(flags, shape):
    solid = flags.reshape(tuple(reversed(shape))) != 0
    m = np.zeros_like(solid)
    for c in C[1:]:
        for k in (1, -1, 2):
            m |= np.roll(solid, tuple(-k * c[::-1]), (0, 1, 2))
    return int((m & ~solid).sum())


@pytest.mark.parametrize("precision,shape,d,steps,every", [
    ("fp64", (19, 23, 17), 6.0, 20, 6), ("fp32", (19, 23, 17), 6.0, 20, 6),
    ("fp64", (60, 62, 58), 24.0, 6, 4), ("fp32", (60, 62, 58), 24.0, 6, 4)])
def test_ragged_box_and_large_sphere(orc, lib, precision, shape, d, steps, every):  # noqa: F811
    pos = tuple(0.5 * n + o for n, o in zip(shape, (0.31, -0.22, 0.17)))
    tau, F, rel = 0.7, (1e-5, -3e-6, 2e-6), 1e-9 if precision == "fp64" else 1e-4
    u0 = workloads.fourier_velocity_field(shape, 2, 1e-2, 21)
    du = workloads.fourier_velocity_field(shape, 3, 1.0, 22)
    sim = make_sim(lib, shape, pos, d, tau, precision)
    J, gt, gf, gu = run(lib, sim, tau, F, u0, steps, every, axis=1)
    assert d < 24 or near_cells(sim.flags(), shape) > 4864
    args = (shape, tau, pos, d, steps)
    Jo, dtau, _ = orc.drag_tangent(*args, u0=u0, body_force=F, dtau=1.0, axis=1)
    assert J == pytest.approx(Jo, rel=max(rel, 1e-10))
    assert gt == pytest.approx(dtau, rel=rel)
    for a in range(3):
        _, dF, _ = orc.drag_tangent(*args, u0=u0, body_force=F, dforce=np.eye(3)[a], axis=1)
        assert gf[a] == pytest.approx(dF, rel=rel, abs=rel * abs(gf).max())
    _, dU, _ = orc.drag_tangent(*args, u0=u0, body_force=F, du0=du, axis=1)
    assert float((gu * du).sum()) == pytest.approx(dU, rel=rel)
