"""Gradients of the mean drag on one handle whose sphere is released, moved and held again between the calls: those of
a handle that begins at the new place, in FP64 to 1e-12 of the largest entry (the same sums in the same order)."""
import numpy as np
import pytest

from paper_2103_10882_gb300 import workloads
from test_gpu_adjoint import forward, lib, run  # noqa: F401

pytestmark = pytest.mark.gpu
SHAPE, POS, D, TAU, F, STEPS, EVERY = (22, 19, 24), (10.3, 9.6, 11.2), 6.0, 0.7, (1e-5, 0.0, 2e-6), 12, 5
U0 = workloads.fourier_velocity_field(SHAPE, 2, 1e-2, 21)


def held(lib, pos):  # noqa: F811
    s = lib.Simulation(SHAPE, precision="fp64", tau=TAU)
    s.add_sphere(pos, D, 5.0)
    s.set_fixed(True)
    return s


def move(s, steps):
    s.set_fixed(False)
    s.set_particle_velocity((0.05, -0.04, 0.045))
    s.step(steps)
    s.set_particle_velocity((0, 0, 0))
    s.set_fixed(True)
    return s.particle()[6:9].copy()


def gradient(lib, s):  # noqa: F811
    return run(lib, s, TAU, F, U0, STEPS, EVERY)


def assert_same(a, b):
    for x, y in zip(a, b):
        assert np.abs(np.asarray(x) - np.asarray(y)).max() <= 1e-12 * np.abs(np.asarray(y)).max()


@pytest.mark.parametrize("steps", [51, 52])
def test_moved_by_steps(lib, steps):  # noqa: F811
    s = held(lib, POS)
    first = gradient(lib, s)
    pos = move(s, steps)
    assert np.abs(pos - POS).max() > 1.0   # by more than a cell
    again = gradient(lib, s)
    fresh = held(lib, pos)
    assert_same(again, gradient(lib, fresh))
    assert abs(again[0] - first[0]) > 1e-6 * abs(first[0])
    s.step(3)   # held: nothing moves
    assert_same(gradient(lib, s), again)


def test_moved_by_load(lib, tmp_path):  # noqa: F811
    s, other = held(lib, POS), held(lib, (12.7, 8.1, 14.4))
    gradient(lib, s)
    other.save(str(tmp_path / "c"))
    s.load(str(tmp_path / "c"))
    assert_same(gradient(lib, s), gradient(lib, other))


def test_backward_after_the_sphere_moved(lib):  # noqa: F811
    import torch
    s = held(lib, POS)
    forward(lib, s, TAU, F, U0, STEPS, EVERY)
    move(s, 3)
    one = torch.ones((), dtype=torch.float64, device="cuda")
    gt = torch.zeros((), dtype=torch.float64, device="cuda")
    with pytest.raises(lib.LbmpError) as e:
        lib.lbmp_drag_backward(s.h, one.data_ptr(), gt.data_ptr(), 0, 0)
    assert e.value.status == 1


def test_backward_after_the_held_sphere_spun(lib):  # noqa: F811
    """The sphere keeps its place; its velocities, zero at both calls, were others in between."""
    import torch
    s = held(lib, POS)
    want = gradient(lib, s)
    J, _, u = forward(lib, s, TAU, F, U0, STEPS, EVERY)
    s.set_particle_velocity((0.02, 0.0, -0.03), (0.01, -0.02, 0.015))
    s.step(1)
    s.set_particle_velocity((0, 0, 0))
    one = torch.ones((), dtype=torch.float64, device="cuda")
    gt, gf, gu = torch.empty_like(one), torch.empty(3, dtype=torch.float64, device="cuda"), torch.empty_like(u)
    lib.lbmp_drag_backward(s.h, one.data_ptr(), gt.data_ptr(), gf.data_ptr(), gu.data_ptr())
    torch.cuda.synchronize()
    assert_same((J, gt.item(), gf.cpu().numpy(), gu.cpu().numpy()), want)
