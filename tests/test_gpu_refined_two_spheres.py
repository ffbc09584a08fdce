"""Two refined handles of one precision in a process: the second, smaller sphere takes nothing from the first's launches
(its boundary kernel keeps a prefix of 2,000 segments in dynamic shared memory, 8 KB)."""
import numpy as np
import pytest

from test_gpu_uniform import lib  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", ["fp32", "fp64"])
def test_small_sphere_added_after_a_large_one(lib, precision):  # noqa: F811
    def large():
        s = lib.Simulation((48, 48, 48), levels=2, precision=precision, tau=0.7)
        s.add_sphere((48.3, 47.8, 48.1), 72.0, 0.5, cv=0.5)
        s.set_gravity((0, 0, -1e-6))
        s.init_fluid()
        return s

    def go(s):
        s.step(2)
        s.regrid()
        s.step(3)
        return s.history()
    alone, first = large(), large()
    want = go(alone)
    second = lib.Simulation((32, 32, 32), levels=2, precision=precision, tau=0.7)
    second.add_sphere((32.2, 31.9, 32.4), 8.0, 0.5, cv=0.5)
    assert np.array_equal(go(first), want)
    second.step(2)
