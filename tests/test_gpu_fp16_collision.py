"""FP16 storage, even rows: the collision of two cells at once relaxes every population by s+ and s- times its distance
from the equilibrium, in FP32 on the stored values, bit for bit as written below.  (Coefficients (1 - s+)/2 and
(1 - s-)/2, rounded, scale the momentum that a collision keeps by up to 1 + 6e-8 in every step, four times what is left
here; in a single step FP16 rounding hides it.)
"""
import numpy as np
import pytest

from lattice_ref import C
from test_gpu_uniform import lib  # noqa: F401

pytestmark = pytest.mark.gpu
F, LD = np.float32, np.longdouble


def fma(a, b, c):
    """a b + c in FP32 with one rounding (the product of two FP32 numbers is exact in the wider type)."""
    return (LD(a) * LD(b) + LD(c)).astype(F)


def collide(g, sp, sm, db, q2):
    """TRT, or MRT with db = s_b - s+, of the stored values g[19, ...] (FP32), written with FP32 operations."""
    w = [F(1) / F(3)] + [F(1) / F(18)] * 6 + [F(1) / F(36)] * 12
    ps = [g[q] + g[q + 1] for q in range(1, 19, 2)]
    pd = [g[q] - g[q + 1] for q in range(1, 19, 2)]
    drho = g[0]
    for p in ps:
        drho = drho + p
    u = []
    for a in range(3):
        t = F(0)
        for k, d in enumerate(pd):
            c = C[2 * k + 1][a]
            t = t + d if c == 1 else (t - d if c == -1 else t)
        u.append(t)
    uu = fma(u[2], u[2], fma(u[1], u[1], u[0] * u[0])) * q2
    n0 = fma(-w[0], fma(F(-1.5), uu, drho), g[0])
    out = [fma(-sp, n0, g[0])]
    n = {0: n0, 1: F(0), 2: F(0)}   # sums of f - f_eq over rest, faces and edges
    for k in range(9):
        q = 2 * k + 1
        cu = F(0)
        for a in range(3):
            cu = cu + u[a] if C[q][a] == 1 else (cu - u[a] if C[q][a] == -1 else cu)
        ep = w[q] * fma(F(-1.5), uu, fma((F(4.5) * q2) * cu, cu, drho))
        em = w[q] * (F(3) * cu)
        np_, nm = F(0.5) * ps[k] - ep, F(0.5) * pd[k] - em
        n[1 if q < 7 else 2] = n[1 if q < 7 else 2] + F(2) * np_
        for at, sign in ((q, -1), (q + 1, 1)):
            out.append(fma(F(sign) * sm, nm, fma(-sp, np_, g[at])))
    if db != 0:
        d4 = n[2] - n[0]
        c16 = F(0.5) * (fma(F(-2), n[1], n[0]) + n[2])
        r, e = fma(F(-1.5), d4, c16), fma(F(1.5), d4, c16)
        out[0] = fma(-(db * w[0]), r, out[0])
        for q in range(1, 19):
            out[q] = fma(F(2) * (db * w[q]), c16, out[q]) if q < 7 else fma(-(db * w[q]), e, out[q])
    return np.stack(out)


@pytest.mark.parametrize("bulk", [1.0, 100.0])
@pytest.mark.parametrize("tau", [0.506, 0.9, 2.5])
def test_pairs_relax_the_distance_from_equilibrium(lib, tau, bulk):  # noqa: F811
    shape, scale = (34, 16, 15), 11
    n3 = tuple(reversed(shape))
    g = np.random.default_rng(5).normal(scale=2.0, size=(19,) + n3).astype(np.float16)   # stored: 2^11 times 1e-3
    s = lib.Simulation(shape, precision="fp16", tau=tau, bulk=bulk, fp16_scale_log2=scale)
    s.set_populations(g.astype(np.float64).reshape(19, -1) * 2.0 ** -scale)
    s.step(1)
    got = s.populations().reshape((19,) + n3) * 2.0 ** scale
    pulled = np.stack([np.roll(g[q], (C[q][2], C[q][1], C[q][0]), axis=(0, 1, 2)) for q in range(19)]).astype(F)
    sp, sm = 1.0 / tau, 1.0 / (0.5 + (3.0 / 16.0) / (tau - 0.5))
    db = 0.0 if bulk == 1.0 else 1.0 / (0.5 + bulk * (tau - 0.5)) - sp
    want = collide(pulled, F(sp), F(sm), F(db), F(2.0 ** -scale)).astype(np.float16)
    assert np.array_equal(got, want.astype(np.float64))
