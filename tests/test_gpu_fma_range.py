"""FP64 with fused multiply-adds at the ends of the exponent range: a step
does not care for the units of density, pressure and field."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_1705_10774_gb300 import ics
from paper_1705_10774_gb300.dispatch import Dispatch
from oracle import Oracle

GAMMA = 5.0 / 3.0


@pytest.mark.parametrize("kw", [{}, {"eta": 1e-3}], ids=["ideal", "ohmic"])
def test_densities_and_pressures_of_any_size(kw):
    """Density, momentum, energy and pressure times 2^k and the field times
    2^(k/2) is the same flow: the same bits, scaled."""
    lay = ics.cartesian((2, 1, 1), (17, 9, 6))
    X, Y, Z = lay.base_cells
    rng = np.random.default_rng(5)
    shape = (Z, Y, X)
    bx, by, bz = ics.curl_faces(*[0.02 * lay.dx * rng.standard_normal(shape) for _ in range(3)], lay.dx)
    f = ics.Fields(rho=1 + 0.3 * rng.random(shape), v=0.5 * rng.standard_normal((3,) + shape),
                   p=0.6 + 0.2 * rng.random(shape), bx=bx + 0.5, by=by + 0.3, bz=bz - 0.2, gamma=GAMMA)
    state, first = ics.to_patches(lay, f), None
    for k in (0, 520, -520, 900, -900):
        m = [2.0 ** k] + 3 * [2.0 ** (k // 2)]
        g = Dispatch(lay.n, lay.lo, precision=2, gamma=GAMMA, cfl=0.4, base_cells=lay.base_cells, box_len=lay.box_len,
                     time_mode=0, **kw)
        g.set_state(*[a * s for a, s in zip(state, m)])
        g.advance(max_sweeps=2)
        out = [a / s for a, s in zip(g.get_state(), m)] + [g.pack(np.arange(lay.npatch), device=False)[1]]
        g.close()
        first = first or out
        assert all(np.array_equal(a, b) for a, b in zip(out, first)), k


def test_slopes_below_the_normal_range():
    """Momenta of 1e-307 in a uniform gas at rest: the limited slopes are
    rounded like any others (the tolerance of the parity tests)."""
    lay = ics.cartesian((2, 1, 1), (17, 9, 6))
    X, Y, Z = lay.base_cells
    rng = np.random.default_rng(6)
    one = np.ones((Z, Y, X))
    f = ics.Fields(rho=one, v=1e-307 * rng.standard_normal((3, Z, Y, X)), p=0.6 * one, bx=0 * one, by=0 * one, bz=0 * one,
                   gamma=GAMMA)
    state = ics.to_patches(lay, f)
    kw = dict(gamma=GAMMA, cfl=0.4, base_cells=lay.base_cells, box_len=lay.box_len, time_mode=0)
    o = Oracle(lay.n, lay.lo, **kw)
    o.set_state(*state)
    o.advance(max_sweeps=1)
    g = Dispatch(lay.n, lay.lo, precision=2, **kw)
    g.set_state(*state)
    g.advance(max_sweeps=1)
    c = int(np.prod(lay.n[0]))
    a, b = (np.asarray(s.get_state()[0]).reshape(lay.npatch, 5, c)[:, 1:4] for s in (g, o))
    g.close()
    assert np.max(np.abs(b)) < 1e-306 and np.max(np.abs(a - b)) <= 1e-11 * np.max(np.abs(b))
