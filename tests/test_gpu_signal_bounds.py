"""The signal speeds of FP64 states, of which only the largest counts: each
cell's is bounded in FP32 and evaluated in FP64 where it may be the largest.
Patches of two kinds of cell, a hot gas at rest and a dense stream whose
speeds differ by a part in 1e5 to a fifth, in units and at ratios of specific
heats where FP32 is short of range or of digits: the speeds are the oracle's,
bit for bit."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_1705_10774_gb300 import ics
from paper_1705_10774_gb300.dispatch import Dispatch
from oracle import Oracle

DELTAS = [s * d for d in (1e-5, 3e-5, 1e-4, 3e-4, 1e-3, 3e-3, 1e-2, 3e-2, 0.1, 0.2) for s in (1, -1)]


def _sum(gamma, rho, p, b, v):
    a2, b2 = gamma * p / rho, [x * x / rho for x in b]
    s = a2 + sum(b2)
    return sum(map(abs, v)) + sum(np.sqrt(0.5 * (s + np.sqrt((a2 + sum(b2) - 2 * x) ** 2 + 4 * x * (sum(b2) - x)))) for x in b2)


def _two_kinds(gamma, scale, b):
    """A patch per entry of DELTAS: rows of alternating cells, the stream's
    speed 1 + delta times the hot gas's.  Pressure and field are uniform."""
    lay = ics.cartesian((len(DELTAS), 1, 1), (32, 4, 4))
    X, Y, Z = lay.base_cells
    stream = np.broadcast_to(np.arange(X) % 2 == 1, (Z, Y, X))
    hot, cold = _sum(gamma, 1.0, 1.0, b, (0,)), _sum(gamma, 100.0, 1.0, b, (0,))
    v = np.zeros((3, Z, Y, X))
    v[1] = np.where(stream, (1 + np.repeat(DELTAS, 32)) * hot - cold, 0.0) * scale
    one = np.ones((Z, Y, X))
    f = ics.Fields(rho=np.where(stream, 100.0, 1.0), v=v, p=one * scale ** 2, bx=one * b[0] * scale,
                   by=one * b[1] * scale, bz=one * b[2] * scale, gamma=gamma)
    return lay, ics.to_patches(lay, f)


def _same_speeds(lay, state, gamma, **kw):
    kw.update(gamma=gamma, cfl=0.2, base_cells=lay.base_cells, box_len=lay.box_len, time_mode=0)
    o = Oracle(lay.n, lay.lo, **kw)
    o.set_state(*state)
    loaded = o.get_times()[2].copy()
    o.advance(max_sweeps=2)
    for precision in (0, 2):
        g = Dispatch(lay.n, lay.lo, precision=precision, **kw)
        g.set_state(*state)
        assert np.array_equal(g.pack(np.arange(lay.npatch), device=False)[1][:, 2], loaded)
        g.advance(max_sweeps=2)
        speed, ref = g.pack(np.arange(lay.npatch), device=False)[1][:, 2], o.get_times()[2]
        if precision == 0:
            assert np.array_equal(speed, ref)
            assert all(np.array_equal(a, b) for a, b in zip(g.get_state(), o.get_state()))
        else:  # the tolerance of the parity tests; cancellation in p at most p / E of the digits
            assert np.max(np.abs(speed / ref - 1)) <= 1e-11 / (gamma - 1)
        g.close()


@pytest.mark.parametrize("gamma", [1.0001, 1.00001, 1.000001])
def test_nearly_isothermal_gas(gamma):
    """gamma - 1 taken from gamma in FP32 is off by up to a twentieth."""
    lay, state = _two_kinds(gamma, 1.0, (0.0, 0.0, 0.0))
    _same_speeds(lay, state, gamma)


@pytest.mark.parametrize("b", [0.0, 0.8])
@pytest.mark.parametrize("scale", [1e-9, 1e9, 4e9, 1e10, 1e12, 1e15])
def test_units_of_large_and_small_velocities(scale, b):
    """The fourth power of a speed leaves FP32's range at 4e9: a magnetised
    gas's speed came out up to 28 % low, and finite."""
    lay, state = _two_kinds(5.0 / 3.0, scale, (b, b, b))
    _same_speeds(lay, state, 5.0 / 3.0)
