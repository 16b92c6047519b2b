"""FP32: the signal speed published with a slice is that of the slice's own
cells.  The update reads each new cell back from shared memory for its speed
and then copies the old values of the next plane over it; the planes of these
states differ so much along z that a value of the next plane would show."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_1705_10774_gb300 import build as B
from paper_1705_10774_gb300 import ics
from paper_1705_10774_gb300.dispatch import Dispatch

GAMMA = 5.0 / 3.0


def _speed(u, nx, ny, nz):
    """Largest sum of |v| + c over the cells of one patch (field energy and
    field speeds left out: below 1e-9 of the pressure's here)."""
    rho, m, E = u[0], u[1:4], u[4]
    v = m / rho
    p = (GAMMA - 1) * (E - 0.5 * rho * (v ** 2).sum(0))
    return float((np.abs(v).sum(0) + 3 * np.sqrt(GAMMA * p / rho)).max())


# the speeds' relative error: p by subtraction from E of 1.5 to 3 p, a few dozen
# roundings of 6e-8 in all
@pytest.mark.parametrize("riemann", [0, 1])
@pytest.mark.parametrize("n", [(32, 8, 9), (17, 9, 12), (24, 16, 5)])
def test_the_published_speed_is_of_the_published_cells(n, riemann):
    lay = ics.cartesian((2, 2, 1), n)
    X, Y, Z = lay.base_cells
    rng = np.random.default_rng(sum(n))
    hot = (np.arange(Z) % 2 == 1)[:, None, None] & np.ones((Z, Y, X), bool)  # every other plane, rho down to 1/16
    rho = np.where(hot, 1.0 / 16, 1.0) * (1 + 0.1 * rng.random((Z, Y, X)))
    f = ics.Fields(rho=rho, v=0.1 * rng.standard_normal((3, Z, Y, X)), p=1 + 0.1 * rng.random((Z, Y, X)),
                   bx=np.full((Z, Y, X), 1e-5), by=np.zeros((Z, Y, X)), bz=np.zeros((Z, Y, X)), gamma=GAMMA)
    state = ics.to_patches(lay, f)
    for vid in [v[0] for v in B.variants() if v[6] == 1 and v[7] == riemann and v[8] == 0] + [-1]:
        g = Dispatch(lay.n, lay.lo, precision=1, riemann=riemann, variant=vid, gamma=GAMMA, cfl=0.3, time_mode=0,
                     base_cells=lay.base_cells, box_len=lay.box_len)
        g.set_state(*state)
        for _ in range(3):
            g.advance(max_sweeps=1)
            speed = g.pack(np.arange(lay.npatch), device=False)[1][:, 2]
            u = np.asarray(g.get_state()[0], np.float64)
            c = int(np.prod(n))
            for P in range(lay.npatch):
                want = _speed(u[5 * c * P:5 * c * (P + 1)].reshape(5, -1), *n)
                assert abs(speed[P] - want) <= 1e-5 * want, (vid, P)
        g.close()
