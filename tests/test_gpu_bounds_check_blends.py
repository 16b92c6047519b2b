"""The bounds-checked build on neighbours blended in time: FP32 values of two
slices are copied side by side and blended once both have arrived, those of
three are loaded one by one.  Every address lies in the slices, and the results
are the regular build's, bit for bit, for ragged tiles, by sweeps and by the
ready queue."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_1705_10774_gb300.dispatch import Dispatch

from test_gpu_tile_edges import _case


@pytest.mark.parametrize("precision", [0, 1, 2])
@pytest.mark.parametrize("order,dispatcher", [(1, 1), (2, 1), (1, 0)])
@pytest.mark.parametrize("n", [(33, 9, 5), (7, 20, 4)])
def test_blended_neighbours_stay_in_bounds(n, order, dispatcher, precision):
    lay, state = _case(n, sum(n), (4, 2, 2))
    u, c = state[0].copy(), int(np.prod(n))
    u[4 * c:5 * c] += 300.0  # a hot patch: steps spread over a factor
    res = []
    for checked in (False, True):
        g = Dispatch(lay.n, lay.lo, precision=precision, time_mode=1, time_order=order, dispatcher=dispatcher, nslices=5,
                     gamma=5.0 / 3.0, cfl=0.3, base_cells=lay.base_cells, box_len=lay.box_len, checked=checked)
        g.set_state(u, *state[1:])
        st = g.advance(t_end=0.05 * lay.dx)
        assert st["status"] == 0 and st["patch_updates"] > lay.npatch
        res.append(list(g.get_state()) + [g.times()[0]])
        g.close()
    assert all(np.array_equal(a, b) for a, b in zip(*res))
