"""The kernels that pass over whole patches with several blocks on one patch:
loading, reading back, the loaded state's signal speed, diagnostics and
packages, for a single large patch, a few ragged ones and cold cells whose
pressure FP32 cannot resolve."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_1705_10774_gb300 import ics
from paper_1705_10774_gb300.dispatch import Dispatch
from oracle import Oracle


def _state(n, p, seed, cold):
    lay = ics.cartesian(p, n)
    X, Y, Z = lay.base_cells
    rng = np.random.default_rng(seed)
    shape = (Z, Y, X)
    A = [0.1 * lay.dx * rng.standard_normal(shape) for _ in range(3)]
    bx, by, bz = ics.curl_faces(*A, lay.dx)
    pr = np.full(shape, 1e-9) if cold else 0.5 + rng.random(shape)
    f = ics.Fields(rho=np.exp(rng.standard_normal(shape)), v=3 * rng.standard_normal((3,) + shape), p=pr, bx=bx + 0.5,
                   by=by - 0.2, bz=bz + 0.1, gamma=5.0 / 3.0)
    return lay, ics.to_patches(lay, f)


@pytest.mark.parametrize("cold", [False, True])
@pytest.mark.parametrize("n,p", [((61, 47, 33), (1, 1, 1)), ((19, 23, 29), (3, 1, 2)), ((4, 5, 4), (1, 2, 1))])
def test_loaded_state_speeds_and_read_back(n, p, cold):
    lay, state = _state(n, p, 7, cold)
    kw = dict(gamma=5.0 / 3.0, cfl=0.4, base_cells=lay.base_cells, box_len=lay.box_len)
    o = Oracle(lay.n, lay.lo, **kw)
    o.set_state(*state)
    for precision in (0, 2):  # signal speeds: the maximum over cells, bit for bit
        g = Dispatch(lay.n, lay.lo, precision=precision, **kw)
        g.set_state(*state)
        assert np.array_equal(g.pack(np.arange(lay.npatch), device=False)[1][:, 2], o.get_times()[2])
        assert all(np.array_equal(a, b) for a, b in zip(g.get_state(), state))
        dev = [torch.from_numpy(a).cuda() for a in state]
        g.set_state(*dev)
        assert all(np.array_equal(a, b) for a, b in zip(g.get_state(), state))
        f32 = g.get_state(dtype=np.float32)
        assert all(np.array_equal(a, b.astype(np.float32)) for a, b in zip(f32, state))
        d, e = g.diagnostics(), o.diagnostics()
        for k in ("mass", "energy"):
            assert abs(d[k] - e[k]) <= 1e-13 * abs(e[k])
        assert d["max_b"] == e["max_b"] and d["max_divb"] == e["max_divb"]
        g.close()


def test_packages_of_large_patches_round_trip():
    lay, state = _state((45, 38, 27), (2, 2, 2), 3, False)
    owned = np.array([1, 1, 1, 1, 0, 0, 0, 0], np.uint8)
    kw = dict(gamma=5.0 / 3.0, cfl=0.4, base_cells=lay.base_cells, box_len=lay.box_len, time_mode=1)
    a = Dispatch(lay.n, lay.lo, **kw)
    a.set_state(*state)
    b = Dispatch(lay.n, lay.lo, owned=owned, **kw)
    b.set_state(*[np.asarray(x) * 0 + (1 if k == 0 else 0.5) for k, x in enumerate(state)])
    ids = [7, 4, 6]
    for device in (True, False):
        buf, meta = a.pack(ids, device=device)
        b.unpack(ids, buf, meta)
        back, mb = b.pack(ids, device=device)
        host = lambda t: t.cpu().numpy() if device else t
        assert np.array_equal(host(buf), host(back)) and np.array_equal(host(meta), host(mb))
    a.close()
    b.close()
