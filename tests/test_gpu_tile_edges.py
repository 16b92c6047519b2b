"""The update kernel at the edges of its tile shapes: patches one cell short
of, equal to and one cell past the tiles' extents, thin ones, and several
tiles with a ragged last one, for every tile shape of every precision.

FP64 without FMA: state, times and signal speeds equal the oracle's bit for
bit.  The other precisions: every tile shape and z run gives the same bits,
within 1e-11 (FP64 with FMA, the tolerance of the parity tests) or 1e-5 (FP32:
some ten roundings of 6e-8 on each of a few dozen terms per step, two steps)
of the oracle's largest value."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_1705_10774_gb300 import build as B
from paper_1705_10774_gb300 import ics
from paper_1705_10774_gb300.dispatch import Dispatch
from oracle import Oracle

SIZES = [(4, 4, 4), (7, 8, 5), (16, 11, 4), (17, 9, 6), (15, 12, 7), (33, 13, 5), (31, 17, 4), (24, 8, 9), (49, 4, 4)]


def _case(n, seed, patches=(2, 2, 2)):
    lay = ics.cartesian(patches, n)
    X, Y, Z = lay.base_cells
    rng = np.random.default_rng(seed)
    shape = (Z, Y, X)
    A = [0.02 * lay.dx * rng.standard_normal(shape) for _ in range(3)]
    bx, by, bz = ics.curl_faces(*A, lay.dx)
    f = ics.Fields(rho=1 + 0.3 * rng.random(shape), v=0.5 * rng.standard_normal((3,) + shape),
                   p=0.6 + 0.2 * rng.random(shape), bx=bx + 0.5, by=by + 0.3, bz=bz - 0.2, gamma=5.0 / 3.0)
    return lay, ics.to_patches(lay, f)


@pytest.mark.parametrize("precision", [0, 1, 2])
@pytest.mark.parametrize("n", SIZES)
def test_every_tile_shape_at_its_edges(n, precision):
    lay, state = _case(n, sum(n))
    kw = dict(gamma=5.0 / 3.0, cfl=0.4, base_cells=lay.base_cells, box_len=lay.box_len, time_mode=0)
    o = Oracle(lay.n, lay.lo, **kw)
    o.set_state(*state)
    o.advance(max_sweeps=2)
    ref, (_, _, speed) = o.get_state(), o.get_times()
    scale = max(float(np.max(np.abs(a))) for a in ref)
    first = None
    ids = [v[0] for v in B.variants() if v[6] == precision and v[7] == 0 and v[8] == 0]
    for vid, tile_z in [(v, 0) for v in ids] + [(-1, 0), (ids[0], 1), (ids[-1], 3)]:
        g = Dispatch(lay.n, lay.lo, precision=precision, variant=vid, tile_z=tile_z, **kw)
        g.set_state(*state)
        g.advance(max_sweeps=2)
        out = g.get_state()
        smax = g.pack(np.arange(lay.npatch), device=False)[1][:, 2].copy()
        g.close()
        if first is None:
            first = out, smax
        for a, b in zip(out, first[0]):
            assert np.array_equal(a, b), (vid, tile_z)
        assert np.array_equal(smax, first[1])
    if precision == 0:
        assert all(np.array_equal(a, b) for a, b in zip(first[0], ref)) and np.array_equal(first[1], speed)
    else:
        tol = 1e-11 if precision == 2 else 1e-5
        assert max(float(np.max(np.abs(a - b))) for a, b in zip(first[0], ref)) <= tol * scale
        assert np.max(np.abs(first[1] - speed)) <= tol * np.max(speed)


@pytest.mark.parametrize("riemann", [0, 1])
@pytest.mark.parametrize("order,grace", [(1, 0.0), (1, 0.4), (2, 0.0)])
@pytest.mark.parametrize("n", [(33, 9, 5), (16, 8, 8), (7, 20, 4)])
def test_fp32_tiles_blend_neighbours_alike(n, order, grace, riemann):
    """FP32 under local steps: the tiles that blend a neighbour's two slices
    after both have arrived give the bits of those that wait for each value
    (the 16 x 8 tiles, and every tile where three slices are blended)."""
    lay, state = _case(n, 3 * sum(n), (4, 2, 2))
    u = state[0].copy()
    off = 0
    for P, (nx, ny, nz) in enumerate(lay.n.astype(int)):  # a hot patch: steps spread over a factor
        c = nx * ny * nz
        u[off + 4 * c:off + 5 * c] += 300.0 if P == 0 else 0.0
        off += 5 * c
    first = None
    for vid in [v[0] for v in B.variants() if v[6] == 1 and v[7] == riemann and v[8] == 0]:
        g = Dispatch(lay.n, lay.lo, precision=1, variant=vid, riemann=riemann, time_mode=1, time_order=order,
                     grace=grace, nslices=5, gamma=5.0 / 3.0, cfl=0.3, base_cells=lay.base_cells, box_len=lay.box_len,
                     sched_capacity=4096)
        g.set_state(*[u] + list(state[1:]))
        g.advance(max_sweeps=12)
        out = list(g.get_state()) + list(g.times()) + list(g.schedule())
        g.close()
        first = first or out
        assert len(np.unique(out[-1])) >= 2  # several step sizes, so times differ
        for a, b in zip(out, first):
            assert np.array_equal(a, b), vid


def _splits(xs, ys, zs):
    """The box cut at every combination of the given extents per axis."""
    lo, n = [], []
    for z in range(len(zs)):
        for y in range(len(ys)):
            for x in range(len(xs)):
                lo.append((sum(xs[:x]), sum(ys[:y]), sum(zs[:z])))
                n.append((xs[x], ys[y], zs[z]))
    return np.array(n), np.array(lo), (sum(xs), sum(ys), sum(zs))


@pytest.mark.parametrize("xs,ys,zs,precision,riemann,nonideal", [
    ((32, 4), (8, 8), (12, 4), 1, 0, 0), ((32, 4), (8, 4), (12, 4), 1, 0, 0), ((32, 4), (8, 4), (12, 4), 1, 1, 0),
    ((16, 4), (12, 4), (12, 4), 2, 0, 0), ((16, 4), (4, 4), (12, 4), 1, 0, 1)])
def test_layouts_whose_wide_tiles_touch_too_many_blocks_keep_the_first_tile(xs, ys, zs, precision, riemann, nonideal):
    """Patches beside thin ones: the map blocks are 4 cells wide, and the wide
    tiles that would be the default touch more of them than a tile's table
    holds; the form's first tile still fits and serves them."""
    n, lo, base = _splits(xs, ys, zs)
    c = np.prod(n, axis=1)
    u = np.concatenate([np.concatenate([np.ones(k), np.zeros(3 * k), np.full(k, 2.0)]) for k in c])
    state = [u, np.full(int(np.sum((n[:, 0] + 1) * n[:, 1] * n[:, 2])), 0.3),
             np.zeros(int(np.sum(n[:, 0] * (n[:, 1] + 1) * n[:, 2]))), np.zeros(int(np.sum(n[:, 0] * n[:, 1] * (n[:, 2] + 1))))]
    g = Dispatch(n, lo, gamma=5.0 / 3.0, cfl=0.4, base_cells=base, box_len=tuple(b / 8.0 for b in base), time_mode=0,
                 precision=precision, riemann=riemann, eta=1e-3 * nonideal, gamma_ad=75.0 * nonideal)
    g.set_state(*state)
    g.advance(max_sweeps=2)
    for a, b in zip(g.get_state(), state):  # a uniform state stays
        assert np.allclose(a, b, rtol=0, atol=1e-6)
    g.close()


@pytest.mark.parametrize("riemann", [0, 1])
@pytest.mark.parametrize("n", [(33, 9, 5), (16, 8, 8), (7, 20, 4)])
def test_fp32_ready_queue_tiles_end_as_the_sweeps_do(n, riemann):
    """FP32 under local steps: every tile of the ready-queue kernel, whose
    copies and blends run beside publishing neighbours, ends in the sweeps' bits."""
    lay, state = _case(n, 3 * sum(n), (4, 2, 2))
    u, c = state[0].copy(), int(np.prod(n))
    u[4 * c:5 * c] += 300.0
    t_end = 0.05 * lay.dx
    first = None
    ids = [v[0] for v in B.variants() if v[6] == 1 and v[7] == riemann and v[8] == 0]
    for dispatcher, vid in [(1, -1)] + [(0, v) for v in ids + [-1]]:
        g = Dispatch(lay.n, lay.lo, precision=1, variant=vid, riemann=riemann, time_mode=1, dispatcher=dispatcher,
                     gamma=5.0 / 3.0, cfl=0.3, base_cells=lay.base_cells, box_len=lay.box_len)
        g.set_state(*[u] + list(state[1:]))
        st = g.advance(t_end=t_end)
        out = list(g.get_state()) + [g.times()[0]]
        g.close()
        assert st["patch_updates"] > lay.npatch
        first = first or out
        for a, b in zip(out, first):
            assert np.array_equal(a, b), (dispatcher, vid)
