"""An id of the update kernel's variants means the same tile for good."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_1705_10774_gb300 import dispatch as D

from test_gpu_tile_edges import _splits


def _context(variant, precision):
    # thin patches beside wide ones: a tile of 16 x 8 touches 120 blocks of the
    # patch map, one of 16 x 12 150, more than a tile's table holds
    n, lo, base = _splits((16, 4), (12, 4), (12, 4))
    return D.Dispatch(n, lo, gamma=5.0 / 3.0, cfl=0.4, base_cells=base, box_len=tuple(b / 20.0 for b in base), time_mode=0,
                      precision=precision, variant=variant), n


@pytest.mark.parametrize("variant,precision", [(0, 0), (1, 0), (2, 2), (3, 2), (4, 2)])
def test_ids_of_16x8_tiles_take_the_layouts_those_tiles_fit(variant, precision):
    """Without a GPU the layout is accepted and the allocation fails."""
    try:
        _context(variant, precision)[0].close()
    except D.DispatchError as e:
        assert e.code in (D.DSP_ERR_OOM, D.DSP_ERR_CUDA)


@pytest.mark.parametrize("variant,precision", [(1, 2), (3, 0), (4, 1), (26, 0), (99, 2)])
def test_ids_of_other_forms_are_refused(variant, precision):
    with pytest.raises(D.DispatchError) as e:
        _context(variant, precision)
    assert e.value.code == D.DSP_ERR_INVALID_ARG


@pytest.mark.gpu
@pytest.mark.parametrize("variant,same,precision", [(1, 0, 0), (3, 2, 2), (4, 2, 2)])
def test_a_requested_id_runs_and_is_reported(variant, same, precision):
    outs = []
    for v in (variant, same):
        g, n = _context(v, precision)
        rng = np.random.default_rng(1)
        c = np.prod(n, axis=1)
        u = np.concatenate([np.concatenate([1 + 0.1 * rng.random(k), 0.1 * rng.standard_normal(3 * k), 2 + 0.1 * rng.random(k)])
                            for k in c])
        g.set_state(u, np.full(int(np.sum((n[:, 0] + 1) * n[:, 1] * n[:, 2])), 0.3),
                    np.zeros(int(np.sum(n[:, 0] * (n[:, 1] + 1) * n[:, 2]))),
                    np.zeros(int(np.sum(n[:, 0] * n[:, 1] * (n[:, 2] + 1)))))
        assert {t["variant"] for t in g.tuning()} == {v}
        g.advance(max_sweeps=2)
        outs.append(g.get_state())
        g.close()
    assert all(np.array_equal(a, b) for a, b in zip(*outs))
