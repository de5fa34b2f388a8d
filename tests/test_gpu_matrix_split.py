"""The column maxima of an influence matrix are found by several blocks per
column when there are few columns, and its boxes' depths by a warp per ray.
Columns computed one at a time (the most blocks each), all at once, and in a
set large enough for one block each must be the same, bit for bit, also where
the threshold is decided by the column's maximum."""
import numpy as np
import pytest

from paper_2307_01416_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("rel", [0.0, 0.3])
def test_columns_do_not_depend_on_the_set(rel):
    import torch
    from paper_2307_01416_gb300 import vpmc
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    g, hu = W.water_phantom((40, 36, 70), (2.0, 2.5, 2.0), (-40.0, -45.0, 0.0))
    hu = hu.copy()
    hu[20:24, :, :20] = 700                                    # a slab of bone across part of the field
    beam = W.Beam(direction=(0.0, 0.0, 1.0), bev_x=(1.0, 0.0, 0.0), iso=(0.0, 0.0, 60.0), source_to_iso=200.0)
    pb = W.Problem(ct=g, hu=hu, curve=W.HUCurve(), scoring=g, beams=[beam])
    spots = W.make_spots([(0, 60.0 + 15.0 * i, 4.0 * i - 8.0, 3.0 - 2.0 * i, 2.0, 1.0, 300, 1.0) for i in range(5)])
    eng = vpmc.Engine(pb)

    def columns(s):
        m, _ = eng.influence_matrix(s, [W.Scenario()], W.Options(seed=3), rel_threshold=rel)
        r = np.repeat(np.arange(m[0]["shape"][0]), np.diff(m[0]["row_ptr"].cpu().numpy()))
        c, v = m[0]["col"].cpu().numpy(), m[0]["val"].cpu().numpy()
        return [(r[c == i], v[c == i]) for i in range(len(s))]

    together = columns(spots)
    many = columns(np.concatenate([spots, np.repeat(spots[:1], 2500)]))[:len(spots)]
    for i, (rows, vals) in enumerate(together):
        assert len(rows) and np.all(vals >= rel * vals.max() * (1 - 1e-6))
        assert np.array_equal(rows, many[i][0]) and np.array_equal(vals, many[i][1])
    alone = columns(spots[:1])[0]                              # (the stream of a spot is its index: the first only)
    assert np.array_equal(alone[0], together[0][0]) and np.array_equal(alone[1], together[0][1])
    eng.close()
