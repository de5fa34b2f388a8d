"""Doses of spots with weights.  A lane sums its history's weighted deposits
over the steps of a voxel visit and adds them once, so no step's weight may be
lost or taken from another spot.  The columns of the spots are taken one by one
from the unit-weight path (a dose call each: the generator's streams depend on
the spot's number, so the other spots keep their place with no histories).
With weights that are powers of two the FP32 product with the scale is exact,
and a step's deposit differs from the weighted column's by its rounding alone:
half a unit for each of at most n steps, and half a unit times the weight in
the column.  Spots of 33 histories share warps."""
import numpy as np
import pytest

from paper_2307_01416_gb300 import workloads as W

pytestmark = pytest.mark.gpu

UNIT_GY = 2.0 ** -24 * 1.602176634e-10          # one unit of a deposit over 1 kg


@pytest.mark.parametrize("aggregate", [0, 1])
@pytest.mark.parametrize("weights", [(0.5, 2.0, 1.0), (0.25, 0.0, 8.0)], ids=str)
@pytest.mark.parametrize("n_hist", [33, 500])
def test_weighted_dose_is_the_sum_of_the_weighted_columns(aggregate, weights, n_hist):
    import torch
    from paper_2307_01416_gb300 import vpmc
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    pb, _ = W.pencil_beam_water(1, shape=(20, 20, 60))
    rows = [(0, e, x, -2.0, 2.0, 2.0, n_hist, 1.0) for e, x in ((100.0, 1.0), (90.0, 2.0), (110.0, -4.0))]
    eng = vpmc.Engine(pb)

    def dose(sp, **kw):
        d, st, _ = eng.run_spots(W.make_spots(sp), opts=W.Options(seed=3), block_size=128, **kw)
        return d.cpu().numpy().astype(np.float64), st["steps"]

    want, steps = 0.0, 0
    for j, w in enumerate(weights):
        column, n = dose([r if i == j else r[:6] + (0, 1.0) for i, r in enumerate(rows)])
        want, steps = want + w * column, steps + n
    got, n = dose([r[:7] + (w,) for r, w in zip(rows, weights)], aggregate=aggregate)
    assert n == steps and got.max() > 0.0
    voxel_kg = 8.0e-6                               # 2 mm cubes of water
    unit = UNIT_GY / voxel_kg * (0.5 + 0.5 * max(weights))
    # (a voxel's steps are at most all of them; the doses are FP32)
    assert np.max(np.abs(got - want) - 4 * 2.0 ** -24 * want) <= unit * steps
    eng.close()
