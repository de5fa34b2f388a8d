"""Openings whose raster cells take the two exact opening tests -- the cell's
local edges, and all edges by the whole warp (more than 12 edges in a cell) --
against the oracle, history by history in deterministic mode: a concave star,
a small circle of 1,024 edges and a wavy contour of 2,048, with parallel and
divergent walls.  Tolerances are those of the per-history parity; a contour
with many corners has more step starts within 10 um of a wall."""
import numpy as np
import pytest

from paper_2307_01416_gb300 import workloads as W
from tests.test_gpu_parity import _per_history_parity
from tests.test_raster_local import _star, _wavy

pytestmark = pytest.mark.gpu

SHAPES = {"star": _star(24, 14.0, 6.0, 0.3), "small circle": W.regular_polygon(1.5, 1024), "wavy": _wavy(2048, 5)}


@pytest.mark.parametrize("shape", list(SHAPES))
@pytest.mark.parametrize("sad", [0.0, 400.0])
def test_opening_per_history(shape, sad):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    pb, spots = W.water_aperture_case(20.0, True, hist_per_layer=4000, max_layers=2, shape=(40, 40, 80))
    pb.beams[0].polygon = SHAPES[shape]
    pb.beams[0].ap_sad = sad
    _, st, rec, _, _ = _per_history_parity(pb, spots, W.Scenario(), W.Options(seed=77, mcs=False, straggling=False),
                                           max_flagged=0.04)
    assert 0.02 * st["e_in"] < st["e_aperture"] and np.any(rec["fate"] <= 2)
