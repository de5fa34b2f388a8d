"""Protons that move exactly along an axis (no divergence, no scattering): a
direction component is zero, and the distance to that axis' faces is infinite
-- or undefined on a face itself.  Spots without width on voxel faces, edges
and centres, along +z and -x, against the oracle history by history, with one
grid and with a finer CT under the scoring grid; in full physics the same spots
must conserve energy."""
import numpy as np
import pytest

from paper_2307_01416_gb300 import workloads as W
from tests.test_gpu_parity import _per_history_parity

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("fine", [False, True], ids=["one grid", "finer CT"])
@pytest.mark.parametrize("along", ["+z", "-x"])
def test_axis_parallel_protons(fine, along):
    import torch
    from paper_2307_01416_gb300 import vpmc
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    g, hu = W.water_phantom((40, 40, 60), (2.0, 2.0, 2.0), (-40.0, -40.0, 0.0))
    ct, hu_ct = (W.water_phantom((80, 80, 80), (1.0, 1.0, 1.5), g.origin) if fine else (g, hu))
    if along == "+z":
        beam = W.Beam(direction=(0.0, 0.0, 1.0), bev_x=(1.0, 0.0, 0.0), iso=(0.0, 0.0, 0.0), source_to_iso=10.0)
    else:
        beam = W.Beam(direction=(-1.0, 0.0, 0.0), bev_x=(0.0, 1.0, 0.0), iso=(0.0, 0.0, 60.0), source_to_iso=50.0)
    pb = W.Problem(ct=ct, hu=hu_ct, curve=W.HUCurve(), scoring=g, beams=[beam])
    spots = W.make_spots([(0, e, x, y, 0.0, 0.0, 40, 1.0) for e in (60.0, 95.0) for x in (0.0, 1.0, -6.0, 0.5)
                          for y in (0.0, 3.0, -2.0)])
    _per_history_parity(pb, spots, W.Scenario(), W.Options(seed=21, mcs=False, straggling=False), max_flagged=0.05)
    eng = vpmc.Engine(pb)
    _, st, _ = eng.run_spots(spots, opts=W.Options(seed=22))
    assert st["errors"] == 0 and abs((st["e_dep"] + st["e_leak"]) / st["e_in"] - 1.0) < 1e-6
    eng.close()
