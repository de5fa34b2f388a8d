"""Scoring by voxel visits: a lane sums its history's deposits while the
history stays in one voxel.  The sums are integers, so the dose must not
depend on which scoring path took them: the unit-weight path (32-bit totals),
the run-time path (64-bit totals: a zero-weight spot switches the unit path
off) and the warp-aggregated one.  Checked bit for bit where the paths can
differ: one lane, a warp and one more, the three grid nestings, and histories
that the iteration cap stops inside a voxel."""
import numpy as np
import pytest

from paper_2307_01416_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def _problem(grids):
    pb, _ = W.pencil_beam_water(1, shape=(20, 20, 60))
    if grids == "nested xy":                    # 1 x 1 x 1.5 mm CT under a 2 mm grid
        pb.ct = W.Grid((40, 40, 80), (1.0, 1.0, 1.5), pb.scoring.origin)
        pb.hu = np.zeros((80, 40, 40), dtype=np.int16)
    elif grids == "not nested":                 # 4 mm CT columns under 2 mm voxels
        pb.ct = W.Grid((10, 10, 60), (4.0, 4.0, 2.0), pb.scoring.origin)
        pb.hu = np.zeros((60, 10, 10), dtype=np.int16)
    return pb


@pytest.mark.parametrize("grids", ["one grid", "nested xy", "not nested"])
@pytest.mark.parametrize("n_hist", [1, 33, 2000])
@pytest.mark.parametrize("cap", [0, 61])
def test_scoring_paths_agree(grids, n_hist, cap):
    import torch
    from paper_2307_01416_gb300 import vpmc
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    eng = vpmc.Engine(_problem(grids))
    spot = (0, 100.0, 1.0, -2.0, 3.0, 2.0, n_hist, 1.0)
    unit = W.make_spots([spot])
    general = W.make_spots([spot, spot[:6] + (7, 0.0)])
    doses = []
    for spots, agg in ((unit, 0), (unit, 1), (general, 0)):
        d = torch.full((60, 20, 20), -1.0, dtype=torch.float32, device="cuda")
        try:
            eng.run_spots(spots, opts=W.Options(seed=3), dose_out=d, aggregate=agg, block_size=128, chunk=32,
                          timeout_iters=cap)
            assert cap == 0
        except vpmc.VpmcError as e:             # every history meets a cap of 61 iterations
            assert cap and e.status == -4
        doses.append(d.cpu().numpy())
    assert doses[0].sum() > 0.0 and np.array_equal(doses[0], doses[1]) and np.array_equal(doses[0], doses[2])
    eng.close()
