"""Calls with fewer histories than the persistent blocks have lanes: the launch
leaves out warps that the work cannot fill.  At the edges of that rule (one
history, one warp more, one chunk per SM, one more than the smallest block
takes) the dose must be the one of any other block shape, bit for bit, and the
energy must be conserved; an empty voxel's dose is zero."""
import numpy as np
import pytest

from paper_2307_01416_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("per_sm", [0, 32, 128, 129, 1000], ids=lambda n: f"{n} per SM")
@pytest.mark.parametrize("extra", [1, 33])
def test_small_calls_do_not_depend_on_the_launch(per_sm, extra):
    import torch
    from paper_2307_01416_gb300 import vpmc
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    n = per_sm * torch.cuda.get_device_properties(0).multi_processor_count + extra
    pb, spots = W.water_aperture_case(20.0, True, max_layers=2, shape=(40, 40, 80))
    spots["n_hist"] = W.split_histories(n, len(spots))
    eng = vpmc.Engine(pb)
    ref = None
    for block, chunk in ((0, 0), (32, 32), (896, 7)):
        dose, st, _ = eng.run_spots(spots, opts=W.Options(seed=7), block_size=block, chunk=chunk)
        d = dose.cpu().numpy()
        assert st["errors"] == 0 and np.isfinite(d).all()
        out = sum(st[k] for k in ("e_dep", "e_leak", "e_rs", "e_aperture"))
        assert abs(out / st["e_in"] - 1.0) < 1e-6
        if ref is None:
            ref = (d, st["steps"], st["steps_rs"], st["steps_aperture"])
        assert np.array_equal(d, ref[0])
        assert (st["steps"], st["steps_rs"], st["steps_aperture"]) == ref[1:]
    eng.close()
