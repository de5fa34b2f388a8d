"""Small pieces of work (opts.chunk) in the beam line: a warp of the source
kernel fills its lanes from as many pieces as it needs, so a piece of 4
histories costs the fetch (8 atomics a warp beside some 45 slab steps of 32
lanes), not seven eighths of the lanes.  The beam line may take 1.8 times what
it takes with whole warps; lanes left empty take 2.7 times.  The dose does not
depend on the piece."""
import numpy as np
import pytest

from paper_2307_01416_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("chunk", [4, 7, 33])
def test_small_pieces_fill_the_warps(chunk):
    import torch
    from paper_2307_01416_gb300 import vpmc
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    pb, spots = W.water_aperture_case(20.0, True, 500_000, max_layers=4)
    eng = vpmc.Engine(pb)
    runs = {c: [eng.run_spots(spots, opts=W.Options(seed=9), chunk=c)[:2] for _ in range(4)] for c in (32, chunk)}
    ms = {c: min(st["ms_devices"] for _, st in r) for c, r in runs.items()}
    (dose, st), (ref, st_ref) = runs[chunk][-1], runs[32][-1]
    eng.close()
    assert np.array_equal(dose.cpu().numpy(), ref.cpu().numpy())
    for k in ("steps", "steps_rs", "steps_aperture", "errors", "e_rs", "e_aperture"):
        assert st[k] == st_ref[k]
    assert ms[chunk] <= 1.8 * ms[32], ms
