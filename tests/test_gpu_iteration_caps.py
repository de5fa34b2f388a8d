"""Iteration caps on both sides of the one up to which a history's deposits are
summed in 32 bits (2^19), and the longest.  No history here comes near a cap, so
dose, records and influence matrix must not depend on it, bit for bit."""
import numpy as np
import pytest

from paper_2307_01416_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("cap", [1 << 19, (1 << 19) + 1, 2 ** 31 - 1])
def test_results_do_not_depend_on_the_cap(cap):
    import torch
    from paper_2307_01416_gb300 import vpmc
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    pb, _ = W.pencil_beam_water(1, shape=(20, 20, 180))
    spots = W.make_spots([(0, 250.0, 1.0, -2.0, 3.0, 2.0, 3000, 1.0), (0, 71.3, 3.0, 2.0, 3.0, 2.0, 1000, 1.0)])
    eng = vpmc.Engine(pb)
    (dose, st, rec), (ref, st_ref, rec_ref) = (eng.run_spots(spots, opts=W.Options(seed=5), records=4000, timeout_iters=c)
                                               for c in (cap, 0))
    assert np.array_equal(dose.cpu().numpy(), ref.cpu().numpy()) and st["steps"] == st_ref["steps"]
    assert np.array_equal(rec, rec_ref) and rec["e_dep"].max() > 200.0
    (a, _), (b, _) = (eng.influence_matrix(spots, [W.Scenario()], W.Options(seed=5), timeout_iters=c) for c in (cap, 0))
    for k in ("row_ptr", "col", "val"):
        assert torch.equal(a[0][k], b[0][k])
    eng.close()
