"""The objective's block sums.  Every 32 rows hold one term of 1 and 31 terms
of a quarter of an FP32 half-ulp of it: added one by one in FP32 they vanish,
3.8 units in the last place of the block's sum.  The products, the terms and
the class weights are exact in FP32, so the reported value may be off by the
block sums' one rounding and its own: 2 x 2^-24."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_rows", [32, 128, 4096])
def test_small_terms_of_a_block_are_not_lost(n_rows):
    import torch
    from paper_2307_01416_gb300 import vpmc
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    u = np.full(n_rows, 2.0 ** -13 - 2.0 ** -20)     # underdose of a row; its term is u^2
    u[::32] = 1.0
    val = (2.0 - u).astype(np.float32)
    assert np.array_equal(val.astype(np.float64), 2.0 - u)
    m = {"row_ptr": torch.arange(n_rows + 1, dtype=torch.int64, device="cuda"),
         "col": torch.zeros(n_rows, dtype=torch.int32, device="cuda"), "val": torch.from_numpy(val).cuda(),
         "shape": (n_rows, 1)}
    cls = torch.ones(n_rows, dtype=torch.uint8, device="cuda")
    h, _, _ = vpmc.robust_optimize([m], cls, torch.ones(1, device="cuda"), 2.0, iterations=1)
    want = np.sum(u * u) / n_rows
    assert abs(float(h[0]) - want) <= 2.0 ** -23 * want
