"""Full-matrix products with more rows than the launch's warps take at once:
one row less, as many and one more, so that the first warp comes round again
and the last one stays idle.  Tolerance: an FP32 sum of n products, 2e-6 of the
largest, as for the other row lengths."""
import numpy as np
import pytest

from tests.test_gpu_row_kernels import _dev, _matrix

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("extra", [-1, 0, 1, 6])
def test_rows_beyond_one_pass(extra):
    import torch
    from paper_2307_01416_gb300 import vpmc
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    warps = torch.cuda.get_device_properties(0).multi_processor_count * 16 * 8 - 1
    n_rows = 4 * warps + extra
    m, A = _matrix(n_rows, 70, [0, 0, 1, 8, 9, 65], 3 + extra)
    x = np.random.default_rng(5).uniform(0.0, 2.0, 70).astype(np.float32)
    d = A @ x.astype(np.float64)
    xd = torch.from_numpy(x).cuda()
    got = vpmc.weights_dose(_dev(m), xd).cpu().numpy().astype(np.float64)
    assert np.max(np.abs(got - d)) <= 2e-6 * d.max()
    cls = np.ones(n_rows, dtype=np.uint8)
    out = vpmc.target_indices([_dev(m)], torch.from_numpy(cls).cuda(), 30.0, xd)
    near = np.abs(d - 30.0) <= 1e-5 * 30.0
    assert abs(out[0, 0] * n_rows - np.sum(d >= 30.0)) <= near.sum() + 1e-6 * n_rows
    assert out[0, 3] == pytest.approx(d.max() / 30.0, rel=2e-6)
