"""The surrogate's tensor-core kernels where their tiles can go wrong, against
the oracle: forward at the edges of a 128-row tile, of the four tile pipelines
of a CTA and of the grid (a pipeline's second tile, whole and ragged), with a
row of NaN among them; the gradient with one row, a ragged tile and several
tiles per CTA.  BF16 operands, FP32 sums: the tolerances are those of the
network's parity tests (1e-2 relative, the gradient per tensor)."""
import numpy as np
import pytest

from oracle import surrogate_oracle as S
from tests.test_gpu_surrogate import _batch, _dev, _flat, _params, _unflat

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def eng():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2307_01416_gb300 import vpmc
    e = vpmc.Engine(vpmc.surrogate_training_problem())
    yield e
    e.close()


@pytest.mark.parametrize("n", [129, 511, 512, 513, 152 * 512 - 1, 152 * 512, 152 * 512 + 129])
def test_forward_tiles(eng, n):
    import torch
    P = _params(4)
    eng.surrogate_set_weights(_flat(P))
    x, _, _ = _batch(n, n)
    bad = n // 2
    x[bad] = np.nan
    z = eng.surrogate_forward(_dev(torch, x)).cpu().numpy().astype(np.float64)
    ok = np.arange(n) != bad
    zo, _ = S.forward(P, x[ok].astype(np.float64), bf16_ops=True)
    assert np.max(np.abs(z[ok] - zo) / np.maximum(np.abs(zo), 1.0)) < 1e-2
    # relu(NaN) is 0 in the kernels: a NaN input gives the outputs of h1 = 0
    h2 = np.maximum(P["b2"], 0.0)
    zn = S.bf16(P["W3"]) @ S.bf16(h2) + P["b3"]
    assert np.max(np.abs(z[bad] - zn) / np.maximum(np.abs(zn), 1.0)) < 1e-2


@pytest.mark.parametrize("n", [1, 129, 152 * 128 + 5, 3 * 152 * 128])
def test_gradient_tiles(eng, n):
    import torch
    P = _params(6)
    eng.surrogate_set_weights(_flat(P))
    x, t, y = _batch(n, 50 + n)
    g, loss = eng.surrogate_gradient(_dev(torch, x), _dev(torch, y), _dev(torch, t))
    z, cache = S.forward(P, x.astype(np.float64), bf16_ops=True)
    go = S.backward(cache, S.loss_grad(z, t.astype(np.float64), y.astype(np.float64)), bf16_ops=True)
    assert loss == pytest.approx(S.loss(z, t.astype(np.float64), y.astype(np.float64)), rel=2e-3)
    gu = _unflat(g.cpu().numpy())
    for k in gu:
        ref = np.asarray(go[k])
        assert np.linalg.norm(gu[k] - ref) <= 1e-2 * np.linalg.norm(ref) + 1e-12, k
