"""The plan kernels where a row's length decides their path, against FP64:
rows of 0 to several batches of a sub-warp, with out-of-range spots, in the
full-matrix products (dose of the weights, target indices), and dense target
rows in the optimiser (a warp per row; the other optimiser tests' rows are
short and take eight lanes).  A dose is an FP32 sum of n products: 2e-6 of the
largest as in the optimiser's parity tests; the 15 iterations keep 1e-4."""
import numpy as np
import pytest

from oracle import optimizer_oracle as Q

pytestmark = pytest.mark.gpu

LENGTHS = [0, 1, 7, 8, 9, 63, 64, 65, 71, 128, 129, 300]


def _matrix(n_rows, n_cols, lengths, seed, strays=True):
    g = np.random.default_rng(seed)
    length = np.asarray(lengths)[g.integers(0, len(lengths), n_rows)]
    rp = np.zeros(n_rows + 1, dtype=np.int64)
    np.cumsum(length, out=rp[1:])
    col = np.concatenate([np.sort(g.choice(n_cols, k, replace=False)) for k in length]).astype(np.int32)
    val = g.uniform(0.1, 1.0, col.size).astype(np.float32)
    clean = np.zeros((n_rows, n_cols))
    clean[np.repeat(np.arange(n_rows), length), col] = val
    if strays:                                       # entries that every product skips
        k = np.flatnonzero(g.random(col.size) < 0.01)
        clean[np.repeat(np.arange(n_rows), length)[k], col[k]] = 0.0
        col[k] = np.where(g.random(k.size) < 0.5, -1, n_cols + 3)
        val[k] = np.inf
    return {"row_ptr": rp, "col": col, "val": val, "shape": (n_rows, n_cols)}, clean


def _dev(m):
    import torch
    return {k: torch.from_numpy(v).cuda() if isinstance(v, np.ndarray) else v for k, v in m.items()}


@pytest.mark.parametrize("n_rows", [1, 3, 1003, 9731])
def test_full_matrix_products(n_rows):
    import torch
    from paper_2307_01416_gb300 import vpmc
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    n_cols = 400
    mats = [_matrix(n_rows, n_cols, LENGTHS, 10 * n_rows + s) for s in range(3)]
    g = np.random.default_rng(n_rows)
    x = g.uniform(0.0, 2.0, n_cols).astype(np.float32)
    cls = g.integers(0, 3, n_rows).astype(np.uint8)
    cls[0] = 1
    xd, dp = torch.from_numpy(x).cuda(), 30.0
    doses = [A @ x.astype(np.float64) for _, A in mats]
    for (m, _), d in zip(mats, doses):
        got = vpmc.weights_dose(_dev(m), xd).cpu().numpy().astype(np.float64)
        assert np.max(np.abs(got - d)) <= 2e-6 * max(np.max(d), 1.0)
    got = vpmc.target_indices([_dev(m) for m, _ in mats], torch.from_numpy(cls).cuda(), dp, xd)
    t = cls == 1
    for s, d in enumerate(doses):
        r = Q.target_indices(d, cls, dp)
        near = np.abs(d - dp) <= 1e-5 * dp
        assert abs(got[s, 0] - r["V100"]) * t.sum() <= np.sum(near & t) + 1e-9
        assert abs(got[s, 2] - r["CI100"]) * t.sum() <= np.sum(near) + 1e-9
        assert got[s, 1] == pytest.approx(r["Dmin"], rel=2e-6, abs=1e-7)
        assert got[s, 3] == pytest.approx(r["RHI100"], rel=2e-6)


@pytest.mark.parametrize("lengths", [[0, 5, 130, 300, 390], [128], [129]], ids=["mixed", "128", "129"])
def test_optimiser_rows(lengths):
    import scipy.sparse as sp
    import torch
    from paper_2307_01416_gb300 import vpmc
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    n_rows, n_cols = 4099, 400                       # classes over more than one block of 4,096 voxels
    mats = [_matrix(n_rows, n_cols, lengths, 7 + s) for s in range(2)]
    for m, A in mats:                                # strays carry finite values here
        m["val"][~np.isfinite(m["val"])] = 1.0
    g = np.random.default_rng(3)
    cls = g.integers(0, 3, n_rows).astype(np.uint8)
    x0 = g.uniform(0.5, 1.5, n_cols).astype(np.float32)
    dp = float(np.mean((mats[0][1] @ x0)[cls == 1])) / 1.3
    p = Q.OptParams(prescription=dp, lr=0.05)
    x_ref, h_ref = Q.optimise([sp.csr_matrix(A) for _, A in mats], x0.astype(np.float64), cls, p, 15)
    x = torch.from_numpy(x0.copy()).cuda()
    h, _, _ = vpmc.robust_optimize([_dev(m) for m, _ in mats], torch.from_numpy(cls).cuda(), x, dp, iterations=15, lr=0.05)
    assert np.max(np.abs(h - h_ref) / h_ref) <= 1e-4
    assert np.max(np.abs(x.cpu().numpy() - x_ref)) <= 1e-4 * np.mean(x0)
