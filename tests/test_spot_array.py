"""The binding's spot list copied field by field equals the row-by-row copy,
byte for byte: contiguous, strided and reversed views, other field types and
orders, one spot and none."""
import numpy as np
import pytest

from paper_2307_01416_gb300 import vpmc
from paper_2307_01416_gb300 import workloads as W


def _spots(n):
    g = np.random.default_rng(n)
    return W.make_spots([(int(b), e, x, y, 3.0, 2.0, int(h), w) for b, e, x, y, h, w in
                         zip(g.integers(0, 64, n), g.uniform(1, 250, n), g.normal(0, 9, n), g.normal(0, 9, n),
                             g.integers(0, 1 << 33, n), g.uniform(0, 3, n))])


@pytest.mark.parametrize("n", [1, 2, 257])
@pytest.mark.parametrize("view", ["whole", "every other", "reversed", "packed types"])
def test_fields_equal_rows(n, view):
    s = _spots(n)
    if view == "every other":
        s = s[::2]
    elif view == "reversed":
        s = s[::-1]
    elif view == "packed types":
        t = np.dtype([("weight", np.float32), ("n_hist", np.uint32), ("y", np.float32), ("x", np.int16), ("beam", np.int64),
                      ("sigma", np.float64), ("div_mrad", np.float32), ("energy", np.float32), ("note", "S3")])
        p = np.zeros(n, dtype=t)
        for k in s.dtype.names:
            p[k] = s[k] if k != "n_hist" else s[k] % 1000
        s = p
    a = vpmc.spot_array(s)
    assert len(a) == len(s) and bytes(a) == bytes(vpmc.spot_array(list(s)))


def test_no_spots_and_refusals():
    assert len(vpmc.spot_array(_spots(2)[:0])) == 1
    s = _spots(3).astype([(k, np.float64) for k in W.SPOT_DTYPE.names])
    s["n_hist"][1] = np.nan                       # not a count: refused by either path
    with pytest.raises(ValueError):
        vpmc.spot_array(s)
