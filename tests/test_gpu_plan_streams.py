"""Plan calls on a stream of the caller's own, with inputs that the legacy
default stream is still making (it sleeps 0.1 s first): every call waits for
them, as it would on the default stream itself."""
import numpy as np
import pytest

from paper_2307_01416_gb300 import workloads as W

pytestmark = pytest.mark.gpu

SHAPE, SPOTS, DP = (20, 20, 24), 40, 2.0


@pytest.fixture(scope="module")
def plan():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    mats = [{k: torch.from_numpy(v).cuda() if isinstance(v, np.ndarray) else v for k, v in m.items()}
            for m in W.synthetic_spot_matrices(SHAPE, SPOTS, 3)]
    cls = torch.from_numpy(W.synthetic_structure_classes(SHAPE, 4.0)).cuda().reshape(-1).contiguous()
    x = torch.from_numpy(np.random.default_rng(2).uniform(0.5, 1.5, SPOTS).astype(np.float32)).cuda()
    torch.cuda.synchronize()
    return torch, mats, cls, x


def _optimise(mats, cls, x, stream):
    from paper_2307_01416_gb300 import vpmc
    history, _, _ = vpmc.robust_optimize(mats, cls, x, DP, iterations=5, stream=stream)
    return np.concatenate([history, x.cpu().numpy()])


def _indices(mats, cls, x, stream):
    from paper_2307_01416_gb300 import vpmc
    return vpmc.target_indices(mats, cls, DP, x, stream=stream)


def _dose(mats, cls, x, stream):
    from paper_2307_01416_gb300 import vpmc
    return vpmc.weights_dose(mats[0], x, stream=stream).cpu().numpy()


@pytest.mark.parametrize("call", [_optimise, _indices, _dose])
@pytest.mark.parametrize("late", ["weights", "classes", "values"])
def test_inputs_made_on_the_default_stream(plan, call, late):
    torch, mats, cls, x = plan
    side = torch.cuda.Stream()
    want = call(mats, cls, x.clone(), None)
    mats = [{**m, "val": m["val"].clone()} for m in mats]
    cls, x = cls.clone(), x.clone()
    made = {"weights": [x], "classes": [cls], "values": [m["val"] for m in mats]}[late]
    kept = [t.clone() for t in made]
    for t in made:
        t.zero_()
    torch.cuda.synchronize()
    torch.cuda._sleep(200_000_000)
    for t, k in zip(made, kept):
        t.copy_(k)
    got = call(mats, cls, x, side)
    torch.cuda.synchronize()
    assert np.array_equal(got, want)
