"""Performance cases of the proton Monte Carlo engine.

The work a treatment-planning program has this package do, each through its
public entry points: dose of a few or of many spots, robust
influence-matrix sets, spot-weight optimisation over such a set, evaluation
of a plan, and the learned aperture surrogate (track generation, training,
network outputs).  A case is a dict of plain values; prepare() makes what the
program has in hand before the call, run() is one call, work() the bytes and
operations that the call cannot do without, exact() the same result in 64
bits where plain torch can give it.
"""
import math

import numpy as np
import torch

from paper_2307_01416_gb300 import vpmc
from paper_2307_01416_gb300 import workloads as W

# lane-operations of one condensed-history step (a minimal implementation of
# the step's formulas) in the voxelised patient and in a homogeneous slab
OPS_PATIENT_STEP = 299
OPS_SLAB_STEP = 254
NET_FLOPS = 2 * (6 * 128 + 128 * 128 + 128 * 45)     # one row through the network
DOSE_PRESCRIPTION = 2.0


def listed():
    return [
        # a serving loop that asks for one beamlet's quick dose through the
        # entry point that allocates nothing: launches and latency
        {"name": "beamlet_quick", "kind": "pencil", "energy": 100.0, "histories": 2000, "nx": 50, "ny": 50, "nz": 150,
         "spacing": 2.0, "noalloc": True},
        # the pencil beam in water of the engine's own configuration
        {"name": "pencil_water", "kind": "pencil", "energy": 100.0, "histories": 100_000, "nx": 50, "ny": 50,
         "nz": 150, "spacing": 2.0, "noalloc": False},
        # commissioning dose: water phantom behind range shifter and brass
        # aperture, four energy layers of 1e6 protons
        {"name": "aperture_water", "kind": "aperture", "diameter": 20.0, "range_shifter": True, "layers": 4,
         "per_layer": 1_000_000},
        # forward dose of a three-field head plan at planning statistics
        {"name": "head_dose", "kind": "head", "volume": 8.4, "histories": 32_000_000},
        # robust influence-matrix set: 13 scenarios of the small-target plan
        {"name": "head_im13", "kind": "matrix", "volume": 0.4, "histories": 7_500_000, "scenarios": 13},
        # single-beamlet edge sweep as one influence matrix on a 1 mm grid:
        # 97 energies, few histories per column
        {"name": "edge_sweep_im", "kind": "edge", "range_shifter": False, "beamlets": 97, "per_beamlet": 20_000},
        # re-optimisation of a small plan (a few hundred spots)
        {"name": "optimise_small", "kind": "optimise", "nx": 36, "ny": 36, "nz": 40, "spots": 300, "scenarios": 13,
         "target": 7.0, "iterations": 60},
        # optimisation over the head plan's 13 matrices (some 6e7 entries each)
        {"name": "optimise_head", "kind": "optimise", "nx": 128, "ny": 128, "nz": 120, "spots": 5220, "scenarios": 13,
         "target": 6.3, "iterations": 50},
        # plan evaluation: target indices over the 13 scenarios and the
        # nominal dose of the weights
        {"name": "evaluate_head", "kind": "evaluate", "nx": 128, "ny": 128, "nz": 120, "spots": 5220, "scenarios": 13,
         "target": 6.3},
        # network outputs for a batch of brass entries (not a whole tile more)
        {"name": "net_forward", "kind": "forward", "rows": 4_194_381},
        # training epoch of the surrogate on a million tracks
        {"name": "net_train", "kind": "train", "rows": 1_000_000, "batch": 16_384, "epochs": 1},
        # training tracks: plain brass transport of the eight training openings
        {"name": "brass_tracks", "kind": "tracks", "per_opening": 250_000, "network": False},
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng):
    kind = rng.choice(["pencil", "pencil", "aperture", "head", "matrix", "edge", "optimise", "evaluate", "forward",
                       "train", "tracks"])
    if kind == "pencil":
        h = rng.choice([1.0, 2.0, 2.5, 3.0])
        nx, ny, nz = (int(rng.uniform(lo, hi) / h) for lo, hi in ((60.0, 120.0), (60.0, 120.0), (200.0, 340.0)))
        # the entry point without allocations holds up to 2^21 voxels
        return {"kind": kind, "energy": round(rng.uniform(71.3, 228.8), 2), "histories": int(_log(rng, 2000, 2_000_000)),
                "nx": nx, "ny": ny, "nz": nz, "spacing": h, "noalloc": nx * ny * nz <= 1 << 21 and rng.random() < 0.6}
    if kind == "aperture":
        return {"kind": kind, "diameter": rng.choice([10.0, 20.0, 30.0, 40.0]), "range_shifter": rng.random() < 0.6,
                "layers": rng.randint(1, 6), "per_layer": int(_log(rng, 20_000, 1_500_000))}
    if kind == "head":
        return {"kind": kind, "volume": round(_log(rng, 0.4, 43.0), 2), "histories": int(_log(rng, 500_000, 32_000_000))}
    if kind == "matrix":
        n = rng.choice([1, 3, 7, 13])
        return {"kind": kind, "volume": round(_log(rng, 0.3, 0.5), 3), "histories": int(_log(rng, 300_000, 7_500_000)),
                "scenarios": n}
    if kind == "edge":
        return {"kind": kind, "range_shifter": rng.random() < 0.5, "beamlets": rng.randint(3, 97),
                "per_beamlet": int(_log(rng, 2000, 100_000))}
    if kind in ("optimise", "evaluate"):
        nx, ny, nz = rng.randint(33, 128), rng.randint(33, 128), rng.randint(37, 120)
        c = {"kind": kind, "nx": nx, "ny": ny, "nz": nz, "spots": int(_log(rng, 150, 5220)),
             "scenarios": rng.choice([1, 3, 13]), "target": round(rng.uniform(3.0, min(7.0, 0.2 * min(nx, ny, nz))), 2)}
        if kind == "optimise":
            c["iterations"] = rng.randint(10, 60)
        return c
    if kind == "forward":
        return {"kind": kind, "rows": int(_log(rng, 1, 4_194_381))}
    if kind == "train":
        batch = int(_log(rng, 512, 20_000))
        return {"kind": kind, "rows": batch * rng.randint(1, 40) + rng.randint(1, batch), "batch": batch,
                "epochs": rng.randint(1, 2)}
    return {"kind": "tracks", "per_opening": int(_log(rng, 2000, 250_000)), "network": rng.random() < 0.4}


# ---------------------------------------------------------------- inputs
def _counts(rng, total, n):
    """n log-uniform history counts (a factor of 20 apart at most) of about `total` in all."""
    w = np.exp(rng.uniform(0.0, math.log(20.0), n))
    return np.maximum(np.ceil(w * (total / w.sum())), 1).astype(np.int64)


def _head(case, seed):
    rng = np.random.default_rng(seed)
    problem, spots, _, _ = W.head_plan(case["volume"])
    spots["n_hist"] = _counts(rng, case["histories"], len(spots))
    return problem, spots


def _matrices(case, seed):
    """Influence matrices of a three-field plan (0, 90, 270 degrees) on a
    2 mm grid, as CSR on the GPU: per spot a Gaussian lateral profile, a
    plateau and a peak at the spot's depth, kept above 1e-4 of the column's
    maximum, with the noise of a Monte Carlo column.  The scenarios shift the
    spots and scale their depths."""
    dev = torch.device("cuda")
    g = torch.Generator(device=dev)
    g.manual_seed(int(seed))
    shape = (case["nx"], case["ny"], case["nz"])
    n, rt = case["spots"], case["target"]
    ctr = [0.5 * s for s in shape]
    per = (n + 2) // 3
    sigma, half = 1.9, 8
    rnd = lambda *s: torch.rand(*s, generator=g, device=dev)  # noqa: E731
    rad, ang = (rt + 3.0) * rnd(n).sqrt(), 2 * math.pi * rnd(n)
    la, lb, dep, amp = rad * ang.cos(), rad * ang.sin(), (2 * rnd(n) - 1) * (rt + 2.5), 1e-9 * (0.5 + rnd(n))
    field = torch.arange(n, device=dev) // per
    lateral = [(0, 2), (1, 2), (1, 2)]
    axis, sign = [1, 0, 0], [1.0, -1.0, 1.0]
    shifts = [(0.0, 0.0, 0.0, 1.0)]
    for k in range(12):
        v = [0.0, 0.0, 0.0]
        v[(k // 2) % 3] = 1.5 if k % 2 == 0 else -1.5
        shifts.append((*v, 1.0 + (0.035 if k % 2 == 0 else -0.035) * (k >= 6)))
    mats = []
    nd = int(max(shape[0], shape[1]) // 2 + rt + 8)
    o = torch.arange(-half, half + 1, device=dev)
    k = torch.arange(nd, device=dev)
    for sx, sy, sz, scale in shifts[: case["scenarios"]]:
        sh = (sx, sy, sz)
        keys, vals = [], []
        for f in range(3):
            j = torch.nonzero(field == f).reshape(-1)
            if j.numel() == 0:
                continue
            ax, sg, (a, b) = axis[f], sign[f], lateral[f]
            pa, pb = ctr[a] + sh[a] + la[j], ctr[b] + sh[b] + lb[j]
            enter = 0.0 if sg > 0 else float(shape[ax])
            peak = (sg * (ctr[ax] + sh[ax] - enter) + dep[j]) * scale            # depth of the peak from the entrance
            ia, ib = pa.floor().long()[:, None] + o, pb.floor().long()[:, None] + o
            ga = torch.exp(-0.5 * ((ia + 0.5 - pa[:, None]) / sigma) ** 2)
            gb = torch.exp(-0.5 * ((ib + 0.5 - pb[:, None]) / sigma) ** 2)
            dz = k + 0.5 - peak[:, None]
            gd = torch.where(dz <= 0, 0.3 + 0.7 * torch.exp(-0.125 * dz * dz), torch.exp(-0.5 * dz * dz))
            v = ga[:, :, None, None] * gb[:, None, :, None] * gd[:, None, None, :]
            idx = [None, None, None]
            idx[a], idx[b] = ia[:, :, None, None], ib[:, None, :, None]
            idx[ax] = (k if sg > 0 else shape[ax] - 1 - k)[None, None, None, :]
            inside = v > 1e-4
            for d in range(3):
                inside &= (idx[d] >= 0) & (idx[d] < shape[d])
            row = idx[0] + shape[0] * (idx[1] + shape[1] * idx[2])
            keys.append((row * n + j[:, None, None, None])[inside])
            vals.append((v * amp[j][:, None, None, None])[inside])
            del v, row, inside
        key, order = torch.sort(torch.cat(keys))
        val = torch.cat(vals)[order]
        val = (val * (1 + 0.05 * torch.randn(val.shape, generator=g, device=dev)).clamp_min(0.1)).float()
        row = torch.div(key, n, rounding_mode="floor")
        ptr = torch.zeros(shape[0] * shape[1] * shape[2] + 1, dtype=torch.int64, device=dev)
        ptr[1:] = torch.bincount(row, minlength=ptr.numel() - 1).cumsum(0)
        mats.append({"row_ptr": ptr, "col": (key - row * n).int(), "val": val, "shape": (ptr.numel() - 1, n)})
        del keys, vals, key, order, row
    # structures: the spherical target (1) and the ring five voxels around it (2)
    x, y, z = (torch.arange(s, device=dev) + 0.5 - c for s, c in zip(shape, ctr))
    r = (x[None, None, :] ** 2 + y[None, :, None] ** 2 + z[:, None, None] ** 2).sqrt().reshape(-1)
    cls = ((r <= rt).to(torch.uint8) + 2 * ((r > rt) & (r <= rt + 5.0)).to(torch.uint8)).contiguous()
    # initial weights: the nominal mean target dose is 1.3 of the prescription
    x0 = 0.5 + rnd(n)
    dose = _product64(mats[0], x0.double())
    x0 = (x0 * (1.3 * DOSE_PRESCRIPTION / dose[cls == 1].mean())).float()
    return mats, cls, x0


def _network(seed):
    g = np.random.default_rng(seed)
    return np.concatenate([g.standard_normal(128 * 6) * math.sqrt(2 / 6), 0.1 * g.standard_normal(128),
                           g.standard_normal(128 * 128) * math.sqrt(2 / 128), 0.1 * g.standard_normal(128),
                           g.standard_normal(45 * 128) * 0.5 * math.sqrt(1 / 128),
                           0.1 * g.standard_normal(45)]).astype(np.float32)


def _rows(n, seed):
    """Network inputs with the ranges of its features (edge distance, energy,
    two angles, curvature, relative range), labels and targets."""
    dev = torch.device("cuda")
    g = torch.Generator(device=dev)
    g.manual_seed(int(seed))
    u = torch.rand(n, 6, generator=g, device=dev)
    z = torch.randn(n, 7, generator=g, device=dev)
    feat = 2 * u - 1
    feat[:, 2:4] = z[:, 5:].clamp(-3, 3)
    label = (u[:, 0] < 0.6).to(torch.int32)
    target = z[:, :5] * label[:, None]
    return feat.contiguous(), target.contiguous(), label


def prepare(case, seed):
    kind = case["kind"]
    s = {"kind": kind, "case": case}
    if kind == "pencil":
        problem, s["spots"] = W.pencil_beam_water(case["histories"], case["energy"], shape=(case["nx"], case["ny"], case["nz"]),
                                                  spacing=(case["spacing"],) * 3)
        s["engine"], s["opts"] = vpmc.Engine(problem), W.Options(seed=seed)
        if case["noalloc"]:
            s["dose"] = torch.empty((case["nz"], case["ny"], case["nx"]), dtype=torch.float32, device="cuda")
    elif kind == "aperture":
        problem, s["spots"] = W.water_aperture_case(case["diameter"], case["range_shifter"], case["per_layer"],
                                                    max_layers=case["layers"])
        s["engine"], s["opts"] = vpmc.Engine(problem), W.Options(seed=seed)
    elif kind == "head":
        problem, s["spots"] = _head(case, seed)
        s["engine"], s["opts"] = vpmc.Engine(problem), W.Options(seed=seed)
    elif kind == "matrix":
        problem, s["spots"] = _head(case, seed)
        s["engine"], s["opts"] = vpmc.Engine(problem), W.Options(seed=seed)
        s["scenarios"] = W.robust_scenarios()[: case["scenarios"]]
    elif kind == "edge":
        problem = W.edge_beamlet_problem(case["range_shifter"])
        s["spots"] = np.concatenate([W.edge_beamlet_spot(e, case["per_beamlet"])
                                     for e in W.machine_energies()[: case["beamlets"]]])
        s["engine"], s["opts"] = vpmc.Engine(problem), W.Options(seed=seed)
        s["scenarios"] = [W.Scenario()]
    elif kind in ("optimise", "evaluate"):
        s["mats"], s["cls"], s["x0"] = _matrices(case, seed)
    elif kind == "forward":
        s["engine"] = vpmc.Engine(vpmc.surrogate_training_problem())
        s["engine"].surrogate_set_weights(_network(seed))
        s["feat"] = _rows(case["rows"], seed)[0]
    elif kind == "train":
        s["engine"], s["weights"] = vpmc.Engine(vpmc.surrogate_training_problem()), _network(seed)
        s["feat"], s["target"], s["label"] = _rows(case["rows"], seed)
    else:
        s["engine"], s["opts"] = vpmc.Engine(vpmc.surrogate_training_problem()), W.Options(seed=seed)
        if case["network"]:
            s["engine"].surrogate_set_weights(_network(seed))
    if kind in ("matrix", "edge"):
        # the plan's own store of its matrices, of fixed size: a column keeps
        # some 7,000 voxels of the 2 mm grid and 1e5 of the 1 mm grid
        size = (len(s["scenarios"]), len(s["spots"]) * (12_000 if kind == "matrix" else 400_000))
        s["row_ptr"] = torch.empty((size[0], problem.scoring.nvox + 1), dtype=torch.int64, device="cuda")
        s["col"] = torch.zeros(size, dtype=torch.int32, device="cuda")
        s["val"] = torch.zeros(size, dtype=torch.float32, device="cuda")
    return s


# ---------------------------------------------------------------- one call
_COUNTS = ("histories", "steps", "errors", "steps_rs", "steps_aperture")
_ENERGIES = ("e_in", "e_dep", "e_leak", "e_rs", "e_aperture", "e_nuc")


def _tally(st, names):
    return [st[k] for k in names]


def run(s):
    kind, case = s["kind"], s["case"]
    if kind == "pencil" and case["noalloc"]:
        st = s["engine"].run_spots_noalloc(s["spots"], s["dose"], opts=s["opts"])
        return {"dose": s["dose"], "counts": _tally(st, _COUNTS), "energies": _tally(st, _ENERGIES)}
    if kind in ("pencil", "aperture", "head"):
        dose, st, _ = s["engine"].run_spots(s["spots"], opts=s["opts"])
        return {"dose": dose, "counts": _tally(st, _COUNTS), "energies": _tally(st, _ENERGIES)}
    if kind in ("matrix", "edge"):
        mats, st = s["engine"].influence_matrix(s["spots"], s["scenarios"], s["opts"])
        for i, m in enumerate(mats):
            for k in ("row_ptr", "col", "val"):
                s[k][i, : m[k].numel()].copy_(m[k])
        return {"row_ptr": s["row_ptr"], "col": s["col"], "val": s["val"], "counts": _tally(st, _COUNTS),
                "energies": _tally(st, _ENERGIES)}
    if kind == "optimise":
        x = s["x0"].clone()
        history, _, _ = vpmc.robust_optimize(s["mats"], s["cls"], x, DOSE_PRESCRIPTION, iterations=case["iterations"])
        return {"weights": x, "history": history}
    if kind == "evaluate":
        return {"indices": vpmc.target_indices(s["mats"], s["cls"], DOSE_PRESCRIPTION, s["x0"]),
                "dose": vpmc.weights_dose(s["mats"][0], s["x0"])}
    if kind == "forward":
        return {"z": s["engine"].surrogate_forward(s["feat"])}
    if kind == "train":
        s["engine"].surrogate_set_weights(s["weights"])
        loss = s["engine"].surrogate_train(s["feat"], s["target"], s["label"], batch=case["batch"], epochs=case["epochs"])
        return {"weights": s["engine"].surrogate_get_weights(), "loss": loss}
    n = len(W.SURROGATE_RADII)
    feat, target, label = s["engine"].surrogate_tracks(list(range(n)), case["per_opening"], s["opts"],
                                                       use_surrogate=case["network"])
    return {"feat": feat, "target": target, "label": label}


# ---------------------------------------------------------------- what a call cannot do without
def _patient_steps(energy):
    """Condensed-history steps of one proton in water: one per millimetre,
    and one per 1 % of the energy over the last 56 mm of its range."""
    return max(0.022 * energy ** 1.77 - 56.0, 0.0) + 100.0 * math.log(min(energy, 83.0) / 0.5)


def work(case):
    kind = case["kind"]
    if kind == "pencil":
        nv = case["nx"] * case["ny"] * case["nz"]
        return {"bytes": 6.0 * nv, "flops": case["histories"] * _patient_steps(case["energy"]) * OPS_PATIENT_STEP}
    if kind == "aperture":
        n = case["layers"] * case["per_layer"]
        slab = 45.0 if case["range_shifter"] else 0.0
        inside = math.pi * (0.5 * case["diameter"]) ** 2 / (math.pi * (0.5 * case["diameter"] + 10.0) ** 2)
        return {"bytes": 6.0 * 100 * 100 * 150,
                "flops": n * (slab * OPS_SLAB_STEP + inside * _patient_steps(80.0 if slab else 105.0) * OPS_PATIENT_STEP)}
    if kind in ("head", "matrix"):
        n = case["histories"] * case.get("scenarios", 1)
        nnz = 0 if kind == "head" else 8.0e6 * case["scenarios"]
        return {"bytes": 2.0 * 256 * 256 * 160 + 4.0 * 128 * 128 * 120 + 8.0 * nnz,
                "flops": 0.5 * n * _patient_steps(95.0) * OPS_PATIENT_STEP + case["histories"] * 45.0 * OPS_SLAB_STEP}
    if kind == "edge":
        n = case["beamlets"] * case["per_beamlet"]
        return {"bytes": 6.0 * 40 * 40 * 350 + 8.0 * 96_000 * case["beamlets"],
                "flops": n * 0.4 * _patient_steps(110.0) * OPS_PATIENT_STEP}
    if kind in ("optimise", "evaluate"):
        nd = min(0.5 * max(case["nx"], case["ny"]), 60.0)
        nnz = case["spots"] * 210.0 * nd
        if kind == "evaluate":
            n = nnz * (case["scenarios"] + 1)
            return {"bytes": 8.0 * n + 12.0 * case["nx"] * case["ny"] * case["nz"] * case["scenarios"], "flops": 2.0 * n}
        rt = case["target"]
        rows = 4.19 * (rt + 5.0) ** 3
        share = min(1.0, rows / (case["spots"] and 3 * math.pi * (rt + 11.0) ** 2 * nd))
        n = nnz * share
        # every iteration reads the target and ring rows of all scenarios, and those of one for the gradient
        return {"bytes": 8.0 * n * case["scenarios"] + case["iterations"] * 6.0 * n * (case["scenarios"] + 1),
                "flops": case["iterations"] * 2.0 * n * (case["scenarios"] + 1)}
    if kind == "forward":
        return {"bytes": (6 + 45) * 4.0 * case["rows"] + 4.0 * 23213, "flops": float(NET_FLOPS) * case["rows"]}
    if kind == "train":
        n = case["rows"] * case["epochs"]
        return {"bytes": 48.0 * n + 24.0 * 23213 * math.ceil(case["rows"] / case["batch"]) * case["epochs"],
                "flops": 3.0 * NET_FLOPS * n}
    n = 8.0 * case["per_opening"]
    return {"bytes": 48.0 * n, "flops": n * (NET_FLOPS if case["network"] else 60.0 * OPS_SLAB_STEP)}


# ---------------------------------------------------------------- the same results in 64 bits
def _product64(m, x):
    n = m["shape"][0]
    row = torch.repeat_interleave(torch.arange(n, device=x.device), m["row_ptr"].diff())
    return torch.zeros(n, dtype=torch.float64, device=x.device).index_add_(0, row, m["val"].double() * x[m["col"].long()])


def _exact_optimise(case, mats, cls, x0):
    """Adam on the worst scenario's objective, clamped at zero."""
    keep = torch.nonzero(cls > 0).reshape(-1)
    target = cls[keep] == 1
    nt, nr = int(target.sum()), max(int((~target).sum()), 1)
    parts = []
    for m in mats:
        length = (m["row_ptr"][1:] - m["row_ptr"][:-1])[keep]
        row = torch.repeat_interleave(torch.arange(keep.numel(), device=x0.device), length)
        first = torch.repeat_interleave(m["row_ptr"][keep] - (length.cumsum(0) - length), length)
        at = first + torch.arange(row.numel(), device=x0.device)
        parts.append((row, m["col"][at].long(), m["val"][at].double()))
    x = x0.double()
    step = 0.05 * float(x.mean())
    m1, m2 = torch.zeros_like(x), torch.zeros_like(x)
    dp, history = DOSE_PRESCRIPTION, []
    for it in range(1, case["iterations"] + 1):
        fs, slopes = [], []
        for row, col, val in parts:
            d = torch.zeros(keep.numel(), dtype=torch.float64, device=x.device).index_add_(0, row, val * x[col])
            under, over = (dp - d).clamp_min(0) * target, (d - 1.05 * dp).clamp_min(0) * target
            ring = (d - 0.6 * dp).clamp_min(0) * ~target
            fs.append((under ** 2).sum() / nt + 0.5 * (over ** 2).sum() / nt + 0.2 * (ring ** 2).sum() / nr)
            slopes.append(2 * (0.5 * over - under) / nt + 0.4 * ring / nr)
        fs = torch.stack(fs)
        w = int(fs.argmax())
        history.append(float(fs[w]))
        row, col, val = parts[w]
        g = torch.zeros_like(x).index_add_(0, col, val * slopes[w][row])
        m1, m2 = 0.9 * m1 + 0.1 * g, 0.999 * m2 + 0.001 * g * g
        x = (x - step * (m1 / (1 - 0.9 ** it)) / ((m2 / (1 - 0.999 ** it)).sqrt() + 1e-8)).clamp_min(0)
    return {"weights": x, "history": np.array(history)}


def exact(case, seed):
    kind = case["kind"]
    if kind == "optimise":
        return _exact_optimise(case, *_matrices(case, seed))
    if kind == "evaluate":
        mats, cls, x0 = _matrices(case, seed)
        x, dp, rows = x0.double(), DOSE_PRESCRIPTION, []
        for m in mats:
            d = _product64(m, x)
            t, n = d[cls == 1], int((cls == 1).sum())
            rows.append([float((t >= dp).sum()) / n, float(t.min()) / dp, float((d >= dp).sum()) / n, float(t.max()) / dp])
        return {"indices": np.array(rows), "dose": _product64(mats[0], x)}
    if kind == "forward":
        w = torch.from_numpy(_network(seed)).cuda().double()
        w1, b1, w2, b2, w3, b3 = w.split([768, 128, 16384, 128, 5760, 45])
        x = _rows(case["rows"], seed)[0].double()
        h = (x @ w1.view(128, 6).T + b1).clamp_min(0)
        h = (h @ w2.view(128, 128).T + b2).clamp_min(0)
        return {"z": h @ w3.view(45, 128).T + b3}
    # random histories and what is trained on them have no value of this kind
    return None
