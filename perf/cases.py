"""What a user of the library has it do, as measurable cases: steps of boosted-frame runs in 2D, 3D and 1D, a batched
ensemble, the labelling of stage runs, and the surrogate's training and serving.

A case is a dict of plain values; ``prepare`` makes the state a user's program holds before the call (a context with
plasma, laser and a few dozen steps behind it; a network and its data), ``run`` is one pass through the public entry
points. A pass of a run advances it and reads the six field components and the diagnostics back, the loop of
``stage_labels`` and of a lab-frame monitor; the run goes on from pass to pass, with plasma streaming in throughout.
"""
import math

import numpy as np
import torch

from paper_1009_2727_gb300 import workloads as W
from paper_1009_2727_gb300.pic import Ensemble, Simulation
from paper_1009_2727_gb300.surrogate import MLP, stage_labels

C = 299792458.0
WIDTHS = (6, 256, 256, 256, 4)   # the surrogate's default network


def listed():
    return [
        # The 0.1 GeV-class stage at full size (13.2 M electrons), mixed precision, in the layout the autotuner picks
        # for it: the production run of one stage.
        {"name": "stage2d", "kind": "stage", "precision": "mixed", "nz": 4096, "nx": 256, "ppc": 4, "order": 3,
         "gather": "energy", "strides": "", "theta": 0.1, "tile": "8x16", "sort": 64, "warm": 96, "steps": 8},
        # The same stage with the wide-band filter S(1:2:4) of the paper's high-gamma runs, in the default layout.
        {"name": "stage2d_wideband", "kind": "stage", "precision": "mixed", "nz": 1536, "nx": 224, "ppc": 2,
         "order": 3, "gather": "energy", "strides": "1:2:4", "theta": 0.1, "tile": "", "sort": 0, "warm": 80,
         "steps": 16},
        # The double-precision run that a mixed one is checked against, a quarter of the length and half the width.
        {"name": "stage2d_fp64", "kind": "stage", "precision": "fp64", "nz": 1024, "nx": 128, "ppc": 4, "order": 3,
         "gather": "energy", "strides": "", "theta": 0.1, "tile": "", "sort": 0, "warm": 60, "steps": 4},
        # The smallest 2D runs (double precision, Yee, one filter pass): convergence studies and regression runs,
        # where every launch counts.
        {"name": "small2d_fp64", "kind": "parity2", "precision": "fp64", "nz": 256, "nx": 64, "order": 3,
         "gather": "energy", "warm": 120, "steps": 20},
        # Eight runs of uneven size advanced together: a parameter scan in one process.
        {"name": "ensemble", "kind": "ensemble", "runs": 8, "warm": 64, "steps": 8},
        # Labelling of eight complete stage runs with their test beams (about a thousand steps each): how the
        # surrogate's training set is made.
        {"name": "labels", "kind": "labels", "runs": 8},
        # The 3D stage at full size (11.2 M electrons), with the damping that keeps the whole stage stable.
        {"name": "stage3d", "kind": "stage3", "precision": "mixed", "nz": 1024, "ny": 128, "nx": 128, "order": 3,
         "gather": "energy", "warm": 60, "steps": 3},
        # The smallest 3D runs, double precision.
        {"name": "small3d_fp64", "kind": "parity3", "precision": "fp64", "nz": 64, "ny": 24, "nx": 24, "order": 3,
         "gather": "energy", "warm": 40, "steps": 20},
        # The 1D stage in the lab frame with the moving window, mixed precision: twenty thousand steps of a grid that
        # fits in one multiprocessor.
        {"name": "window1d", "kind": "window1", "precision": "mixed", "nz": 952, "ppc": 10, "filtered": True,
         "warm": 1200, "steps": 200},
        # A boosted 1D run in double precision with damping, compensated filter and ions.
        {"name": "boost1d_fp64", "kind": "boost1", "precision": "fp64", "nz": 400, "ppc": 4, "order": 3,
         "gather": "energy", "warm": 200, "steps": 50},
        # A serving batch of the trained surrogate: a scan over stage parameters.
        {"name": "serve", "kind": "serve", "n": 100000},
        # Training the surrogate on 2048 labelled runs, four epochs of the default batch, at a fine-tuning rate.
        {"name": "train", "kind": "train", "n": 2048, "batch": 64, "epochs": 4},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["stage", "stage", "stage", "parity2", "ensemble", "labels", "stage3", "parity3", "window1",
                       "boost1", "serve", "serve", "train"])
    order = rng.choice([3, 3, 3, 1])
    gather = rng.choice(["energy", "energy", "energy", "momentum"])
    if kind == "stage":
        precision = rng.choice(["mixed", "mixed", "fp64"])
        strides = rng.choice(["", "", "", "1:2", "1:2:3", "1:2:4"])
        nx = rng.randint(150, 256) if strides else rng.randint(80, 256)
        nz = _log(rng, 256, 4096 if precision == "mixed" else 1024)
        return {"kind": kind, "precision": precision, "nz": nz, "nx": nx, "ppc": rng.randint(1, 4), "order": order,
                "gather": gather, "strides": strides, "theta": rng.choice([0.0, 0.1, 0.5]),
                "tile": rng.choice(["", "8x16", "16x16"]), "sort": rng.choice([0, 16, 64]), "warm": 64,
                "steps": rng.randint(3, 8)}
    if kind == "parity2":
        return {"kind": kind, "precision": rng.choice(["fp64", "mixed"]), "nz": rng.randint(200, 400),
                "nx": rng.randint(48, 96), "order": order, "gather": gather, "warm": 100, "steps": rng.randint(10, 25)}
    if kind == "ensemble":
        return {"kind": kind, "runs": rng.randint(2, 8), "warm": 48, "steps": rng.randint(3, 8)}
    if kind == "labels":
        return {"kind": kind, "runs": rng.randint(1, 8)}
    if kind == "stage3":
        return {"kind": kind, "precision": "mixed", "nz": _log(rng, 128, 1024), "ny": rng.randint(64, 128),
                "nx": rng.randint(64, 128), "order": order, "gather": gather, "warm": 48, "steps": rng.randint(2, 3)}
    if kind == "parity3":
        return {"kind": kind, "precision": rng.choice(["fp64", "mixed"]), "nz": rng.randint(60, 120),
                "ny": rng.randint(24, 40), "nx": rng.randint(24, 40), "order": order, "gather": gather, "warm": 40,
                "steps": rng.randint(5, 20)}
    if kind == "window1":
        return {"kind": kind, "precision": rng.choice(["mixed", "fp64"]), "nz": _log(rng, 500, 4000),
                "ppc": rng.randint(4, 12), "filtered": rng.random() < 0.7, "warm": 800, "steps": rng.randint(20, 100)}
    if kind == "boost1":
        return {"kind": kind, "precision": rng.choice(["fp64", "mixed"]), "nz": _log(rng, 300, 4000),
                "ppc": rng.randint(2, 8), "order": order, "gather": gather, "warm": 200, "steps": rng.randint(20, 50)}
    if kind == "serve":
        return {"kind": kind, "n": _log(rng, 1, 100000)}
    return {"kind": kind, "n": _log(rng, 256, 2048), "batch": rng.choice([16, 48, 64, 100, 128]),
            "epochs": rng.randint(2, 4)}


# ---------------------------------------------------------------------------------------------------------------------
# inputs: the repository's recipes with the pulse and the density moved by the seed

def _moved(w, r):
    la, pl = w["laser"], w["plasma"]
    la["a0"] *= r.uniform(0.9, 1.1)
    la["tau_fwhm"] *= r.uniform(0.95, 1.05)
    la["phase"] = r.uniform(0.0, 2.0 * math.pi)
    pl["n0"] *= r.uniform(0.9, 1.1)
    return w


def _driven(w):
    """The antenna starts close to the pulse's peak, so that a few dozen steps drive the plasma as the thousands of
    steps of a whole stage do (the boost slows the emission by (1 + beta) gamma)."""
    w["laser"]["t_peak"] = 0.25 * w["laser"]["tau_fwhm"]
    return w


def _dz(w):
    g = w["gamma_boost"]
    return (1.0 + math.sqrt(1.0 - 1.0 / g ** 2)) * g * w["dz_lab"]


def _workload(c, seed):
    r = np.random.default_rng(seed)
    k = c["kind"]
    if k == "stage":
        w = W.shrink(W.stage_2d(), c["nx"], c["nz"], theta=c["theta"], order=c["order"], gather=c["gather"],
                     precision=c["precision"], plasma={"ppc_x": c["ppc"], "ppc_z": c["ppc"]})
        dz = _dz(w)
        w["dt"] = dz / (math.sqrt(2.0) * C)       # the low-instability step
        if c["strides"]:
            # the four passes and their compensation at each stride; the antenna and the plasma's front move in past
            # the wider guard
            w["filter_strides"] = [int(v) for v in c["strides"].split(":")]
            w["filter_passes"], w["filter_compensate"] = 4, 1
            ant = w["pml_cells"] + 3 + 5 * sum(w["filter_strides"]) + 4
            w["laser"]["z_antenna"] = ant * dz
            w["plasma"]["z_start_lab"] = w["gamma_boost"] * (ant + 6) * dz
        return _moved(_driven(w), r)
    if k == "parity2":
        return _moved(W.shrink(W.parity_2d(), c["nx"], c["nz"], order=c["order"], gather=c["gather"],
                               precision=c["precision"]), r)
    if k == "stage3":
        return _moved(_driven(W.shrink3(W.stage_3d(), c["nx"], c["ny"], c["nz"], theta=0.5, order=c["order"],
                                        gather=c["gather"], precision=c["precision"])), r)
    if k == "parity3":
        return _moved(W.shrink3(W.parity_3d(), c["nx"], c["ny"], c["nz"], order=c["order"], gather=c["gather"],
                                precision=c["precision"]), r)
    if k == "window1":
        w = W.app1_lwfa(c["filtered"])
        dz = w["dz_lab"]
        w["nz"], w["precision"] = c["nz"], c["precision"]
        w["plasma"].update(ppc_z=c["ppc"], z_start_lab=(c["nz"] - 60) * dz, length_lab=0.0)
        w["laser"]["z_antenna"] = (c["nz"] - 80) * dz
        return _moved(w, r)
    w = W.parity_1d()
    w.update(nz=c["nz"], precision=c["precision"], order=c["order"], gather=c["gather"])
    w["plasma"]["ppc_z"] = c["ppc"]
    return _moved(w, r)


def _stage_runs(n, seed):
    """complete stage runs inside the recipe's stable range"""
    r = np.random.default_rng(seed)
    return [W.stage_run(r.uniform(23.8, 24.8), r.uniform(0.6, 1.4), r.uniform(9e-6, 18e-6), r.uniform(22e-15, 35e-15),
                        r.uniform(0.25e-3, 0.45e-3), r.uniform(4.2, 5.2), beam_seed=int(r.integers(1 << 30)),
                        name=f"label_{i}") for i in range(n)]


def _network(seed):
    """weights as a trained surrogate's: He-scaled layers and small biases, one flat vector"""
    r = np.random.default_rng(seed)
    p = []
    for a, b in zip(WIDTHS[:-1], WIDTHS[1:]):
        s = math.sqrt(6.0 / a) * (0.5 if b == WIDTHS[-1] else 1.0)
        p += [r.uniform(-s, s, b * a), r.uniform(-0.1, 0.1, b)]
    return np.concatenate(p).astype(np.float32)


def _queries(n, seed):
    """standardised stage parameters (uniform over the recipe's box) and smooth targets with a little scatter"""
    r = np.random.default_rng(seed + 1)
    x = r.uniform(-1.7, 1.7, (n, WIDTHS[0])).astype(np.float32)
    t = np.stack([np.sin(x[:, 0] + 0.5 * x[:, 1]), np.tanh(x[:, 1] * x[:, 4]), 0.3 * x[:, 2] + 0.1 * x[:, 3] ** 2,
                  np.cos(x[:, 5]) * x[:, 4]], 1) + 0.02 * r.standard_normal((n, WIDTHS[-1]))
    return x, t.astype(np.float32)


def prepare(case, seed):
    k = case["kind"]
    if k in ("serve", "train"):
        net = MLP(WIDTHS)
        net.set_params(_network(seed))
        x, t = _queries(case["n"], seed)
        if k == "train":
            return {"case": case, "net": net, "x": x, "t": t}
        xd = torch.as_tensor(x).cuda()
        return {"case": case, "net": net, "x": xd, "y": torch.empty((case["n"], WIDTHS[-1]), device="cuda")}
    if k == "labels":
        return {"case": case, "runs": _stage_runs(case["runs"], seed)}
    if k == "ensemble":
        # the recipe's runs, their pulses and densities moved by the seed (their sizes are the recipe's)
        r = np.random.default_rng(seed)
        sim = Ensemble([_moved(_driven(w), r) for w in W.ensemble_2d(case["runs"])])
    else:
        tile = tuple(int(v) for v in case["tile"].split("x")) if case.get("tile") else None
        sim = Simulation(_workload(case, seed), tile=tile, sort_every=case.get("sort", 0))
    sim.step(case["warm"])
    sim.sync()
    return {"case": case, "sim": sim}


def _stats(sim):
    s = sim.stats()
    return np.array([s["n_electrons"], s["field_energy"]], dtype=np.float32)


def run(state):
    case = state["case"]
    k = case["kind"]
    if k == "serve":
        state["net"].forward_device(state["x"].data_ptr(), case["n"], state["y"].data_ptr())
        return state["y"]
    if k == "train":
        curve = state["net"].train(state["x"], state["t"], case["epochs"], case["batch"], lr=2e-5)
        return {"curve": curve, "params": state["net"].get_params()}
    if k == "labels":
        _, labels, valid = stage_labels(state["runs"])
        return {"labels": labels.astype(np.float32), "valid": valid}
    sim = state["sim"]
    sim.step(case["steps"])
    if k == "ensemble":
        sim.sync()
        return {"stats": [_stats(m) for m in sim.members],
                "fields": [m.field_device(c).float() for m in sim.members for c in (0, 1, 2)]}
    # the mixed path's fields are FP32
    mixed = case["precision"] == "mixed"
    fields = [sim.field_device(c) for c in range(6)]
    return {"stats": _stats(sim), "fields": [f.float() for f in fields] if mixed else fields}


# ---------------------------------------------------------------------------------------------------------------------
# what a pass cannot do without

def _step_work(dim, nodes, electrons, fp64, order):
    """bytes and operations of one step: every particle read and written once (positions, momenta, weight, id; the
    weight and id are only read), the fields' 21 values a node (E, the two Friedman histories and B read, E, B and one
    history written); gather, push and deposit"""
    b = 8 if fp64 else 4
    per = (dim + 3 + 1) * b + 4 + (dim + 3) * b
    ns = order + 1
    gather = 6 * 2 * sum(ns ** d for d in range(1, dim + 1))
    deposit = 3 * 2 * (ns + 1) ** dim
    return {"bytes": electrons * per + nodes * 21 * b, "flops": electrons * (gather + deposit + 120) + nodes * 120}


def _domain(n, pml, guard):
    return max(n - 2 * (pml + guard), 2)


def work(case):
    k = case["kind"]
    macs = sum(a * b for a, b in zip(WIDTHS[:-1], WIDTHS[1:]))
    npar = macs + sum(WIDTHS[1:])
    if k == "serve":
        return {"bytes": case["n"] * 4 * (WIDTHS[0] + WIDTHS[-1]) + 2 * macs, "flops": 2 * macs * case["n"]}
    if k == "train":
        steps = case["epochs"] * (case["n"] // case["batch"])
        # the weights and their two moments stay on the chip between steps; data and final state move once
        return {"bytes": case["n"] * 40 + 12 * npar, "flops": steps * (6 * macs * case["batch"] + 12 * npar)}
    if k in ("ensemble", "labels"):
        ws = W.ensemble_2d(case["runs"]) if k == "ensemble" else _stage_runs(case["runs"], 0)
        out = {"bytes": 0, "flops": 0}
        for w in ws:
            el = _domain(w["nx"], 16, 10) * w["plasma"]["ppc_x"] * w["plasma"]["ppc_z"]
            # a labelled run holds a plasma of finite length
            el *= _domain(w["nz"], 16, 10) if k == "ensemble" else min(
                w["plasma"]["length_lab"] / w["gamma_boost"] / _dz(w), w["nz"]) * 0.5
            s = _step_work(2, (w["nx"] + 1) * (w["nz"] + 1), el, False, 3)
            n = case["steps"] if k == "ensemble" else w["steps"]
            out = {q: out[q] + n * s[q] for q in out}
        return out
    fp64 = case["precision"] == "fp64"
    order = case.get("order", 3)
    if k in ("stage", "parity2"):
        h = 5 * sum(int(v) for v in case["strides"].split(":")) if case.get("strides") else 5 if k == "stage" else 1
        pml, ppc = (16, case["ppc"]) if k == "stage" else (8, 2)
        guard = order // 2 + 4 + h
        el = _domain(case["nx"], pml, guard) * _domain(case["nz"], pml, guard) * ppc * ppc
        dim, nodes = 2, (case["nx"] + 1) * (case["nz"] + 1)
    elif k in ("stage3", "parity3"):
        pml, guard = (16, order // 2 + 9) if k == "stage3" else (4, order // 2 + 5)
        el = 2 * _domain(case["nx"], pml, guard) * _domain(case["ny"], pml, guard) * _domain(case["nz"], pml, guard)
        dim, nodes = 3, (case["nx"] + 1) * (case["ny"] + 1) * (case["nz"] + 1)
    else:
        el, dim, nodes = case["nz"] * case["ppc"], 1, case["nz"] + 1
    s = _step_work(dim, nodes, el, fp64, order)
    return {"bytes": case["steps"] * s["bytes"] + 6 * 8 * nodes, "flops": case["steps"] * s["flops"]}


# ---------------------------------------------------------------------------------------------------------------------
# the network in 64 bits

def _layers(p):
    out, o = [], 0
    for a, b in zip(WIDTHS[:-1], WIDTHS[1:]):
        out.append((p[o:o + a * b].reshape(b, a), p[o + a * b:o + a * b + b]))
        o += a * b + b
    return out


def _gelu(z):
    return 0.5 * z * (1.0 + torch.erf(z / math.sqrt(2.0)))


def _splitmix(state):
    m = (1 << 64) - 1
    state = (state + 0x9e3779b97f4a7c15) & m
    z = ((state ^ (state >> 30)) * 0xbf58476d1ce4e5b9) & m
    z = ((z ^ (z >> 27)) * 0x94d049bb133111eb) & m
    return state, z ^ (z >> 31)


def exact(case, seed):
    """The network's outputs and its trained parameters in 64 bits. The runs have none here: a step of the whole method
    in 64 bits is a second PIC code (the test oracle is one), over twenty seconds for most of these boxes."""
    if case["kind"] not in ("serve", "train"):
        return None
    p = torch.as_tensor(_network(seed)).double()
    x, t = (torch.as_tensor(v).double() for v in _queries(case["n"], seed))
    if case["kind"] == "serve":
        h = x
        for i, (w, b) in enumerate(_layers(p)):
            h = h @ w.T + b
            if i + 2 < len(WIDTHS):
                h = _gelu(h)
        return h
    # AdamW over shuffled minibatches, as the entry point documents them
    m, v, s, step = torch.zeros_like(p), torch.zeros_like(p), 0, 0
    lr, wd, b1, b2, eps = 2e-5, 1e-4, 0.9, 0.999, 1e-8
    curve, nb = [], case["n"] // case["batch"]
    for _ in range(case["epochs"]):
        perm = list(range(case["n"]))
        for i in range(case["n"] - 1, 0, -1):
            s, z = _splitmix(s)
            j = z % (i + 1)
            perm[i], perm[j] = perm[j], perm[i]
        total = 0.0
        for k in range(nb):
            rows = torch.tensor(perm[k * case["batch"]:(k + 1) * case["batch"]])
            q = p.clone().requires_grad_(True)
            h = x[rows]
            for i, (w, b) in enumerate(_layers(q)):
                h = h @ w.T + b
                if i + 2 < len(WIDTHS):
                    h = _gelu(h)
            loss = ((h - t[rows]) ** 2).mean()
            loss.backward()
            g = q.grad
            step += 1
            m = b1 * m + (1 - b1) * g
            v = b2 * v + (1 - b2) * g * g
            p = p - lr * ((m / (1 - b1 ** step)) / ((v / (1 - b2 ** step)).sqrt() + eps) + wd * p)
            total += loss.item()
        curve.append(total / nb)
    return {"curve": np.array(curve), "params": p.numpy()}
