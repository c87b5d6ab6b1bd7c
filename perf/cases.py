"""The workloads this framework is timed on: what they are, their inputs, one
pass of each through the public entry points, and the work a pass cannot do
without.

A case's "path" says which call a user makes:
  anneal    qp_anneal_ex of a field's path QUBO, then qp_decode_batch of the
            final states (one solver call of a mission planner).  "begin" > 0
            or "end" < sweeps: a segment of the schedule resumed from the
            states the segment before it returned.
  dense     the same with the dense form (every term of S explicit).
  batch     qp_batch_run: many uneven fields in one launch.
  exchange  qp_anneal_pt: replica exchange over a temperature ladder.
  repair    qp_repair_batch with 2-opt of a finished anneal's states.
  forward   qp_ws_forward: step logits of many cells.
  train     qp_ws_train_step over some mini-batches, then the parameters (the
            end of an epoch).
  seed      warmstart.device_seed: one warm-start seed per field.
"""
import math

import numpy as np
import torch

from paper_2608_25376_gb300 import inputs, qpath, warmstart

# integer operations of one flip attempt: neighbour sum, the two one-hot
# terms, their products with the weights, the sign and the two compares
ATTEMPT_OPS = 17
PARAMS = (256 * 16 + 256) + 3 * (256 * 256 + 256)


def listed():
    return [
        # a small plot (the paper's largest grid): one call of a few milliseconds, all latency
        dict(name="anneal_6x6", path="anneal", rows=6, cols=6, obstacles=0.0, replicas=64, sweeps=500, begin=0,
             end=500, t0=1000.0, scale=100, skip=False),
        # the 10x10 workload of the benchmark, whole
        dict(name="anneal_10x10", path="anneal", rows=10, cols=10, obstacles=0.10, replicas=1024, sweeps=5000,
             begin=0, end=5000, t0=1000.0, scale=100, skip=False),
        # one checkpoint segment of the warm-start comparison on a 16x16 field, resumed from states
        dict(name="segment_16x16", path="anneal", rows=16, cols=16, obstacles=0.10, replicas=1024, sweeps=2000,
             begin=400, end=500, t0=1000.0, scale=100, skip=False),
        # the headline field and replica count, on a schedule of 1000 sweeps
        dict(name="anneal_24x24", path="anneal", rows=24, cols=24, obstacles=0.15, replicas=4096, sweeps=1000,
             begin=0, end=1000, t0=1000.0, scale=100, skip=False),
        # a field beyond 512 cells
        dict(name="anneal_31x32", path="anneal", rows=31, cols=32, obstacles=0.10, replicas=512, sweeps=40,
             begin=0, end=40, t0=1000.0, scale=100, skip=False),
        # the dense form of the 10x10 field
        dict(name="dense_10x10", path="dense", rows=10, cols=10, obstacles=0.10, replicas=1024, sweeps=1000,
             t0=1000.0),
        # uneven fields of 4..16 cells a side with irregular boundaries, one launch
        dict(name="batch_256", path="batch", fields=256, shapes=2026, replicas=32, sweeps=500),
        # replica exchange on the 10x10 field, the ladder of the benchmark
        dict(name="exchange_10x10", path="exchange", rows=10, cols=10, obstacles=0.10, groups=32, levels=32,
             every=25, rounds=20),
        # every final state of a 24x24 anneal made a flight path, 2-opt until no move helps
        dict(name="repair_24x24", path="repair", rows=24, cols=24, obstacles=0.15, replicas=1024, sweeps=200,
             passes=-1),
        # logits of the cells of a hundred fields
        dict(name="forward_16384", path="forward", cells=16384),
        # four mini-batches of 64 fields of 8..16 cells a side
        dict(name="train_64_fields", path="train", steps=4, fields=64, shapes=1000),
        # the warm-start seeds of eight held-out 16x16 fields, one call each
        dict(name="seed_16x16", path="seed", rows=16, cols=16, obstacles=0.10, fields=8),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    path = rng.choice(["anneal", "anneal", "anneal", "anneal", "segment", "segment", "dense", "batch", "exchange",
                       "repair", "forward", "train", "seed"])
    p = round(rng.uniform(0.0, 0.2), 3)
    if path in ("anneal", "segment"):
        side = rng.uniform(math.log(3.0), math.log(34.0))
        rows = max(3, min(34, int(round(math.exp(side + rng.uniform(-0.15, 0.15))))))
        cols = max(3, min(34, int(round(math.exp(side + rng.uniform(-0.15, 0.15))))))
        C = cells(dict(rows=rows, cols=cols, obstacles=p))
        replicas = _log_int(rng, 1, 4096)
        budget = 6.0e10 if C <= 512 else 1.5e9  # flip attempts
        most = int(max(8, min(4000, budget / (replicas * (C - 1.0) ** 2), 4.0e5 / C)))
        sweeps = _log_int(rng, 8, most)
        case = dict(path="anneal", rows=rows, cols=cols, obstacles=p, replicas=replicas, sweeps=sweeps, begin=0,
                    end=sweeps, t0=rng.choice([1000.0, 1000.0, 300.0]), scale=rng.choice([100, 100, 100, 1000]),
                    skip=rng.random() < 0.2)
        if path == "segment":
            case["begin"] = rng.randrange(0, sweeps)
            case["end"] = rng.randrange(case["begin"] + 1, sweeps + 1)
        return case
    if path == "dense":
        return dict(path="dense", rows=rng.randrange(3, 12), cols=rng.randrange(3, 12), obstacles=p,
                    replicas=_log_int(rng, 16, 1024), sweeps=_log_int(rng, 50, 500), t0=1000.0)
    if path == "batch":
        return dict(path="batch", fields=_log_int(rng, 8, 256), shapes=rng.randrange(1, 10000),
                    replicas=_log_int(rng, 4, 64), sweeps=_log_int(rng, 50, 400))
    if path == "exchange":
        return dict(path="exchange", rows=rng.randrange(4, 15), cols=rng.randrange(4, 15), obstacles=p,
                    groups=_log_int(rng, 2, 32), levels=rng.randrange(4, 33), every=rng.randrange(5, 26),
                    rounds=rng.randrange(4, 17))
    if path == "repair":
        return dict(path="repair", rows=rng.randrange(6, 25), cols=rng.randrange(6, 25), obstacles=p,
                    replicas=_log_int(rng, 1, 1024), sweeps=rng.randrange(50, 201), passes=rng.choice([0, 1, -1, -1]))
    if path == "forward":
        return dict(path="forward", cells=_log_int(rng, 9, 16384))
    if path == "train":
        return dict(path="train", steps=rng.randrange(1, 5), fields=_log_int(rng, 4, 64),
                    shapes=rng.randrange(1, 10000))
    return dict(path="seed", rows=rng.randrange(4, 17), cols=rng.randrange(4, 17), obstacles=p,
                fields=rng.randrange(1, 9))


def cells(case):
    """Free cells of the case's field: the obstacles are a fixed count, their places come from the seed."""
    grid = case["rows"] * case["cols"]
    return max(2, grid - int(round(case["obstacles"] * grid)))


def _field(case, seed):
    """A rows x cols field with the case's number of obstacles at places drawn from the seed, start at a free cell
    of the first row that has one."""
    rng = np.random.Generator(np.random.PCG64(seed))
    grid = case["rows"] * case["cols"]
    mask = np.ones(grid, np.uint8)
    mask[rng.permutation(grid)[:grid - cells(case)]] = 0
    return inputs.Field(case["rows"], case["cols"], mask, int(np.flatnonzero(mask)[0]))


def _chains(replicas, C):
    """Output buffers of an anneal and of its decode."""
    return dict(states=torch.zeros((replicas, C * C), dtype=torch.uint8, device="cuda"),
                energies=torch.zeros(replicas, dtype=torch.int64, device="cuda"),
                best=torch.zeros(replicas, dtype=torch.int64, device="cuda"),
                paths=torch.zeros((replicas, C), dtype=torch.int32, device="cuda"),
                lengths=torch.zeros(replicas, dtype=torch.int64, device="cuda"))


def _serpentine(field):
    """Each free cell's step in the row-by-row sweep of the field that turns at the row ends."""
    grid = np.arange(field.rows * field.cols).reshape(field.rows, field.cols)
    grid[1::2] = grid[1::2, ::-1].copy()
    free = np.asarray(field.free_mask, np.uint8).reshape(-1) != 0
    order = grid.reshape(-1)[free[grid.reshape(-1)]]
    ident = np.cumsum(free) - 1
    steps = np.empty(int(free.sum()), np.int32)
    steps[ident[order]] = np.arange(steps.size, dtype=np.int32)
    return steps


def _params(rng):
    """He-uniform weights and small biases in the flat parameter layout."""
    out = []
    for fan_in in (16, 256, 256, 256):
        lim = math.sqrt(6.0 / fan_in)
        out += [rng.uniform(-lim, lim, 256 * fan_in), rng.uniform(-0.05, 0.05, 256)]
    return np.concatenate(out).astype(np.float32)


def _features(cell_count, rng):
    """Features of `cell_count` cells: whole fields of 8..16 cells a side, the last one cut."""
    parts, have = [], 0
    while have < cell_count:
        for f in inputs.fields_8_16(16, seed=int(rng.integers(1 << 30))):
            parts.append(qpath.qp_ws_features(f))
            have += len(parts[-1])
            if have >= cell_count:
                break
    return np.ascontiguousarray(np.concatenate(parts)[:cell_count])


def _batches(case, seed):
    """The mini-batches of a training case: features, labels and each cell's number of steps.  The fields' shapes are
    the case's; which fields share a batch comes from the seed."""
    fields = inputs.fields_8_16(case["steps"] * case["fields"], seed=case["shapes"])
    order = np.random.Generator(np.random.PCG64(seed)).permutation(len(fields))
    out = []
    for k in range(case["steps"]):
        part = [fields[i] for i in order[k * case["fields"]:(k + 1) * case["fields"]]]
        labels = [_serpentine(f) for f in part]
        out.append((np.concatenate([qpath.qp_ws_features(f) for f in part]), np.concatenate(labels),
                    np.concatenate([np.full(y.size, y.size, np.int32) for y in labels])))
    return out


def prepare(case, seed):
    path = case["path"]
    rng = np.random.Generator(np.random.PCG64([seed, 77]))
    s = dict(case=case, seed=seed)
    if path in ("anneal", "dense"):
        C, R = cells(case), case["replicas"]
        flags = qpath.QP_DENSE if path == "dense" else qpath.QP_STRUCTURED
        s.update(handle=qpath.qp_build_qubo(_field(case, seed), scale=case.get("scale", 100), flags=flags),
                 out=_chains(R, C), init=None,
                 schedule=qpath.schedule(case["sweeps"], case["t0"], 1.0, case.get("begin", 0),
                                         case.get("end", case["sweeps"])))
        if s["schedule"].sweep_begin > 0:  # the states the segment before this one returned
            s["init"] = torch.zeros((R, C * C), dtype=torch.uint8, device="cuda")
            before = qpath.schedule(case["sweeps"], case["t0"], 1.0, 0, s["schedule"].sweep_begin)
            qpath.qp_anneal_ex(s["handle"], R, before, seed, None, s["init"], s["out"]["energies"],
                               stream=torch.cuda.current_stream())
    elif path == "batch":
        fields = inputs.batch(case["fields"], case["shapes"])
        R = case["replicas"]
        hs = [qpath.qp_build_qubo(f) for f in fields]
        states = [torch.zeros((R, f.n_cells ** 2), dtype=torch.uint8, device="cuda") for f in fields]
        energies = torch.zeros((len(fields), R), dtype=torch.int64, device="cuda")
        best = torch.zeros((len(fields), R), dtype=torch.int64, device="cuda")
        s.update(states=states, energies=energies, best=best,
                 batch=qpath.qp_batch_create(hs, R, qpath.schedule(case["sweeps"]), seed, states, list(energies),
                                             list(best)))
    elif path == "exchange":
        C, R = cells(case), case["groups"] * case["levels"]
        s.update(handle=qpath.qp_build_qubo(_field(case, seed)), out=_chains(R, C),
                 schedule=qpath.pt_schedule(case["levels"], 2.0, 1000.0, case["every"], case["rounds"]),
                 levels=torch.zeros(R, dtype=torch.int32, device="cuda"),
                 swaps=torch.zeros(case["groups"] * (case["levels"] - 1), dtype=torch.int64, device="cuda"))
    elif path == "repair":
        C, R = cells(case), case["replicas"]
        s.update(handle=qpath.qp_build_qubo(_field(case, seed)), out=_chains(R, C),
                 status=torch.zeros(R, dtype=torch.int32, device="cuda"))
        qpath.qp_anneal_ex(s["handle"], R, qpath.schedule(case["sweeps"]), seed, None, s["out"]["states"],
                           s["out"]["energies"], stream=torch.cuda.current_stream())
    elif path == "forward":
        s.update(model=qpath.WarmStartModel(), feats=_features(case["cells"], rng),
                 logits=torch.zeros((case["cells"], qpath.WS_STEPS), dtype=torch.float32, device="cuda"))
        qpath.qp_ws_set_params(s["model"], _params(rng))
    elif path == "train":
        s.update(model=qpath.WarmStartModel(), batches=_batches(case, seed))
        qpath.qp_ws_set_params(s["model"], _params(rng))
    else:
        fields = [_field(case, int(rng.integers(1 << 30))) for _ in range(case["fields"])]
        s.update(model=qpath.WarmStartModel(), fields=fields, handles=[qpath.qp_build_qubo(f) for f in fields])
        qpath.qp_ws_set_params(s["model"], _params(rng))
    return s


def run(s):
    case = s["case"]
    path = case["path"]
    stream = torch.cuda.current_stream()
    if path in ("anneal", "dense"):
        o = s["out"]
        qpath.qp_anneal_ex(s["handle"], case["replicas"], s["schedule"], s["seed"], s["init"], o["states"],
                           o["energies"], o["best"], stream=stream,
                           flags=qpath.QP_ANNEAL_SKIP_SETTLED if case.get("skip") else 0)
        qpath.qp_decode_batch(s["handle"], case["replicas"], o["states"], o["paths"], o["lengths"], stream=stream)
        return o
    if path == "batch":
        s["batch"].run(stream)
        return dict(states=torch.cat([x.reshape(-1) for x in s["states"]]), energies=s["energies"], best=s["best"])
    if path == "exchange":
        o = s["out"]
        qpath.qp_anneal_pt(s["handle"], case["groups"], s["schedule"], s["seed"], None, o["states"], o["energies"],
                           o["best"], s["levels"], s["swaps"], stream=stream)
        return dict(states=o["states"], energies=o["energies"], best=o["best"], levels=s["levels"], swaps=s["swaps"])
    if path == "repair":
        o = s["out"]
        qpath.qp_repair_batch(s["handle"], case["replicas"], o["states"], case["passes"], o["paths"], o["lengths"],
                              s["status"], stream=stream)
        return dict(paths=o["paths"], lengths=o["lengths"], status=s["status"])
    if path == "forward":
        return qpath.qp_ws_forward(s["model"], s["feats"], s["logits"], stream=stream)
    if path == "train":
        losses = [qpath.qp_ws_train_step(s["model"], x, y, t, 1e-3, stream=stream) for x, y, t in s["batches"]]
        return dict(losses=np.array(losses), params=qpath.qp_ws_get_params(s["model"]))
    seeds = [warmstart.device_seed(h, f, s["model"], stream=stream) for h, f in zip(s["handles"], s["fields"])]
    return dict(states=torch.stack([a for a, _ in seeds]), lengths=np.array([b for _, b in seeds]))


def work(case):
    path = case["path"]
    if path == "forward":
        M = case["cells"]
        return {"bytes": M * (16 * 4 + 256 * 4) + PARAMS * 2, "flops": 2 * M * (16 * 256 + 3 * 256 * 256)}
    if path == "train":
        M = sum(f.n_cells for f in inputs.fields_8_16(case["steps"] * case["fields"], seed=case["shapes"]))
        # forward, input gradients (not of the first layer) and weight gradients; per step the parameters and the two
        # moments are read and written
        return {"bytes": M * (16 * 4 + 8) + case["steps"] * PARAMS * 4 * 6,
                "flops": 2 * M * (2 * 16 * 256 + 9 * 256 * 256)}
    if path == "seed":
        C, n = cells(case), case["fields"]
        return {"bytes": n * (C * 16 * 4 + C * C * 5) + PARAMS * 2,
                "flops": n * (2 * C * (16 * 256 + 3 * 256 * 256) + 4 * C * C)}
    if path == "batch":
        cs = [f.n_cells for f in inputs.batch(case["fields"], case["shapes"])]
        return {"bytes": sum(2 * c * c + case["replicas"] * (c * c + 16) for c in cs),
                "flops": ATTEMPT_OPS * case["replicas"] * case["sweeps"] * sum((c - 1) ** 2 for c in cs)}
    C = cells(case)
    if path == "repair":
        R = case["replicas"]
        # the states, the distances and the paths; one scan of the 2-opt moves of every path
        return {"bytes": R * (C * C + 4 * C + 12) + 4 * C * C, "flops": R * (C * C + 4 * C * C // 2)}
    R = case["groups"] * case["levels"] if path == "exchange" else case["replicas"]
    sweeps = (case["every"] * case["rounds"] if path == "exchange"
              else case.get("end", case["sweeps"]) - case.get("begin", 0))
    states = R * C * C * (2 if case.get("begin") else 1)
    form = (2 * C ** 4 if path == "dense" else 2 * C * C)
    return {"bytes": states + form + R * (16 + 4 * C + 8), "flops": ATTEMPT_OPS * R * sweeps * (C - 1) ** 2}


def _network64(params, x):
    """Activations of the four layers in 64 bits; the parameters are the fp32 ones."""
    h, at, layers = [torch.from_numpy(np.asarray(x, np.float64))], 0, []
    for k, fan_in in enumerate((16, 256, 256, 256)):
        w = torch.from_numpy(np.asarray(params[at:at + 256 * fan_in], np.float64)).reshape(256, fan_in)
        b = torch.from_numpy(np.asarray(params[at + 256 * fan_in:at + 256 * fan_in + 256], np.float64))
        at += 256 * fan_in + 256
        z = h[-1] @ w.T + b
        h.append(torch.relu(z) if k < 3 else z)
        layers.append(w)
    return h, layers


def exact(case, seed):
    path = case["path"]
    rng = np.random.Generator(np.random.PCG64([seed, 77]))
    if path == "forward":
        x = _features(case["cells"], rng)
        return _network64(_params(rng), x)[0][-1]
    if path != "train":
        return None  # whole numbers
    batches = _batches(case, seed)
    params = torch.from_numpy(_params(rng).astype(np.float64))
    m, v = torch.zeros_like(params), torch.zeros_like(params)
    losses = []
    for k, (x, y, t) in enumerate(batches, 1):
        h, layers = _network64(params.numpy(), x)
        M = x.shape[0]
        valid = torch.arange(256)[None, :] < torch.from_numpy(t.astype(np.int64))[:, None]
        logp = torch.log_softmax(h[-1].masked_fill(~valid, -math.inf), dim=1)
        label = torch.from_numpy(y.astype(np.int64))[:, None]
        losses.append(float(-logp.gather(1, label).mean()))
        dz = logp.exp()
        dz.scatter_add_(1, label, torch.full((M, 1), -1.0, dtype=torch.float64))
        dz /= M
        grads = []
        for layer in (3, 2, 1, 0):
            grads += [dz.sum(0), (dz.T @ h[layer]).reshape(-1)]
            if layer:
                dz = (dz @ layers[layer]) * (h[layer] > 0)
        g = torch.cat(grads[::-1])
        m = 0.9 * m + 0.1 * g
        v = 0.999 * v + 0.001 * g * g
        params = params - 1e-3 * (m / (1 - 0.9 ** k)) / ((v / (1 - 0.999 ** k)).sqrt() + 1e-8)
    return dict(losses=np.array(losses), params=params)
