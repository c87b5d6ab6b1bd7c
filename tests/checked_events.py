"""Cases of the event-driven sweep, the repair, the walk and the decode for the
checked build of the library.  The sweep: every place its distances can be read from (matrix in shared memory, table of grid
differences, matrix in global memory), both distance types, row lengths that
fill the padded row and that do not, rows of one and of several blocks, states
from nothing and from many cells, single fields and batches.  The others: with
and without a distance table, states that are no paths.  Each is compared with
the CPU reference, then the library's record of failed checks must be empty:
no index outside its array, and no distance from an entry that nothing wrote.
Run by tests/test_gpu_device_checks_events.py in a fresh interpreter with
QPATH_LIBRARY pointing at the checked library; prints one JSON line and exits
non-zero on any mismatch."""
import json
import os
import sys

import numpy as np

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
sys.path.insert(0, ROOT)

import torch  # noqa: E402

import oracle  # noqa: E402
from oracle import mlp_ref, repair_ref  # noqa: E402
from paper_2608_25376_gb300 import inputs, qpath  # noqa: E402


def strip(rows, cols, cells, seed=3):
    """A rows x cols grid with the given number of free cells, mostly not at its corners."""
    rng = np.random.default_rng(seed)
    order = [g for g in rng.permutation(rows * cols) if g not in (0, rows * cols - 1)]
    m = np.zeros(rows * cols, np.uint8)
    m[order[:cells]] = 1
    return inputs.Field(rows, cols, m, int(np.flatnonzero(m)[cells // 2]))


def cross(n):
    """The middle row and column of an n x n grid: no cell near a corner."""
    m = np.zeros((n, n), np.uint8)
    m[n // 2, :] = m[:, n // 2] = 1
    return inputs.Field(n, n, m.reshape(-1), n // 2)


# name: field, scale, A (0: the default), sweeps, replicas, T0, T1, density of the initial state
SINGLE = {
    "matrix-i16-8x8": (inputs.rect(8, 8), 100, 0, 40, 6, 1000.0, 1.0, None),
    "matrix-i16-67": (strip(9, 9, 67), 100, 0, 30, 5, 1500.0, 300.0, 0.04),
    "matrix-i32-8x8": (inputs.rect(8, 8), 30000, 0, 40, 6, 3e5, 300.0, None),
    "matrix-i32-61": (strip(8, 8, 61), 30000, 0, 30, 5, 4e5, 300.0, 0.3),
    "matrix-i16-136": (strip(12, 12, 136), 100, 0, 12, 4, 1500.0, 50.0, 0.02),
    "table-i16-18x18": (inputs.rect(18, 18), 100, 0, 6, 3, 1500.0, 50.0, None),
    "table-i16-257": (strip(18, 18, 257), 100, 0, 6, 3, 2000.0, 300.0, 0.01),
    "table-i32-112": (strip(14, 14, 112), 4000, 0, 12, 4, 60000.0, 200.0, 0.05),
    "table-i32-320": (strip(19, 19, 320), 3000, 0, 5, 3, 60000.0, 200.0, 0.005),
    "global-i16-304": (inputs.rect(1, 304, start=7), 100, 900, 5, 3, 2500.0, 100.0, 0.01),
    "global-i32-304": (inputs.rect(1, 304, start=7), 3000, 9000, 5, 3, 40000.0, 2000.0, 0.01),
    "global-i32-290": (inputs.rect(1, 290, start=7), 3000, 9000, 5, 3, 40000.0, 2000.0, None),
    "global-i32-120": (strip(1, 300, 120), 3000, 9000, 8, 4, 40000.0, 2000.0, 0.05),
    # |dE| fits int32 with the distances of its cells, not with those to the corner of its bounding box
    "corner-i32-109": (cross(55), 170000, 100000, 5, 4, 1e5, 5e4, 0.05),
    "table-i32-109": (cross(55), 17000, 10000, 5, 4, 1e5, 5e4, 0.05),
}
# fields, replicas, sweeps, replicas per CTA
BATCH = {
    "small": ([inputs.rect(8, 8), strip(9, 9, 67), inputs.rect(4, 4)], 6, 24, 4),
    "wide": ([strip(18, 18, 257), inputs.rect(8, 8), strip(12, 12, 136)], 4, 5, 4),
}


def singles(results):
    for name, (f, scale, A, S, R, T0, T1, density) in SINGLE.items():
        P = oracle.Problem(f.rows, f.cols, f.free_mask, f.start, A=A or None, scale=scale)
        init = None
        if density is not None:
            init = (np.random.default_rng(5).random((R, P.n)) < density).astype(np.uint8)
        ref = oracle.anneal_structured(P, R, S, T0=T0, T1=T1, seed=11, init_states=init)
        st = torch.zeros((R, P.n), dtype=torch.uint8, device="cuda")
        E, B = (torch.zeros(R, dtype=torch.int64, device="cuda") for _ in range(2))
        qpath.qp_anneal_ex(qpath.qp_build_qubo(f, A=A, scale=scale), R, qpath.schedule(S, T0, T1), 11,
                           None if init is None else torch.from_numpy(init).cuda(), st, E, B,
                           stream=torch.cuda.current_stream())
        torch.cuda.synchronize()
        results[name] = bool((st.cpu().numpy() == ref.states).all() and (E.cpu().numpy() == ref.energies).all()
                             and (B.cpu().numpy() == ref.best).all())


def batches(results):
    for name, (fs, R, S, W) in BATCH.items():
        refs = []
        for i, f in enumerate(fs):
            P = oracle.Problem(f.rows, f.cols, f.free_mask, f.start)
            refs.append(oracle.anneal_structured(P, R, S, seed=5 + i))
        hs = [qpath.qp_build_qubo(f) for f in fs]
        for flags in (0, qpath.QP_BATCH_D_SHARED):
            try:
                sts = [torch.zeros((R, h.info["n"]), dtype=torch.uint8, device="cuda") for h in hs]
                Es = [torch.zeros(R, dtype=torch.int64, device="cuda") for _ in hs]
                b = qpath.qp_batch_create(hs, R, qpath.schedule(S), 5, sts, Es, replicas_per_cta=W, flags=flags)
            except qpath.QpError as e:
                results[f"batch-{name}-{flags}"] = f"{e}"
                continue
            b.run(torch.cuda.current_stream())
            torch.cuda.synchronize()
            results[f"batch-{name}-{flags}"] = all(
                bool((s.cpu().numpy() == r.states).all() and (e.cpu().numpy() == r.energies).all())
                for s, e, r in zip(sts, Es, refs))


# Field and scale of the repair, the walk and the decode; "none": too wide for a distance table.
PATHS = {
    "2": (inputs.rect(1, 2), 100), "33": (strip(7, 7, 33), 100), "64-i32": (strip(9, 9, 64), 20000),
    "129": (strip(12, 13, 129), 100), "none-90": (strip(1, 300, 90), 100), "300": (strip(18, 18, 300), 100),
    "513": (strip(24, 24, 513), 100),
}


def paths(results):
    stream = torch.cuda.current_stream()
    for name, (f, scale) in PATHS.items():
        h = qpath.qp_build_qubo(f, scale=scale)
        C = h.info["C"]
        d = qpath.qp_export_dist(h)
        start = int(np.cumsum(f.free_mask)[f.start] - 1)
        rng = np.random.default_rng(C)
        # a path, one with a few cells flipped, random cells, no cell
        X = np.zeros((4, C, C), np.uint8)
        X[:2, np.arange(C), np.r_[start, rng.permutation([i for i in range(C) if i != start])].astype(int)] = 1
        X[1] ^= (rng.random((C, C)) < 1.0 / C).astype(np.uint8)
        X[2] = rng.random((C, C)) < 3.0 / C
        st = torch.from_numpy(X.reshape(4, -1)).cuda()
        p = torch.zeros((4, C), dtype=torch.int32, device="cuda")
        n = torch.zeros(4, dtype=torch.int64, device="cuda")
        s = torch.zeros(4, dtype=torch.int32, device="cuda")
        qpath.qp_decode_batch(h, 4, st, p, n, stream=stream)
        torch.cuda.synchronize()
        on = X != 0
        cells = np.where(on.any(2), C - 1 - on[:, :, ::-1].argmax(2), -1)
        ok = (on.sum(1) == 1).all(1) & (on.sum(2) == 1).all(1)
        lengths = np.where(ok, d[cells[:, :-1], cells[:, 1:]].astype(np.int64).sum(1), -1)
        results[f"decode-{name}"] = bool((p.cpu().numpy() == cells).all() and (n.cpu().numpy() == lengths).all())
        passes = -1 if C < 100 else 1  # the reference takes C^3 a pass
        good = True
        if C <= 300:
            qpath.qp_repair_batch(h, 4, st, passes, p, n, s, stream=stream)
            torch.cuda.synchronize()
            for r in range(4):
                path, length, status = repair_ref.repair(X[r].reshape(-1).tolist(), d.tolist(), C, start, passes)
                good &= p[r].cpu().tolist() == path and int(n[r]) == length and int(s[r]) == status
            results[f"repair-{name}"] = bool(good)
        for score, slack in ((None, 0), (rng.normal(0, 5, C).astype(np.float32), 0),
                             (rng.normal(0, 5, C).astype(np.float32), 2 * scale)):
            _, path, ln = qpath.qp_ws_walk(h, None if score is None else torch.from_numpy(score).cuda(), slack)
            torch.cuda.synchronize()
            ref = mlp_ref.walk(d, C, start, score, slack)
            results[f"walk-{name}-{slack}-{score is None}"] = path.cpu().numpy().tolist() == ref


def main():
    assert os.environ.get("QPATH_LIBRARY"), "run with QPATH_LIBRARY set to the checked build"
    assert qpath.qp_device_checks()[0], "the loaded library was built without device checks"
    oracle.build()
    results = {}
    singles(results)
    batches(results)
    paths(results)
    enabled, first_failure = qpath.qp_device_checks()
    print(json.dumps({"enabled": enabled, "first_failure": first_failure, "results": results}))
    return 0 if enabled and first_failure == 0 and all(v is True for v in results.values()) else 1


if __name__ == "__main__":
    sys.exit(main())
