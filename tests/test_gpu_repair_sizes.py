"""The repair where its kernels change or could go wrong, path for path against
the plain reference: state sizes off the 16-byte grid, rows of several cells,
fields whose smallest distance is not one grid step, 32-bit distances, a grid
too wide for a distance table, every pass limit."""
import numpy as np
import pytest

from conftest import has_gpu
from oracle import repair_ref
from paper_2608_25376_gb300 import build as qbuild
from paper_2608_25376_gb300 import inputs, qpath

pytestmark = pytest.mark.gpu


def field(rows, cols, cells, seed, pitch=1):
    """`cells` free cells among those whose row and column are multiples of `pitch`."""
    rng = np.random.default_rng(seed)
    ok = [r * cols + c for r in range(0, rows, pitch) for c in range(0, cols, pitch)]
    mask = np.zeros(rows * cols, np.uint8)
    mask[rng.permutation(ok)[:cells]] = 1
    return inputs.Field(rows, cols, mask, int(np.flatnonzero(mask)[cells // 2]))


CASES = {
    "2": (field(1, 2, 2, 0), 100), "3": (field(2, 2, 3, 0), 100), "33": (field(6, 6, 33, 1), 100),
    "64": (field(8, 8, 64, 2), 100), "pitch-2": (field(17, 17, 70, 3, pitch=2), 100),
    "int32": (field(9, 9, 70, 4), 40000), "129": (field(12, 12, 129, 5), 100),
    "line-no-table": (field(1, 300, 90, 6), 100), "wide": (field(3, 200, 120, 7), 100),
}


@pytest.mark.parametrize("name", list(CASES))
def test_repair(name):
    if not has_gpu():
        pytest.skip("no CUDA device")
    import torch
    qbuild.build()
    f, scale = CASES[name]
    h = qpath.qp_build_qubo(f, scale=scale)
    C = h.info["C"]
    d = qpath.qp_export_dist(h).tolist()
    start = int(np.cumsum(f.free_mask)[f.start] - 1)
    rng = np.random.default_rng(C)
    X = np.zeros((9, C, C), np.uint8)
    for r in range(9):
        perm = np.r_[start, rng.permutation([i for i in range(C) if i != start])].astype(int)
        X[r, np.arange(C), perm] = 1
        if r % 3 == 1:  # rows of none and of several cells, cells twice
            X[r] ^= (rng.random((C, C)) < 1.0 / C).astype(np.uint8)
        if r % 3 == 2:
            X[r] = rng.random((C, C)) < 3.0 / C
    X[8] = 0
    buf = torch.zeros(X.size + 16, dtype=torch.uint8, device="cuda")
    for passes, shift in ((0, 0), (1, 1), (2, 0), (-1, 5)):
        st = buf[shift:shift + X.size]
        st.copy_(torch.from_numpy(X.reshape(-1)))
        p = torch.zeros((9, C), dtype=torch.int32, device="cuda")
        n = torch.zeros(9, dtype=torch.int64, device="cuda")
        s = torch.zeros(9, dtype=torch.int32, device="cuda")
        qpath.qp_repair_batch(h, 9, st, passes, p, n, s, stream=torch.cuda.current_stream())
        torch.cuda.synchronize()
        rows = range(9) if passes >= 0 or C < 70 else (0, 1, 2, 8)  # the reference takes C^3 a pass
        for r in rows:
            path, length, status = repair_ref.repair(X[r].reshape(-1).tolist(), d, C, start, passes)
            assert p[r].cpu().tolist() == path and int(n[r]) == length and int(s[r]) == status, (name, passes, r)
