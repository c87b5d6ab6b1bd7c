"""The greedy fix of states that are no paths (no 2-opt), path for path against
the plain reference: rows of none, one, several and most cells, cells taken
twice, fields around a multiple of 32 and 128 cells, both distance types."""
import numpy as np
import pytest

from conftest import has_gpu
from oracle import repair_ref
from paper_2608_25376_gb300 import build as qbuild
from paper_2608_25376_gb300 import inputs, qpath

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("side,cells,scale", [(6, 31, 100), (6, 33, 30000), (12, 128, 100), (12, 129, 8000),
                                              (17, 256, 100), (17, 257, 3000), (18, 289, 3000), (23, 513, 100)])
def test_greedy_fix(side, cells, scale):
    if not has_gpu():
        pytest.skip("no CUDA device")
    import torch
    qbuild.build()
    rng = np.random.default_rng(cells)
    mask = np.zeros(side * side, np.uint8)
    mask[rng.permutation(side * side)[:cells]] = 1
    f = inputs.Field(side, side, mask, int(np.flatnonzero(mask)[cells // 2]))
    h = qpath.qp_build_qubo(f, scale=scale)
    d = qpath.qp_export_dist(h).tolist()
    start, C, R = cells // 2, cells, 6
    X = np.zeros((R, C, C), np.uint8)
    X[0, np.arange(C), np.r_[start, rng.permutation([i for i in range(C) if i != start])].astype(int)] = 1
    X[0, C // 2] = X[0, 1]  # a cell taken twice
    for r, density in ((1, 1.0 / C), (2, 3.0 / C), (3, 0.3), (4, 0.9)):
        X[r] = rng.random((C, C)) < density
    X[5, ::2] = rng.random((len(X[5, ::2]), C)) < 0.05
    st = torch.from_numpy(X.reshape(R, -1)).cuda()
    p = torch.zeros((R, C), dtype=torch.int32, device="cuda")
    n = torch.zeros(R, dtype=torch.int64, device="cuda")
    s = torch.zeros(R, dtype=torch.int32, device="cuda")
    qpath.qp_repair_batch(h, R, st, 0, p, n, s, stream=torch.cuda.current_stream())
    torch.cuda.synchronize()
    for r in range(R):
        path, length, status = repair_ref.repair(X[r].reshape(-1).tolist(), d, C, start, 0)
        assert p[r].cpu().tolist() == path and int(n[r]) == length and int(s[r]) == status, r
