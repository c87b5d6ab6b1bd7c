"""The event-driven sweep from states of many cells (half of them, all, a few
rows full): the state's records, column sums, energy and first sweeps against the
oracle, for fields around the sizes where the layout changes and for rows that
start at every byte offset."""
import numpy as np
import pytest

from conftest import has_gpu
from paper_2608_25376_gb300 import build as qbuild
from paper_2608_25376_gb300 import inputs, qpath

pytestmark = pytest.mark.gpu


def strip(rows, cols, cells, seed=3):
    rng = np.random.default_rng(seed)
    m = np.zeros(rows * cols, np.uint8)
    m[rng.permutation(rows * cols)[:cells]] = 1
    return inputs.Field(rows, cols, m, int(np.flatnonzero(m)[cells // 2]))


FIELDS = {"15": (strip(4, 5, 15), 100, 0), "16": (inputs.rect(4, 4), 100, 0), "17": (strip(4, 5, 17), 100, 0),
          "33": (strip(6, 6, 33), 100, 0), "92-i32": (strip(10, 10, 92), 30000, 0), "125": (strip(12, 12, 125), 100, 0),
          "126": (strip(12, 12, 126), 100, 0), "236": (strip(16, 16, 236), 100, 0), "257": (strip(17, 17, 257), 100, 0),
          "257-i32": (strip(17, 17, 257), 3000, 0), "line-300": (inputs.rect(1, 300, start=7), 100, 900)}


@pytest.mark.parametrize("name", list(FIELDS))
def test_states_of_many_cells(orc, name):
    if not has_gpu():
        pytest.skip("no CUDA device")
    import torch
    qbuild.build()
    f, scale, A = FIELDS[name]
    P = orc.Problem(f.rows, f.cols, f.free_mask, f.start, A=A or None, scale=scale)
    h = qpath.qp_build_qubo(f, A=A, scale=scale)
    rng = np.random.default_rng(P.C)
    C, R = P.C, 9
    x = np.zeros((R, C, C), np.uint8)
    for r, density in enumerate((0.05, 0.15, 0.4, 0.5, 0.9, 1.0)):
        x[r] = (rng.random((C, C)) < density) * rng.integers(1, 256, (C, C))
    x[6, ::3] = 1  # every third row full
    x[7, :, ::4] = 1  # every fourth column: rows of a cell in each four bytes
    x[8, C // 2, :min(C, 3)] = 1  # three cells in one row
    S, T0 = 3, float(P.d.max())
    st = torch.zeros((R, C * C), dtype=torch.uint8, device="cuda")
    E, B, acc = (torch.zeros(R, dtype=torch.int64, device="cuda") for _ in range(3))
    ini = torch.from_numpy(x.reshape(R, -1)).cuda()
    for end in (0, S):  # the state's own energy, and a few sweeps
        ref = orc.anneal_structured(P, R, S, T0=T0, T1=T0 / 9, seed=5, init_states=(x.reshape(R, -1) != 0).astype(np.uint8),
                                    sweep_begin=0, sweep_end=end)
        qpath.qp_anneal_ex(h, R, qpath.schedule(S, T0, T0 / 9, 0, end), 5, ini, st, E, B, accepts_out=acc,
                           stream=torch.cuda.current_stream())
        torch.cuda.synchronize()
        for g, r in ((st, ref.states), (E, ref.energies), (B, ref.best), (acc, ref.accepts)):
            assert np.array_equal(g.cpu().numpy(), r), (name, end)
