"""The batch decode of states at the edges of its layout: state sizes that are
no multiple of 16 bytes (so that states start at every alignment), one to eight
warps per state, feasible states, infeasible ones and set bytes of any value.
A row's entry is its largest set cell (-1 for none); a state whose rows and
columns do not all hold one cell has length -1."""
import numpy as np
import pytest

from conftest import has_gpu
from paper_2608_25376_gb300 import build as qbuild
from paper_2608_25376_gb300 import inputs, qpath

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("cells", [2, 5, 9, 33, 45, 46, 64, 91, 128, 257, 515])
def test_decode_batch(cells):
    if not has_gpu():
        pytest.skip("no CUDA device")
    import torch
    qbuild.build()
    rng = np.random.default_rng(cells)
    side = int(np.ceil(np.sqrt(cells)))
    mask = np.zeros(side * side, np.uint8)
    mask[rng.permutation(side * side)[:cells]] = 1
    f = inputs.Field(side, side, mask, int(np.flatnonzero(mask)[0]))
    h = qpath.qp_build_qubo(f)
    d = qpath.qp_export_dist(h).astype(np.int64)
    C, R = cells, 21
    x = np.zeros((R, C, C), np.uint8)
    for r in range(R):
        x[r, np.arange(C), rng.permutation(C)] = rng.integers(1, 256, C)
        if r % 3 == 1:  # a cell too many, or one moved
            x[r, rng.integers(C), rng.integers(C)] ^= 3
        if r % 3 == 2:
            x[r] = rng.random((C, C)) < 2.0 / C
    on = x != 0
    paths = np.where(on.any(2), C - 1 - on[:, :, ::-1].argmax(2), -1).astype(np.int32)
    ok = (on.sum(1) == 1).all(1) & (on.sum(2) == 1).all(1)
    lengths = np.where(ok, d[paths[:, :-1], paths[:, 1:]].sum(1), -1)
    # an odd offset into a larger buffer: the states start at any byte
    buf = torch.zeros(R * C * C + 16, dtype=torch.uint8, device="cuda")
    for shift in (0, 3):
        st = buf[shift:shift + R * C * C]
        st.copy_(torch.from_numpy(x.reshape(-1)))
        p = torch.full((R, C), 99, dtype=torch.int32, device="cuda")
        n = torch.zeros(R, dtype=torch.int64, device="cuda")
        qpath.qp_decode_batch(h, R, st, p, n, stream=torch.cuda.current_stream())
        torch.cuda.synchronize()
        assert np.array_equal(p.cpu().numpy(), paths) and np.array_equal(n.cpu().numpy(), lengths)
