"""The walk decode at the sizes where its kernel changes (128, 256, 512 cells,
a grid too wide for a distance table) and for both distance types, path for
path against the step-by-step reference."""
import numpy as np
import pytest

from conftest import has_gpu
from oracle import mlp_ref
from paper_2608_25376_gb300 import build as qbuild
from paper_2608_25376_gb300 import inputs, qpath

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("rows,cols,cells,scale", [(1, 2, 2, 100), (6, 6, 33, 100), (12, 12, 128, 100),
                                                   (12, 12, 129, 20000), (16, 16, 256, 100), (17, 17, 257, 2000),
                                                   (24, 24, 512, 100), (24, 24, 513, 100), (1, 300, 280, 100),
                                                   (90, 7, 300, 100)])
def test_walk(rows, cols, cells, scale):
    if not has_gpu():
        pytest.skip("no CUDA device")
    import torch
    qbuild.build()
    rng = np.random.default_rng(cells)
    mask = np.zeros(rows * cols, np.uint8)
    mask[rng.permutation(rows * cols)[:cells]] = 1
    start = int(np.flatnonzero(mask)[cells // 3])
    f = inputs.Field(rows, cols, mask, start)
    h = qpath.qp_build_qubo(f, scale=scale)
    d = qpath.qp_export_dist(h)
    s0 = int(np.cumsum(mask)[start] - 1)
    buf = torch.full((cells * cells + 5,), 9, dtype=torch.uint8, device="cuda")
    for score, slack in ((None, 0), (rng.normal(0, 50, cells).astype(np.float32), 0),
                         (np.round(rng.random(cells) * 3).astype(np.float32), 2 * scale)):
        sd = None if score is None else torch.from_numpy(score).cuda()
        st = buf[5:]
        _, path, ln = qpath.qp_ws_walk(h, sd, slack, state_out=st)
        torch.cuda.synchronize()
        ref = mlp_ref.walk(d, cells, s0, score, slack)
        assert path.cpu().numpy().tolist() == ref
        assert int(ln.item()) == sum(int(d[a, b]) for a, b in zip(ref, ref[1:]))
        x = st.cpu().numpy().reshape(cells, cells)
        assert x.sum() == cells and (x[np.arange(cells), ref] == 1).all()
    assert (buf[:5] == 9).all()


# Without a slack a step is one reduction over (distance, place in the order of
# scores): distances around the largest that fit beside the place, and scores
# that tie, are signed zeros or infinite.
@pytest.mark.parametrize("cells,scale", [(32, 100), (130, 2000), (256, 16384), (257, 25000), (512, 12000), (511, 100)])
def test_walk_ranked(cells, scale):
    if not has_gpu():
        pytest.skip("no CUDA device")
    import torch
    qbuild.build()
    rng = np.random.default_rng(cells + scale)
    mask = np.zeros(24 * 24, np.uint8)
    mask[rng.permutation(24 * 24)[:cells]] = 1
    start = int(np.flatnonzero(mask)[-1])
    h = qpath.qp_build_qubo(inputs.Field(24, 24, mask, start), scale=scale)
    d = qpath.qp_export_dist(h)
    score = np.round(rng.normal(0, 2, cells)).astype(np.float32)
    score[::7], score[3::11], score[5::13] = -0.0, np.inf, -np.inf
    for sc in (score, np.zeros(cells, np.float32), None):
        _, path, ln = qpath.qp_ws_walk(h, None if sc is None else torch.from_numpy(sc).cuda(), 0)
        torch.cuda.synchronize()
        ref = mlp_ref.walk(d, cells, cells - 1, sc, 0)
        assert path.cpu().numpy().tolist() == ref
        assert int(ln.item()) == sum(int(d[a, b]) for a, b in zip(ref, ref[1:]))
