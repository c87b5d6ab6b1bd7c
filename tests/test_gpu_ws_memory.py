"""Training when the device refuses the large buffers: the layers' weight
gradients are then computed one after the other in one layer's buffers, and
give the bits of the pass that computes them side by side."""
import numpy as np
import pytest

from conftest import has_gpu
from paper_2608_25376_gb300 import build as qbuild
from paper_2608_25376_gb300 import qpath

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("M", [700, 2000])
def test_training_in_less_memory(monkeypatch, M):
    if not has_gpu():
        pytest.skip("no CUDA device")
    qbuild.build()
    Mp = (M + 127) // 128 * 128
    rng = np.random.default_rng(M)
    x = rng.normal(0, 1, (M, 16)).astype(np.float32)
    steps = rng.integers(2, 257, M).astype(np.int32)
    y = (rng.random(M) * steps).astype(np.int32)
    out = []
    for short in (False, True):
        m = qpath.WarmStartModel(seed=3)
        if short:  # below the four layers' transposes (3616 bytes a row), above every other buffer
            monkeypatch.setenv("QPATH_FAIL_ALLOC_OVER", str(3000 * Mp))
        else:
            monkeypatch.delenv("QPATH_FAIL_ALLOC_OVER", raising=False)
        loss, grads = qpath.qp_ws_grads(m, x, y, steps)
        for _ in range(2):
            qpath.qp_ws_train_step(m, x, y, steps, 1e-3)
        out.append((grads, np.float32(loss), qpath.qp_ws_get_params(m)))
    monkeypatch.delenv("QPATH_FAIL_ALLOC_OVER")
    for a, b in zip(*out):
        assert np.array_equal(a, b)
