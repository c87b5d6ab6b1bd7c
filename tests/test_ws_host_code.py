"""The network's host code (qp_ws.cpp) on the CPU, against stand-ins for the
CUDA runtime and the kernels (ws_host_fakes.cpp)."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

from paper_2608_25376_gb300 import build as qbuild

HERE = os.path.dirname(os.path.abspath(__file__))
HOST, MANAGED = -1, -2
ENOMEM = 2


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    so = str(tmp_path_factory.mktemp("ws") / "ws_host.so")
    subprocess.run(["g++", "-O1", "-fPIC", "-std=c++17", "-shared", "-Wl,-Bsymbolic", "-I", qbuild.INC, "-I", qbuild.CSRC,
                    "-I", os.path.join(qbuild._cuda_home(), "include"), os.path.join(qbuild.CSRC, "qp_ws.cpp"),
                    os.path.join(HERE, "ws_host_fakes.cpp"), "-o", so], check=True)
    L = ctypes.CDLL(so)
    L.fake_z2.restype = ctypes.c_void_p
    L.fake_bytes.restype = ctypes.c_size_t
    L.fake_limit.argtypes = [ctypes.c_size_t]
    L.fake_copied.restype = ctypes.c_long
    L.fake_launches.restype = L.fake_error.restype = ctypes.c_char_p
    L.qp_ws_create.argtypes = [ctypes.c_uint64, ctypes.POINTER(ctypes.c_void_p)]
    return L


@pytest.fixture
def model(lib):
    m = ctypes.c_void_p()
    lib.fake_limit(1 << 60)
    lib.fake_place(HOST)
    assert lib.qp_ws_create(1, ctypes.byref(m)) == 0
    lib.fake_launches()
    yield m
    lib.qp_ws_destroy(m)


def ptr(a):
    return ctypes.c_void_p(a.ctypes.data)


def logits(rows):
    """rows x 256 floats at a 16-byte boundary."""
    a = np.zeros(rows * 256 + 4, np.float32)
    at = -a.ctypes.data % 16 // 4
    return a[at:at + rows * 256]


# The kernel may store only into its own GPU's memory: another GPU's is copied, as are managed and host buffers.
@pytest.mark.parametrize("place,direct", [(0, True), (1, False), (MANAGED, False), (HOST, False)])
def test_forward_writes_only_its_own_gpu(lib, model, place, direct):
    M = 130
    out, feats = logits(M), np.zeros((M, 16), np.float32)
    lib.fake_place(place)
    before = lib.fake_copied()
    assert lib.qp_ws_forward(model, ptr(feats), M, ptr(out), None) == 0
    assert (lib.fake_z2() == out.ctypes.data) == direct
    assert (lib.fake_copied() - before == 0) == direct


# What a pass over Mp rows took when every product had its buffers to itself: one layer's transposes and split-K
# partials at a time.  A card whose memory is nearly full has to go on taking the row counts that fitted then.
ROW_BYTES = 5676


def old_training_bytes(Mp):
    splits = max(1, Mp // 512)
    per = -(-(-(-Mp // splits)) // 64) * 64
    return ROW_BYTES * Mp + -(-Mp // per) * 256 * 256 * 4 + 64 * 256 * 4  # and the column sums' slabs


@pytest.mark.parametrize("mode", [0, 1])
def test_forward_memory(lib, model, mode):
    M = 5000
    Mp = 5120
    base = lib.fake_bytes()
    assert lib.qp_ws_set_forward_mode(model, mode) == 0
    lib.fake_limit(base + ROW_BYTES * Mp)
    out, feats = logits(M), np.zeros((M, 16), np.float32)
    assert lib.qp_ws_forward(model, ptr(feats), M, ptr(out), None) == 0, lib.fake_error()
    assert lib.fake_bytes() - base <= ROW_BYTES * Mp
    # every buffer can still be read back, whether or not the pass wrote it
    lib.fake_limit(1 << 60)
    buf = np.zeros(Mp * 1024, np.uint8)
    for which in range(9):
        assert lib.qp_ws_get_buffer(model, which, Mp, ptr(buf)) == 0
    assert lib.qp_ws_get_buffer(model, 0, Mp + 1, ptr(buf)) != 0


def test_training_memory(lib, model):
    M = 5000
    Mp = 5120
    base = lib.fake_bytes()
    feats = np.zeros((M, 16), np.float32)
    labels, steps = np.zeros(M, np.int32), np.full(M, 7, np.int32)
    loss = ctypes.c_float()

    def step():
        return lib.qp_ws_train_step(model, ptr(feats), ptr(labels), ptr(steps), M, ctypes.c_float(1e-3),
                                    ctypes.byref(loss), None)

    lib.fake_limit(base + old_training_bytes(Mp) + 3 * 64 * 256 * 4)  # the slabs of three more layers: no row's worth
    assert step() == 0, lib.fake_error()
    assert lib.fake_launches() == b"ifb" + b"tgcs" + 3 * b"tgs" + b"a"
    assert lib.qp_ws_forward(model, ptr(feats), M, ptr(logits(M)), None) == 0
    lib.fake_launches()
    lib.fake_limit(lib.fake_bytes())  # more rows: refused before any launch, and the model goes on
    more = np.zeros((4 * M, 16), np.float32)
    assert lib.qp_ws_forward(model, ptr(more), 4 * M, ptr(logits(4 * M)), None) == ENOMEM
    assert lib.fake_launches() == b""
    lib.fake_limit(1 << 60)
    assert step() == 0
    assert lib.fake_launches() == b"ifbtgcsa"  # all layers side by side
