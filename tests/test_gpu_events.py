"""The event-driven sweep against the CPU oracle, bit for bit: fields at the
edges of its layouts (one warp of columns, the staged distance matrix, the
distance table, neither; spins in shared and in global memory), hot sweeps
with many and with few survivors, states far from one-hot, both distance
types, weights, resumed and settled sweeps."""
import numpy as np
import pytest

from conftest import has_gpu
from paper_2608_25376_gb300 import build as qbuild
from paper_2608_25376_gb300 import inputs, qpath

pytestmark = pytest.mark.gpu


def strip(rows, cols, cells, seed=3):
    """A rows x cols grid with the given number of free cells."""
    rng = np.random.default_rng(seed)
    m = np.zeros(rows * cols, np.uint8)
    m[rng.permutation(rows * cols)[:cells]] = 1
    return inputs.Field(rows, cols, m, int(np.flatnonzero(m)[cells // 2]))


# (field, sweeps, T0, T1, replicas, scale, B, A, initial state's density)
CASES = {
    "1x2": (inputs.rect(1, 2), 40, 500.0, 1.0, 3, 100, 1, 0, None),
    "3x3": (inputs.rect(3, 3), 200, 1000.0, 1.0, 9, 100, 1, 0, None),
    "31-cells": (strip(6, 6, 31), 120, 1000.0, 1.0, 5, 100, 1, 0, None),
    "32-cells": (strip(6, 6, 32), 120, 1000.0, 1.0, 5, 100, 1, 0, 0.3),
    "33-cells": (strip(6, 6, 33), 120, 1000.0, 1.0, 5, 100, 1, 0, None),
    "33-full": (strip(6, 6, 33), 60, 500.0, 1.0, 4, 100, 1, 0, 1.0),
    "65-cells-hot": (strip(9, 9, 65), 80, 1200.0, 400.0, 6, 100, 1, 0, 0.05),
    "10x10": (inputs.obstacles(10, 10, 0.1, seed=1), 300, 1000.0, 1.0, 7, 100, 1, 0, None),
    "10x10-cold": (inputs.obstacles(10, 10, 0.1, seed=1), 60, 100.0, 1.0, 5, 100, 1, 0, 0.5),
    "10x10-B3": (inputs.obstacles(10, 10, 0.1, seed=1), 60, 900.0, 5.0, 5, 100, 3, 4000, None),
    "10x10-B0": (inputs.obstacles(10, 10, 0.1, seed=1), 60, 900.0, 5.0, 5, 100, 0, 0, None),
    "10x10-small-A": (inputs.obstacles(10, 10, 0.1, seed=1), 80, 200.0, 1.0, 5, 100, 1, 480, None),
    "10x10-int32": (inputs.obstacles(10, 10, 0.1, seed=1), 60, 300000.0, 300.0, 5, 30000, 1, 0, None),
    "136-cells": (strip(12, 12, 136), 50, 1000.0, 1.0, 4, 100, 1, 0, None),
    "144-cells-table": (strip(12, 13, 144), 50, 1000.0, 1.0, 4, 100, 1, 0, 0.02),
    "256-cells": (inputs.rect(16, 16), 24, 1500.0, 1.0, 4, 100, 1, 0, None),
    "257-cells": (strip(17, 17, 257), 24, 1500.0, 1.0, 4, 100, 1, 0, 0.01),
    "300-line": (inputs.rect(1, 300, start=7), 8, 2500.0, 100.0, 3, 100, 1, 900, None),
    "300-line-int32": (inputs.rect(1, 300, start=7), 8, 40000.0, 2000.0, 3, 3000, 1, 9000, 0.01),
    "24x24": (inputs.obstacles(24, 24, 0.15, seed=1), 12, 1500.0, 1.0, 4, 100, 1, 0, None),
    "530-cells": (strip(23, 24, 530), 6, 2000.0, 1.0, 3, 100, 1, 0, 0.01),
    "1025-cells": (strip(33, 33, 1025), 3, 2500.0, 10.0, 2, 100, 1, 0, None),
}


def run(h, R, sc, seed, init=None, offset=0, rpc=0, flags=0, kernel=qpath.QP_KERNEL_STRUCTURED):
    import torch
    n = h.info["n"]
    st = torch.full((R, n), 7, dtype=torch.uint8, device="cuda")
    E, B, A = (torch.zeros(R, dtype=torch.int64, device="cuda") for _ in range(3))
    ini = None if init is None else torch.from_numpy(np.ascontiguousarray(init)).cuda()
    qpath.qp_anneal_ex(h, R, sc, seed, ini, st, E, B, kernel=kernel, accepts_out=A, replica_offset=offset,
                       replicas_per_cta=rpc, flags=flags, stream=torch.cuda.current_stream())
    torch.cuda.synchronize()
    return st.cpu().numpy(), E.cpu().numpy(), B.cpu().numpy(), A.cpu().numpy()


@pytest.fixture(scope="module")
def dev():
    if not has_gpu():
        pytest.skip("no CUDA device")
    qbuild.build()


@pytest.mark.parametrize("name", list(CASES))
def test_matches_oracle(dev, orc, name):
    f, S, T0, T1, R, scale, B, A, density = CASES[name]
    P = orc.Problem(f.rows, f.cols, f.free_mask, f.start, A=A or None, B=B, scale=scale)
    h = qpath.qp_build_qubo(f, A=A, B=B, scale=scale)
    assert h.info["A"] == P.A
    init = None
    if density is not None:
        init = (np.random.default_rng(5).random((R, P.n)) < density).astype(np.uint8)
    ref = orc.anneal_structured(P, R, S, T0=T0, T1=T1, seed=11, init_states=init)
    got = run(h, R, qpath.schedule(S, T0, T1), 11, init)
    for g, r in zip(got, (ref.states, ref.energies, ref.best, ref.accepts)):
        assert np.array_equal(g, r), name
    # settled sweeps skipped, other launch shapes, and the chain in two parts
    skip = run(h, R, qpath.schedule(S, T0, T1), 11, init, rpc=2, flags=qpath.QP_ANNEAL_SKIP_SETTLED)
    assert all(np.array_equal(g, r) for g, r in zip(skip, got))
    m = S // 2
    first = run(h, R, qpath.schedule(S, T0, T1, 0, m), 11, init, rpc=1)
    second = run(h, R, qpath.schedule(S, T0, T1, m, S), 11, first[0])
    assert np.array_equal(second[0], got[0]) and np.array_equal(second[1], got[1])
    assert np.array_equal(first[3] + second[3], got[3])
    assert np.array_equal(np.minimum(first[2], second[2]), got[2])


def test_replica_offset(dev, orc):
    f = inputs.obstacles(10, 10, 0.1, seed=1)
    h = qpath.qp_build_qubo(f)
    sc = qpath.schedule(40, 900.0, 20.0)
    whole = run(h, 12, sc, 3)
    part = run(h, 5, sc, 3, offset=7)
    assert all(np.array_equal(w[7:], p) for w, p in zip(whole, part))


# Rows of one block of columns end at 125 cells; above, blocks without a cell of
# the row, an empty column or a survivor are passed over: rows of several cells
# and many survivors, rows and columns that empty and fill, cells in every block.
@pytest.mark.parametrize("cells,T0,density", [(125, 1500.0, 0.02), (126, 1500.0, 0.02), (127, 600.0, None),
                                              (253, 2000.0, 0.008), (254, 900.0, None), (381, 2500.0, 0.005)])
def test_blocks_of_columns(dev, orc, cells, T0, density):
    f = strip(21, 21, cells)
    R, S = 4, 14
    P = orc.Problem(f.rows, f.cols, f.free_mask, f.start)
    init = None if density is None else (np.random.default_rng(7).random((R, P.n)) < density).astype(np.uint8)
    ref = orc.anneal_structured(P, R, S, T0=T0, T1=50.0, seed=13, init_states=init)
    got = run(qpath.qp_build_qubo(f), R, qpath.schedule(S, T0, 50.0), 13, init)
    for g, r in zip(got, (ref.states, ref.energies, ref.best, ref.accepts)):
        assert np.array_equal(g, r)


# More chains than 8 per SM: CTAs of 4 or of 8 chains, the last one in part.
@pytest.mark.parametrize("R", [1217, 1300, 2000, 2433])
def test_many_chains(dev, R):
    h = qpath.qp_build_qubo(strip(5, 5, 22))
    sc = qpath.schedule(6, 900.0, 200.0)
    whole = run(h, R, sc, 3)
    for a, b in ((0, 600), (600, R - 1), (R - 1, R)):
        part = run(h, b - a, sc, 3, offset=a, rpc=1)
        assert all(np.array_equal(w[a:b], p) for w, p in zip(whole, part))
