"""The event-driven kernel from several host threads at once, each on its own
handle and stream: launches of different shapes (matrix, table and global
distances, bitsets in shared and in global memory) set different shared-memory
limits of the same kernels.  Every result equals the one of a call alone, and
the oracle's."""
import threading

import numpy as np
import pytest

from conftest import has_gpu
import oracle
from paper_2608_25376_gb300 import build as qbuild
from paper_2608_25376_gb300 import inputs, qpath

pytestmark = pytest.mark.gpu

# field, replicas, sweeps, replicas per CTA
CASES = [(inputs.obstacles(6, 6, 0.2, seed=3, start=14), 32, 60, 0), (inputs.obstacles(10, 10, 0.1, seed=1), 24, 40, 8),
         (inputs.rect(7, 7), 24, 40, 2), (inputs.obstacles(16, 16, 0.1, seed=5, start=20), 8, 8, 4),
         (inputs.obstacles(18, 18, 0.1, seed=8, start=5), 4, 5, 1), (inputs.rect(24, 24), 3, 4, 3)]


def test_threads():
    if not has_gpu():
        pytest.skip("no CUDA device")
    import torch
    qbuild.build()
    oracle.build()
    out, errors = [[] for _ in CASES], []

    def work(i):
        try:
            f, R, S, rpc = CASES[i]
            s = torch.cuda.Stream()
            for _ in range(4):
                h = qpath.qp_build_qubo(f)
                with torch.cuda.stream(s):
                    st = torch.zeros((R, h.info["n"]), dtype=torch.uint8, device="cuda")
                    E = torch.zeros(R, dtype=torch.int64, device="cuda")
                    qpath.qp_anneal_ex(h, R, qpath.schedule(S), 7, None, st, E, replicas_per_cta=rpc, stream=s)
                s.synchronize()
                out[i].append((st.cpu().numpy(), E.cpu().numpy()))
                h.close()
        except Exception as e:  # reported below, on the main thread
            errors.append((i, repr(e)))

    threads = [threading.Thread(target=work, args=(i,)) for i in range(len(CASES))]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors
    for i, (f, R, S, _) in enumerate(CASES):
        ref = oracle.anneal_structured(oracle.Problem(f.rows, f.cols, f.free_mask, f.start), R, S, seed=7)
        assert len(out[i]) == 4
        for st, E in out[i]:
            assert np.array_equal(E, ref.energies) and np.array_equal(st, ref.states), i
