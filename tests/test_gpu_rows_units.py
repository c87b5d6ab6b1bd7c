"""The row kernel on request (QP_KERNEL_STRUCTURED_ROWS) with more chains than
fit on the GPU at once and enough sweeps for several segments: the persistent
launch over (replica, sweep segment) units, whose chains hand their state from
segment to segment.  States, energies, best energies and accept counts equal
those of the whole chains (spins in shared memory) and of the event-driven
kernel; sampled replicas equal the oracle."""
import pytest

from conftest import has_gpu
from paper_2608_25376_gb300 import build as qbuild
from paper_2608_25376_gb300 import inputs, qpath

pytestmark = pytest.mark.gpu


def run(h, R, sc, kernel):
    import torch
    st = torch.zeros((R, h.info["n"]), dtype=torch.uint8, device="cuda")
    E, B, acc = (torch.zeros(R, dtype=torch.int64, device="cuda") for _ in range(3))
    qpath.qp_anneal_ex(h, R, sc, 7, None, st, E, B, kernel=kernel, accepts_out=acc, stream=torch.cuda.current_stream())
    torch.cuda.synchronize()
    return st, E, B, acc


@pytest.mark.parametrize("n_sweeps,begin", [(1200, 0), (2600, 1300)])
def test_segments_of_the_row_kernel(n_sweeps, begin):
    if not has_gpu():
        pytest.skip("no CUDA device")
    import oracle
    import torch
    qbuild.build()
    f = inputs.obstacles(18, 18, 0.1, seed=8, start=5)  # 292 cells: the spins are in global memory
    h = qpath.qp_build_qubo(f)
    R = 16 * torch.cuda.get_device_properties(0).multi_processor_count + 37  # at most 12 chains fit on an SM
    sc = qpath.schedule(n_sweeps, sweep_begin=begin, sweep_end=n_sweeps)
    got = run(h, R, sc, qpath.QP_KERNEL_STRUCTURED_ROWS)
    for kernel in (qpath.QP_KERNEL_STRUCTURED_ROWS_SHARED, qpath.QP_KERNEL_STRUCTURED):
        for a, b in zip(got, run(h, R, sc, kernel)):
            assert torch.equal(a, b), kernel
    idx = [0, R // 2, R - 1]
    o = oracle.anneal_structured(oracle.Problem(f.rows, f.cols, f.free_mask, f.start), idx, n_sweeps, seed=7,
                                 sweep_begin=begin, sweep_end=n_sweeps)
    for a, b in zip((got[0], got[1], got[2]), (o.states, o.energies, o.best)):
        assert (a.cpu().numpy()[idx] == b).all()
