"""Recorded graphs of chunks that differ only in whether a GEMM runs on CTA
pairs: chunks of many and of few trajectories of one block, alternating in one
call, must give the records of the same call without graphs."""
import pytest

import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2604_08467_gb300 import ptn  # noqa: E402


@pytest.mark.parametrize("n_traj,chunk", [(47, 23), (37, 36), (25, 12)])   # a last chunk of one trajectory
def test_chunks_of_other_forms(n_traj, chunk):
    c2 = W.config_c2()
    plan = ptn.ptn_plan_path(c2["circuit"], c2["block_sizes"], hypersamples=100, est_traj=4096, est_shots=1e6,
                             mem_cap_bytes=40e9)
    tr = ptn.ptn_presample_trajectories(plan, c2["seed"], n_traj)

    def run(graphs):
        s = ptn.ptn_sample_shots(plan, tr, 5, shots_per_traj=100, max_traj_per_chunk=chunk,
                                 precision=ptn.PTN_PREC_FP16X3, use_graphs=graphs)
        return [x.cpu() for x in s.to_torch()[:3]]

    ref = run(0)
    for a, b in zip(ref, run(1)):
        assert torch.equal(a, b)
