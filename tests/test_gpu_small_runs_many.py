"""Fused runs of small steps at the sizes where a launch takes other threads per
instance (152 and 456 instances), on both sides of each line and for
trajectory-level and network-level runs, against one launch per step."""
import numpy as np
import pytest

import workloads as W
from test_gpu_small_runs import marginals

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2604_08467_gb300 import ptn  # noqa: E402

SIZES = [152, 153, 456, 457, 2000]


@pytest.mark.parametrize("n", SIZES)
def test_trajectory_runs(n):
    circ = W.attach_noise(W.brickwork_1d(13, 7, np.random.default_rng(5)), [W.depolarizing_kraus(0.05)])
    fused, plan = marginals(circ, [7, 6], n)
    single, _ = marginals(circ, [7, 6], n, fuse_max=1)
    assert any(s["out_cls"] == 1 and s["fuse_prev"] for b in plan.describe(1)["blocks"] for s in b["steps"])
    for a, b in zip(fused, single):
        assert torch.equal(a, b)


@pytest.mark.parametrize("n", SIZES)
def test_network_runs(n):
    circ = W.paper_random_circuit(70, 420, np.random.default_rng(9))
    plans = [ptn.ptn_plan_path(circ, [10] * 7, hypersamples=8, est_traj=n, est_shots=n, fuse_max=f) for f in (0, 1)]
    assert any(s["out_cls"] == 2 and s["fuse_prev"] for b in plans[0].describe(1)["blocks"] for s in b["steps"])
    shots = ptn.ptn_sample_shots(plans[0], ptn.ptn_presample_trajectories(plans[0], 4, n), 6, shots_per_traj=1)
    words = shots.to_torch()[1].clone()
    out = []
    for plan in plans:
        tr = ptn.ptn_presample_trajectories(plan, 4, n)
        marg = torch.empty((n, 1 << 10), device="cuda")
        Z = torch.empty(n, dtype=torch.float64, device="cuda")
        nt = torch.arange(n, dtype=torch.int32, device="cuda")
        ptn.ptn_contract_batch(plan, tr, 4, nt, words.reshape(-1), marg, Z)
        out.append((marg, Z))
    assert torch.equal(out[0][0], out[1][0]) and torch.equal(out[0][1], out[1][1])
    assert float(out[0][1].min()) > 0
