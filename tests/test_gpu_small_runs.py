"""Fused runs of small trajectory-level steps (one launch, walked by dataflow
levels) against one launch per step (fuse_max = 1): every output is the same
multiply-add chain, so the marginals must be bit-identical."""
import numpy as np
import pytest

import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2604_08467_gb300 import ptn  # noqa: E402


def marginals(circ, blocks, n_traj, **opts):
    plan = ptn.ptn_plan_path(circ, blocks, hypersamples=4, est_traj=n_traj, est_shots=n_traj, **opts)
    tr = ptn.ptn_presample_trajectories(plan, 11, n_traj)
    out = []
    for j, (start, b) in enumerate(plan.blocks):
        nt = torch.arange(n_traj, dtype=torch.int32, device="cuda")
        npf = (torch.arange(n_traj, device="cuda") * 2654435761) % (1 << start)
        marg = torch.empty((n_traj, 1 << b), device="cuda")
        Z = torch.empty(n_traj, dtype=torch.float64, device="cuda")
        ptn.ptn_contract_batch(plan, tr, j, nt, npf, marg, Z)
        out += [marg, Z]
    return out, plan


# 1 trajectory, and the sizes where the threads per trajectory change
@pytest.mark.parametrize("n_traj", [1, 152, 153, 305])
@pytest.mark.parametrize("cache", [False, True])
def test_fused_equals_single_steps(n_traj, cache):
    circ = W.attach_noise(W.brickwork_1d(13, 7, np.random.default_rng(5)), [W.depolarizing_kraus(0.05)])
    fused, plan = marginals(circ, [7, 6], n_traj, cache_intermediates=cache)
    single, _ = marginals(circ, [7, 6], n_traj, cache_intermediates=cache, fuse_max=1)
    assert any(s["fuse_prev"] for b in plan.describe(1)["blocks"] for s in b["steps"])
    for a, b in zip(fused, single):
        assert torch.equal(a, b)


# a run longer than one launch holds (1024 steps), and runs cut short
@pytest.mark.parametrize("fuse_max", [3, 4096])
def test_long_and_cut_runs(fuse_max):
    circ = W.paper_random_circuit(5, 1300, np.random.default_rng(2), frac_2q=0.03)
    fused, plan = marginals(circ, [3, 2], 3, fuse_max=fuse_max)
    single, _ = marginals(circ, [3, 2], 3, fuse_max=1)
    assert any(sum(s["fuse_prev"] for s in b["steps"]) > 1024 for b in plan.describe(1)["blocks"])
    for a, b in zip(fused, single):
        assert torch.equal(a, b)


# network-level runs (blocks listed class by class), past one word of prefix bits;
# the sizes are those where the threads per network change
@pytest.mark.parametrize("n_net", [1, 153, 400])
def test_network_runs(n_net):
    circ = W.paper_random_circuit(70, 420, np.random.default_rng(9))
    fused = ptn.ptn_plan_path(circ, [10] * 7, hypersamples=8, est_traj=n_net, est_shots=n_net)
    single = ptn.ptn_plan_path(circ, [10] * 7, hypersamples=8, est_traj=n_net, est_shots=n_net, fuse_max=1)
    blocks = fused.describe(1)["blocks"]
    assert any(s["out_cls"] == 2 and s["fuse_prev"] for b in blocks for s in b["steps"])
    shots = ptn.ptn_sample_shots(fused, ptn.ptn_presample_trajectories(fused, 4, n_net), 6, shots_per_traj=1)
    words = shots.to_torch()[1].clone()             # prefixes with weight, [n_net, 2]
    for j in (1, 4, 6):
        out = []
        for plan in (fused, single):
            tr = ptn.ptn_presample_trajectories(plan, 4, n_net)
            marg = torch.empty((n_net, 1 << 10), device="cuda")
            Z = torch.empty(n_net, dtype=torch.float64, device="cuda")
            nt = torch.arange(n_net, dtype=torch.int32, device="cuda")
            ptn.ptn_contract_batch(plan, tr, j, nt, words.reshape(-1), marg, Z)
            out.append((marg, Z))
        assert torch.equal(out[0][0], out[1][0]) and torch.equal(out[0][1], out[1][1])
        assert float(out[0][1].min()) > 0
