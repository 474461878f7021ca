"""Levels of more than 64 qubits split into chunks: every chunk's networks are
projected by their own prefixes (two words each), so chunked calls give the bits
of one network at a time and of one chunk, with and without recorded graphs."""
import numpy as np
import pytest

import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2604_08467_gb300 import ptn  # noqa: E402

BLOCKS = [10] * 6 + [7, 7]     # the last one starts at qubit 67


def circuit():
    return W.paper_random_circuit(74, 444, np.random.default_rng(9))


def plan_of(cap=0.0):
    return ptn.ptn_plan_path(circuit(), BLOCKS, hypersamples=8, est_traj=40, est_shots=400, mem_cap_bytes=cap)


def contract(plan, tr, j, traj, words):
    """Marginals and totals of the networks, and the chunks they took (one finalisation each)."""
    b = plan.blocks[j][1]
    marg = torch.empty((len(traj), 1 << b), device="cuda")
    Z = torch.empty(len(traj), dtype=torch.float64, device="cuda")
    ptn.ptn_stats_enable(True)
    ptn.ptn_stats_reset()
    ptn.ptn_contract_batch(plan, tr, j, traj, words.reshape(-1), marg, Z)
    chunks = ptn.ptn_stats_read()["finalize"]["launches"]
    ptn.ptn_stats_enable(False)
    return marg, Z, chunks


@pytest.mark.parametrize("j", [1, 6, 7])
def test_memory_cap_chunks(j):
    whole = plan_of()
    tr = ptn.ptn_presample_trajectories(whole, 4, 40)
    s = ptn.ptn_sample_shots(whole, tr, 6, shots_per_traj=3)
    traj, words, _ = s.to_torch()          # records in order of trajectories; prefixes with weight
    assert words.shape[1] == 2 and len(traj) > 60 and bool((words[:, 1] != 0).any())
    one = plan_of(3e5)
    tr1 = ptn.ptn_presample_trajectories(one, 4, 40)
    marg, Z, chunks = contract(one, tr1, j, traj, words)
    assert chunks > 1
    assert float(Z.min()) > 0
    for i in range(len(traj)):
        m, z, c = contract(one, tr1, j, traj[i:i + 1].contiguous(), words[i:i + 1].contiguous())
        assert c == 1
        assert torch.equal(m[0], marg[i]) and torch.equal(z[0], Z[i])


@pytest.mark.parametrize("graphs", [0, 1])
@pytest.mark.parametrize("per_chunk", [1, 7])
def test_trajectory_chunks(per_chunk, graphs):
    plan = plan_of()
    tr = ptn.ptn_presample_trajectories(plan, 4, 40)
    want = ptn.ptn_sample_shots(plan, tr, 6, shots_per_traj=50).to_torch()
    got = ptn.ptn_sample_shots(plan, tr, 6, shots_per_traj=50, max_traj_per_chunk=per_chunk, use_graphs=graphs).to_torch()
    for a, b in zip(want, got):
        assert torch.equal(a, b)
