"""SIMT steps staged in shared memory (k_contract_rows) and contracted for
groups of networks that share an operand's rows (k_contract_group): the result
of a network must not depend, in any bit, on how many networks of which
prefixes are contracted with it, and must match the statevector."""
import numpy as np
import pytest

import workloads as W
from oracle import statevector as sv

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2604_08467_gb300 import ptn  # noqa: E402

BLOCKS = [4, 5, 3]


def contract(plan, tr, j, traj, prefix):
    nt = torch.tensor(traj, dtype=torch.int32, device="cuda")
    npf = torch.tensor(prefix, dtype=torch.int64, device="cuda")
    marg = torch.empty((len(traj), 1 << BLOCKS[j]), device="cuda")
    Z = torch.empty(len(traj), dtype=torch.float64, device="cuda")
    ptn.ptn_contract_batch(plan, tr, j, nt, npf, marg, Z)
    return marg


@pytest.mark.parametrize("form", [1, 2])       # double layer, ket only
@pytest.mark.parametrize("depth", [7, 10])
def test_batch_does_not_change_a_network(form, depth):
    circ = W.attach_noise(W.brickwork_1d(12, depth, np.random.default_rng(depth)), [W.depolarizing_kraus(0.05)])
    n_traj = 3
    plan = ptn.ptn_plan_path(circ, BLOCKS, hypersamples=8, est_traj=n_traj, est_shots=1000, simt_only=True,
                             network_form=form)
    tr = ptn.ptn_presample_trajectories(plan, 21, n_traj)
    kraus = tr.to_torch()[0].cpu().numpy()
    probs = [np.abs(sv.trajectory_state(circ, kraus[t])) ** 2 for t in range(n_traj)]
    rng = np.random.default_rng(3)
    for j, (start, b) in enumerate(plan.blocks):
        # many networks of the first trajectory, one of the second, in no order of
        # prefixes, and an odd number of the third
        sizes = [min(1 << start, 601), 1, min(1 << start, 37)]
        traj = np.repeat(np.arange(n_traj), sizes)
        prefix = np.concatenate([rng.permutation(1 << start)[:k] for k in sizes])
        got = contract(plan, tr, j, traj, prefix)
        for lo in list(range(0, len(traj), 97)) + [len(traj) - 1]:
            k = min(lo + 1 + lo % 5, len(traj))
            assert torch.equal(contract(plan, tr, j, traj[lo:k], prefix[lo:k]), got[lo:k])
        want = np.array([sv.block_marginals(probs[t], 12, start, b)[int(s)] for t, s in zip(traj, prefix)])
        err = np.linalg.norm(got.cpu().numpy() - want, axis=1) / np.maximum(np.linalg.norm(want, axis=1), 1e-12)
        assert err.max() < 2e-5
