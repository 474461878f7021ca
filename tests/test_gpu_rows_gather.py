"""SIMT steps staged in shared memory whose summed axis is not contiguous in one
operand or in both (k_contract_rows copies such rows 8 bytes at a time): the
marginals must match the statevector, and a network's must not depend, in any
bit, on the networks contracted with it.

Tolerance: FP32 chains of at most 2^8 terms over a few hundred steps, relative
errors of order sqrt(steps) * 2^-24 * a small factor, below 2e-5 in the norm."""
import numpy as np
import pytest

import workloads as W
from oracle import statevector as sv

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2604_08467_gb300 import ptn  # noqa: E402


def gathered(step):
    """Operands with a summed axis in other than memory order, as a pair of bools."""
    k = step["n_sum"]
    if step["kind"] != 0 or step["virt"] or step["fuse_prev"] or not 3 <= k <= 8 or step["n_out"] + k < 12:
        return (False, False)
    return tuple(step["sum_stride"][o] != [1 << q for q in range(k)] for o in (0, 1))


# form 1 double layer, 2 ket only; sides: gathered operands; cls 1 a step per trajectory, 2 per network
@pytest.mark.parametrize("blocks,depth,form,sides,cls", [
    ([10, 4], 8, 1, (False, True), 1),
    ([7, 4, 3], 12, 1, (True, False), 1),
    ([7, 4, 3], 10, 1, (True, False), 2),
    ([7, 4, 3], 10, 2, (True, True), 1),
    ([10, 4], 12, 2, (True, True), 1),
])
def test_gathered_rows(blocks, depth, form, sides, cls):
    n, n_traj = 14, 3
    circ = W.attach_noise(W.brickwork_1d(n, depth, np.random.default_rng(depth)), [W.depolarizing_kraus(0.05)])
    plan = ptn.ptn_plan_path(circ, blocks, hypersamples=8, est_traj=n_traj, est_shots=1000, simt_only=True,
                             network_form=form)
    reached = [j for j, bl in enumerate(plan.describe(1)["blocks"])
               for st in bl["steps"] if gathered(st) == sides and st["out_cls"] == cls]
    assert reached, "the plan has no such step"
    tr = ptn.ptn_presample_trajectories(plan, 21, n_traj)
    kraus = tr.to_torch()[0].cpu().numpy()
    probs = [np.abs(sv.trajectory_state(circ, kraus[t])) ** 2 for t in range(n_traj)]
    rng = np.random.default_rng(3)

    def contract(j, traj, prefix):
        nt = torch.tensor(traj, dtype=torch.int32, device="cuda")
        npf = torch.tensor(prefix, dtype=torch.int64, device="cuda")
        marg = torch.empty((len(traj), 1 << plan.blocks[j][1]), device="cuda")
        Z = torch.empty(len(traj), dtype=torch.float64, device="cuda")
        ptn.ptn_contract_batch(plan, tr, j, nt, npf, marg, Z)
        return marg

    for j in sorted(set(reached)):
        start, b = plan.blocks[j]
        sizes = [min(1 << start, k) for k in (101, 1, 37)]
        traj = np.repeat(np.arange(n_traj), sizes)
        prefix = np.concatenate([rng.permutation(1 << start)[:k] for k in sizes])
        got = contract(j, traj, prefix)
        for lo in sorted({0, len(traj) // 2, len(traj) - 1}):
            assert torch.equal(contract(j, traj[lo:lo + 1], prefix[lo:lo + 1]), got[lo:lo + 1])
        want = np.array([sv.block_marginals(probs[t], n, start, b)[int(s)] for t, s in zip(traj, prefix)])
        err = np.linalg.norm(got.cpu().numpy() - want, axis=1) / np.maximum(np.linalg.norm(want, axis=1), 1e-12)
        assert err.max() < 2e-5
