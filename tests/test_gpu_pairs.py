"""Tensor-core GEMMs on CTA pairs (256 x 256 tiles) against single CTAs (128 x
128): the stacked contraction of a trajectory runs on pairs when its networks
fill enough rows, on single CTAs when contracted a few networks at a time, and
every accumulation is the same, so the marginals must be bit-identical.  Row
counts around whole and half pairs of tiles."""
import numpy as np
import pytest

import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2604_08467_gb300 import ptn  # noqa: E402


@pytest.fixture(scope="module")
def planned():
    c2 = W.config_c2()
    plan = ptn.ptn_plan_path(c2["circuit"], c2["block_sizes"], hypersamples=100, est_traj=4096, est_shots=1e6,
                             mem_cap_bytes=40e9)
    steps = plan.describe(1)["blocks"][1]["steps"]
    deep = [s for s in steps if s["kind"] == 2 and s["n_sum"] > 9]
    assert deep, "the middle block's stacked contraction is segmented"
    return plan, ptn.ptn_presample_trajectories(plan, c2["seed"], 4)


def contract(plan, tr, traj, prefix, prec):
    nt = torch.tensor(traj, dtype=torch.int32, device="cuda")
    npf = torch.tensor(prefix, dtype=torch.int64, device="cuda")
    marg = torch.empty((len(traj), 1 << 10), device="cuda")
    Z = torch.empty(len(traj), dtype=torch.float64, device="cuda")
    ptn.ptn_contract_batch(plan, tr, 1, nt, npf, marg, Z, precision=prec)
    return marg


@pytest.mark.parametrize("prec", [ptn.PTN_PREC_FP32, ptn.PTN_PREC_BF16X3, ptn.PTN_PREC_FP16X3])
@pytest.mark.parametrize("sizes", [(256, 320), (511, 257), (700, 1, 640)])
def test_pairs_equal_single_ctas(planned, prec, sizes):
    plan, tr = planned
    rng = np.random.default_rng(sum(sizes))
    traj = np.repeat(np.arange(len(sizes)), sizes)
    prefix = np.concatenate([np.sort(rng.permutation(1024)[:k]) for k in sizes])
    got = contract(plan, tr, traj, prefix, prec)
    for lo in list(range(0, len(traj), 83)) + [len(traj) - 3]:
        k = min(lo + 3, len(traj))
        assert torch.equal(contract(plan, tr, traj[lo:k], prefix[lo:k], prec), got[lo:k])
