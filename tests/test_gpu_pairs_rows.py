"""Stacked GEMMs on CTA pairs with row counts around whole and half pairs of
tiles (64 networks fill a 128-row tile of the middle 30-qubit block's step),
trajectories of one network among large ones, against the same networks three
at a time on single CTAs.  The launch rule is evaluated for every call, so the
batches here do run on pairs and the small calls do not."""
import numpy as np
import pytest

import workloads as W
from test_gpu_pair_timeout import on_pairs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2604_08467_gb300 import ptn  # noqa: E402


@pytest.fixture(scope="module")
def planned():
    c2 = W.config_c2()
    plan = ptn.ptn_plan_path(c2["circuit"], c2["block_sizes"], hypersamples=100, est_traj=4096, est_shots=1e6,
                             mem_cap_bytes=40e9)
    deep = [s for s in plan.describe(1)["blocks"][1]["steps"] if s["kind"] == 2 and s["n_sum"] > 9]
    return plan, deep, ptn.ptn_presample_trajectories(plan, c2["seed"], 4)


def contract(plan, tr, traj, prefix, prec):
    nt = torch.tensor(traj, dtype=torch.int32, device="cuda")
    npf = torch.tensor(prefix, dtype=torch.int64, device="cuda")
    marg = torch.empty((len(traj), 1 << 10), device="cuda")
    Z = torch.empty(len(traj), dtype=torch.float64, device="cuda")
    ptn.ptn_contract_batch(plan, tr, 1, nt, npf, marg, Z, precision=prec)
    return marg


@pytest.mark.parametrize("prec", [ptn.PTN_PREC_FP32, ptn.PTN_PREC_BF16X3, ptn.PTN_PREC_FP16X3])
@pytest.mark.parametrize("sizes", [(1023, 1024), (1024, 1, 129, 512), (960, 63, 65, 1000), (127, 130, 1023, 1)])
def test_pair_rows(planned, prec, sizes):
    plan, deep, tr = planned
    size = 4 if prec == ptn.PTN_PREC_FP32 else 2
    assert all(on_pairs(s, sum(sizes), len(sizes), size) and not on_pairs(s, 3, 1, size) for s in deep) and deep
    rng = np.random.default_rng(sum(sizes))
    traj = np.repeat(np.arange(len(sizes)), sizes)
    prefix = np.concatenate([np.sort(rng.permutation(1024)[:k]) for k in sizes])
    got = contract(plan, tr, traj, prefix, prec)
    assert bool(torch.isfinite(got).all())
    edges = np.cumsum((0,) + sizes)
    starts = {int(e) + d for e in edges for d in (-3, -1, 0, 61, 63, 125, 127)} | set(range(0, len(traj), 211))
    for lo in sorted(x for x in starts if 0 <= x < len(traj)):
        hi = min(lo + 3, len(traj))
        assert torch.equal(contract(plan, tr, traj[lo:hi], prefix[lo:hi], prec), got[lo:hi])
