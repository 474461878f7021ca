"""Memory caps on blocks listed class by class, whose buffers are larger than those
of the path's own order (the order of plans with fuse_max = 1): a cap that holds a
network in the path's order is accepted, a call is not split into chunks that cost
more launches than the path's order takes, and every result has the bits of the
uncapped call."""
import numpy as np
import pytest

import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2604_08467_gb300 import ptn  # noqa: E402


def one_network(block):
    return 8.0 * (block["arena_const"] + block["arena_traj"] + block["arena_net"]) + 12.0


def test_small_batch_budget_is_accepted():
    circ = W.paper_random_circuit(60, 360, np.random.default_rng(7))

    def plan_of(**o):
        return ptn.ptn_plan_path(circ, [10] * 6, hypersamples=16, est_traj=64, est_shots=256, **o)

    plan = plan_of()
    by_class = [one_network(b) for b in plan.describe(0)["blocks"]]
    in_order = [one_network(b) for b in plan_of(fuse_max=1).describe(0)["blocks"]]
    budget = 1.2 * max(in_order)
    assert max(by_class) > budget
    tr = ptn.ptn_presample_trajectories(plan, 5, 12)
    want = ptn.ptn_sample_shots(plan, tr, 7, shots_per_traj=20).to_torch()
    (status, res), = ptn.ptn_sample_shots_batch([{"plan": plan, "traj": tr, "seed": 7, "shots_per_traj": 20}],
                                                n_workers=1, mem_budget_bytes=budget)
    assert status == 0, status
    for a, b in zip(want, res.to_torch()):
        assert torch.equal(a, b)
    # the plan's own cap is back: the same call again, class by class
    for a, b in zip(want, ptn.ptn_sample_shots(plan, tr, 7, shots_per_traj=20).to_torch()):
        assert torch.equal(a, b)


@pytest.mark.parametrize("cap", [5.2e6, 2.1e7, 8.3e7])
def test_chunked_calls_take_the_listing_with_fewer_launches(cap):
    circ = W.attach_noise(W.brickwork_1d(40, 6, np.random.default_rng(1)), [W.depolarizing_kraus(0.01)])
    n = 256

    def run(j=1, **o):
        plan = ptn.ptn_plan_path(circ, [10] * 4, hypersamples=16, est_traj=n, est_shots=25600, **o)
        tr = ptn.ptn_presample_trajectories(plan, 4, n)
        nt = torch.arange(n, dtype=torch.int32, device="cuda")
        npf = (torch.arange(n, device="cuda") * 2654435761) % (1 << 10)
        marg = torch.empty((n, 1 << 10), device="cuda")
        Z = torch.empty(n, dtype=torch.float64, device="cuda")
        ptn.ptn_stats_enable(True)
        ptn.ptn_stats_reset()
        ptn.ptn_contract_batch(plan, tr, j, nt, npf, marg, Z)
        chunks = ptn.ptn_stats_read()["finalize"]["launches"]
        ptn.ptn_stats_enable(False)
        res = [ptn.ptn_sample_shots(plan, tr, 6, shots_per_traj=4, use_graphs=g).to_torch() for g in (0, 1, 1)]
        return plan.describe(0)["blocks"][j], chunks, (marg, Z), res

    free, _, want, rec = run()
    order, chunks, _, _ = run(fuse_max=1, mem_cap_bytes=cap)
    assert free["arena_traj"] > order["arena_traj"]          # the block is listed class by class
    _, got_chunks, got, rec_cap = run(mem_cap_bytes=cap)
    assert chunks > 1 and got_chunks == chunks
    assert torch.equal(want[0], got[0]) and torch.equal(want[1], got[1])
    for r in rec + rec_cap:
        for a, b in zip(rec[0], r):
            assert torch.equal(a, b)
