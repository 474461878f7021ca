"""Tile tuning against what calls launch: only the steps that run alone are
timed, a step keeps its default (tile 0, with the kernels that stage rows in
shared memory) unless the tuner reports a change, and the default is among the
candidates, so tuning again finds no other reference."""
import numpy as np
import pytest

import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2604_08467_gb300 import ptn  # noqa: E402

N = 32


def direct_launches(plan, tr):
    """SIMT steps launched on their own by one contraction of every block."""
    n = 0
    for j, (start, b) in enumerate(plan.blocks):
        nt = torch.arange(N, dtype=torch.int32, device="cuda")
        npf = torch.zeros(N * ptn.words_of(plan.n_qubits), dtype=torch.int64, device="cuda")
        marg = torch.empty((N, 1 << b), device="cuda")
        Z = torch.empty(N, dtype=torch.float64, device="cuda")
        ptn.ptn_stats_enable(True)
        ptn.ptn_stats_reset()
        ptn.ptn_contract_batch(plan, tr, j, nt, npf, marg, Z)
        n += ptn.ptn_stats_read().get("contract_direct", {"launches": 0})["launches"]
        ptn.ptn_stats_enable(False)
    return n


# the 30-qubit brickwork (trajectory-level runs, a closing |a|^2), and a wide circuit
# whose blocks are listed class by class (network-level runs)
@pytest.mark.parametrize("family", ["brick", "paper"])
def test_tuning_keeps_the_default(family):
    if family == "brick":
        c2 = W.config_c2()
        plan = ptn.ptn_plan_path(c2["circuit"], c2["block_sizes"], hypersamples=100, est_traj=4096, est_shots=1e6)
    else:
        circ = W.paper_random_circuit(70, 420, np.random.default_rng(9))
        plan = ptn.ptn_plan_path(circ, [10] * 7, hypersamples=8, est_traj=N, est_shots=N)
    tr = ptn.ptn_presample_trajectories(plan, 5, N)
    alone = direct_launches(plan, tr)
    for _ in range(2):
        n_tuned, n_changed = ptn.ptn_tune_tiles(plan, tr, n_probe=N, reps=3)
        tiles = [s["tile"] for b in plan.describe(1)["blocks"] for s in b["steps"]]
        assert n_tuned == alone
        assert sum(t != 0 for t in tiles) == n_changed
