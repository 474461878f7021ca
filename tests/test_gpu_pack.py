"""Operand packing by rows (k_pack_rows) and of outer products (k_pack_prod)
over the lengths of the summed axis, in every format: amplitudes of circuits
whose tensor-core steps sum 2^3 .. 2^12 terms, against the statevector.
Tolerances: 1e-5 where operands hold 22 bits or more, 2^-16 relative per
BF16 hi/lo operand pair and product, i.e. 1e-4 over a path, for BF16."""
import numpy as np
import pytest

import workloads as W
from oracle import statevector as sv

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2604_08467_gb300 import ptn  # noqa: E402

TOL = {ptn.PTN_PREC_FP32: 1e-5, ptn.PTN_PREC_FP16X3: 1e-5, ptn.PTN_PREC_BF16X3: 1e-4}


@pytest.mark.parametrize("rows,cols,depth", [(3, 5, 9), (4, 4, 8), (4, 4, 11), (2, 8, 12)])
@pytest.mark.parametrize("prec", sorted(TOL))
@pytest.mark.parametrize("n_traj", [1, 5])
def test_amplitudes_over_summed_lengths(rows, cols, depth, prec, n_traj):
    circ = W.attach_noise(W.grid_4colour(rows, cols, depth, np.random.default_rng(depth)),
                          [W.depolarizing_kraus(0.02), W.amplitude_damping_kraus(0.05)])
    n = rows * cols
    plan = ptn.ptn_plan_path(circ, [8, n - 8], hypersamples=16, est_traj=n_traj, est_shots=100)
    steps = plan.describe(2)["expval"]["steps"]
    assert any(s["kind"] for s in steps)
    tr = ptn.ptn_presample_trajectories(plan, 3, n_traj)
    amp = torch.empty((n_traj, 1 << n), dtype=torch.complex64, device="cuda")
    ptn.ptn_trajectory_amplitudes(plan, tr, 0, n_traj, amp, precision=prec)
    kraus = tr.to_torch()[0].cpu().numpy()
    for t in range(n_traj):
        want = sv.trajectory_state(circ, kraus[t])
        assert np.linalg.norm(amp[t].cpu().numpy() - want) < TOL[prec] * np.linalg.norm(want)
