"""Contractions of 8 and 16 k-blocks on CTA pairs, whose accumulators run one
after the other as segments, against single CTAs, which hold them side by side:
pairs are taken when the tiles outnumber the SMs, so a trajectory contracted
with few others runs on single CTAs and must give the same bits.  Batches just
above the SM count and of odd sizes."""
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
    for j in (0, 1):   # 2^8 terms: 8 k-blocks of FP16 / BF16, 16 of TF32; 256 columns, 8 to 32 tiles a trajectory
        assert any(s["kind"] == 1 and s["n_sum"] == 8 and 16 <= s["n_out"] <= 18
                   for s in plan.describe(1)["blocks"][j]["steps"])
    return plan, ptn.ptn_presample_trajectories(plan, c2["seed"], 37)


@pytest.mark.parametrize("prec", [ptn.PTN_PREC_FP32, ptn.PTN_PREC_BF16X3, ptn.PTN_PREC_FP16X3])
@pytest.mark.parametrize("block,n", [(0, 21), (0, 37), (1, 5), (1, 10), (1, 37)])
def test_short_pairs_equal_single_ctas(planned, prec, block, n):
    plan, tr = planned
    start, b = plan.blocks[block]
    prefix = np.random.default_rng(n).integers(0, 1 << start, n)

    def contract(lo, hi):
        nt = torch.arange(lo, hi, dtype=torch.int32, device="cuda")
        npf = torch.tensor(prefix[lo:hi], dtype=torch.int64, device="cuda")
        marg = torch.empty((hi - lo, 1 << b), device="cuda")
        Z = torch.empty(hi - lo, dtype=torch.float64, device="cuda")
        ptn.ptn_contract_batch(plan, tr, block, nt, npf, marg, Z, precision=prec)
        return marg

    got = contract(0, n)
    assert torch.isfinite(got).all() and (got.sum(1) > 0).all()
    for lo in (0, 3, n - 2):
        assert torch.equal(contract(lo, min(lo + 2, n)), got[lo:lo + 2])
