"""Waits that run out in tensor-core GEMMs on CTA pairs: both CTAs stop, the
copies of both land before either leaves, the call returns PTN_ERR_TIMEOUT, and
with the default limit the same call gives the bits it gave before.  The short
limits above zero stop the two producers of a pair at different stages; whether
they run out depends on the clock, so a call either times out or gives its result."""
import numpy as np
import pytest

import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2604_08467_gb300 import ptn  # noqa: E402

TIMEOUT = 6
SIZES = (1000, 901)     # networks of two trajectories


def on_pairs(step, n_net, n_traj, elem_bytes):
    """The launch rule of a stacked step (kind 2): at least 8 k-blocks, 256 realified
    columns, more 128 x 128 tiles than SMs, 4 row tiles per trajectory."""
    a, b = step["gemm_a"], 1 - step["gemm_a"]
    m = 1 << sum(1 for x, y in zip(step["out_stride"][a], step["out_stride"][b]) if x and not y)
    n2 = 2 << sum(1 for x, y in zip(step["out_stride"][a], step["out_stride"][b]) if y and not x)
    kb = (2 << step["n_sum"]) * elem_bytes // 128
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    return kb >= 8 and n2 >= 256 and n_net * m // 128 * (n2 // 128) > sms and n_net * m >= 4 * 128 * n_traj


@pytest.mark.parametrize("prec,elem_bytes", [(ptn.PTN_PREC_FP32, 4), (ptn.PTN_PREC_FP16X3, 2)])
def test_pairs_leave_after_waits_that_run_out(prec, elem_bytes):
    c2 = W.config_c2()
    plan = ptn.ptn_plan_path(c2["circuit"], c2["block_sizes"], hypersamples=100, est_traj=4096, est_shots=1e6,
                             mem_cap_bytes=40e9)
    steps = plan.describe(1)["blocks"][1]["steps"]
    assert any(s["kind"] == 2 and on_pairs(s, sum(SIZES), len(SIZES), elem_bytes) for s in steps)
    tr = ptn.ptn_presample_trajectories(plan, c2["seed"], len(SIZES))
    rng = np.random.default_rng(3)
    nt = torch.tensor(np.repeat(np.arange(len(SIZES)), SIZES), dtype=torch.int32, device="cuda")
    npf = torch.tensor(np.concatenate([np.sort(rng.permutation(1024)[:k]) for k in SIZES]), device="cuda")

    def run():
        marg = torch.empty((len(nt), 1 << 10), device="cuda")
        Z = torch.empty(len(nt), dtype=torch.float64, device="cuda")
        ptn.ptn_contract_batch(plan, tr, 1, nt, npf, marg, Z, precision=prec)
        torch.cuda.synchronize()
        return marg

    before = run()
    for limit in [0.0, 0.0, 1e-6, 3e-6, 1e-5, 3e-5, 1e-4]:
        ptn.ptn_set_wait_limit(limit)
        try:
            if limit == 0.0:
                with pytest.raises(ptn.PtnError) as e:
                    run()
                assert e.value.status == TIMEOUT
            else:
                try:
                    assert torch.equal(run(), before)
                except ptn.PtnError as err:
                    assert err.status == TIMEOUT
        finally:
            ptn.ptn_set_wait_limit(2.0)
        assert torch.equal(run(), before)
