"""Marginal rows and their totals from the finalisation, at every width where its
units change (several networks per CTA, one, and tiles of 2^12 outcomes), in its
three forms (the root read, a closing |a|^2, a closing outer product), for
network counts that leave the last unit part full: against state vectors, with
totals equal to the rows' FP64 sums and with rows of infinities.  The largest
entry it keeps per row is checked through the exhaustive harvest."""
import numpy as np
import pytest

import workloads as W
from oracle import sampling
from oracle import statevector as sv

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2604_08467_gb300 import ptn  # noqa: E402

E = 150          # error sets; 4 prefixes of the first two qubits each


def two_bricks(n, cut, depth, rng, scale=1.0):
    """Brickwork on qubits 0 .. cut - 1 and on the others, with no gate between them."""
    gates = []
    for lo, m in ((0, cut), (cut, n - cut)):
        for g in W.brickwork_1d(m, depth, rng).gates if m else []:
            gates.append(W.Gate(tuple(q + lo for q in g.qubits), g.matrix))
    gates[2] = W.Gate(gates[2].qubits, gates[2].matrix * scale)      # the first gate of the block's first qubit
    return W.attach_noise(W.Circuit(n, gates, layout="1d"), [W.depolarizing_kraus(0.05)])


def circuit(mode, b, scale=1.0):
    rng = np.random.default_rng(100 * b + len(mode))
    if mode == "product":
        return two_bricks(2 + b, 2 + b // 2, 4, rng, scale), [2, b]
    n = 2 + b + (2 if mode == "root" else 0)
    return two_bricks(n, n, 4, rng, scale), [2, b] + ([2] if mode == "root" else [])


def closing(block):
    """The finalisation's form for a block, from its steps and root."""
    h, r = block["steps"][-1], block["root"]["op"]
    if h["kind"] or h["n_sum"] or h["virt"] or h["fuse_prev"] or h["n_out"] != block["b"]:
        return "root"
    if (r["arena"], r["arena_off"]) != (h["out_arena"], h["out_off"]):
        return "root"
    x, y = ({k: v for k, v in o.items() if k != "conj"} for o in h["ops"])
    return "square" if x == y and x["mode"] == 1 and not x["slices"] else "product"


def planned(mode, b, scale=1.0):
    circ, bs = circuit(mode, b, scale)
    # (fuse_max = 1: the closing product of a narrow block is not part of a fused run)
    plan = ptn.ptn_plan_path(circ, bs, hypersamples=8, est_traj=E, est_shots=4 * E, fuse_max=0 if mode == "root" else 1,
                             network_form={"root": 1, "square": 2, "product": 1}[mode])
    return circ, plan, ptn.ptn_presample_trajectories(plan, 11, E)


def rows_of(plan, tr, j, traj, prefix, prec=ptn.PTN_PREC_FP32):
    nt = torch.tensor(np.asarray(traj), dtype=torch.int32, device="cuda")
    npf = torch.tensor(np.asarray(prefix).astype(np.int64), dtype=torch.int64, device="cuda")
    marg = torch.full((len(traj), 1 << plan.blocks[j][1]), -1.0, device="cuda")
    Z = torch.full((len(traj),), -1.0, dtype=torch.float64, device="cuda")
    ptn.ptn_contract_batch(plan, tr, j, nt, npf, marg, Z, precision=prec)
    return marg.cpu().numpy().astype(np.float64), Z.cpu().numpy()


CASES = [(m, b) for m in ("root", "square", "product") for b in range(1, 14) if m != "product" or b > 1]


@pytest.mark.parametrize("mode,b", CASES)
def test_rows_and_totals(mode, b):
    circ, plan, tr = planned(mode, b)
    form = closing(plan.describe(1)["blocks"][1])       # (an |a|^2 of sliced factors is formed as a product)
    assert form == mode or (mode == "square" and form == "product")
    kraus = tr.to_torch()[0].cpu().numpy()
    traj, prefix = np.repeat(np.arange(E), 4), np.tile(np.arange(4), E)
    probs = {t: np.abs(sv.trajectory_state(circ, kraus[t])) ** 2 for t in range(0, E, 7)}
    full, Zf = rows_of(plan, tr, 1, traj, prefix)
    assert np.isfinite(full).all()
    np.testing.assert_allclose(Zf, full.sum(axis=1), rtol=1e-12)
    for i in range(len(traj)):
        if traj[i] in probs:
            want = sv.block_marginals(probs[traj[i]], circ.n_qubits, 2, b)[prefix[i]]
            assert np.linalg.norm(full[i] - want) < 2e-5 * max(np.linalg.norm(want), 1e-12)
    for n in (1, 3, 4, 5, 17, 257):
        m, Z = rows_of(plan, tr, 1, traj[:n], prefix[:n])
        assert np.array_equal(m, full[:n]) and np.array_equal(Z, Zf[:n])


# one gate scaled so that probabilities are around the largest FP32 number
@pytest.mark.parametrize("mode,b", [(m, b) for m in ("root", "square", "product") for b in (2, 3, 5, 9, 10, 11, 12, 13)])
def test_infinite_rows(mode, b):
    circ, plan, tr = planned(mode, b, scale=(1.2 if mode == "root" else 0.6) * (3.4e38 * 2.0 ** (b + 2)) ** 0.5)
    traj, prefix = np.repeat(np.arange(E), 4), np.tile(np.arange(4), E)
    m, Z = rows_of(plan, tr, 1, traj, prefix)
    with np.errstate(invalid="ignore"):
        want = m.sum(axis=1)
    odd = ~np.isfinite(m).all(axis=1)
    assert odd.any()
    assert np.array_equal(Z[odd], want[odd], equal_nan=True)
    np.testing.assert_allclose(Z[~odd], want[~odd], rtol=1e-12)


@pytest.mark.parametrize("mode,b", [(m, b) for m in ("square", "product") for b in range(1, 15) if m != "product" or b > 1])
def test_largest_entries_through_the_harvest(mode, b):
    circ, plan, tr = planned(mode, b)
    tau = 0.7 / (1 << b)
    res = ptn.ptn_sample_nonprop(plan, tr, 31, mode="exhaustive", threshold=tau)
    (rt, rb, rp), nets = sampling.nbs_nonproportional(lambda j, t, p: rows_of(plan, tr, j, t, p)[0], plan.blocks, 31, E,
                                                      mode="exhaustive", tau=tau)
    t, bits, _ = [x.cpu().numpy() for x in res.to_torch()]
    assert res.nets_per_block == nets and len(rt) > E // 2
    assert np.array_equal(t, rt) and np.array_equal(bits, np.asarray(rb).astype(np.int64))
    assert np.array_equal(res.probs().cpu().numpy(), rp)
