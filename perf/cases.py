"""What the framework is timed on: the calls its users make, at the sizes they make them.

A case is one call (or one short sequence of calls) through the public binding
``paper_2604_08467_gb300.ptn``.  The circuits are the repository's own
workload families (``workloads``): Haar brickwork with depolarizing and
amplitude damping noise, the 4-colour grid, the paper's random circuits, the
hardware-efficient ansatz.  Kinds of cases:

  contract  the marginals of a list of (trajectory, prefix) networks of one block
  sample    pre-sampling, proportional sampling and the records, a whole job
  nonprop   non-proportional sampling with an exhaustive final-block harvest
  draws     the conditional draws of one block from marginals the caller holds
  expval    a trajectory-averaged expectation value and its gradient
  amps      the amplitudes of every trajectory's state

A user keeps one plan per circuit and brings new error sets, prefixes, angles
or marginals to it, so the plan of a case is made once per process (``_plan``)
and everything a seed decides is made by ``prepare``.  ``exact`` recomputes the
floating results in complex128 with plain numpy and torch (its own Philox
draws, matrix product states for the 1D circuits, state vectors up to 16
qubits).
"""
import functools
import math

import numpy as np
import torch

import workloads as W
from paper_2604_08467_gb300 import autograd, ptn

PREC = {"fp32": ptn.PTN_PREC_FP32, "bf16x3": ptn.PTN_PREC_BF16X3, "fp16x3": ptn.PTN_PREC_FP16X3}


def listed():
    return [
        # The headline job: 30 qubits, depth 12, 4096 error sets, 10^6 shots (the benchmark's workload and plan options).
        {"name": "sample_30q", "kind": "sample", "family": "brick", "n": 30, "depth": 12, "b": 10, "search": 1000,
         "traj": 4096, "shots": 1000000, "per_traj": False, "precision": "fp16x3"},
        # Its three blocks on their own: the first block of every error set (no prefix yet), ...
        {"name": "block0_30q_fp32", "kind": "contract", "family": "brick", "n": 30, "depth": 12, "b": 10, "search": 1000,
         "block": 0, "traj": 1024, "draws": 1, "precision": "fp32"},
        # ... the middle block, which carries most of the arithmetic, ...
        {"name": "block1_30q_fp16x3", "kind": "contract", "family": "brick", "n": 30, "depth": 12, "b": 10, "search": 1000,
         "block": 1, "traj": 131, "draws": 244, "precision": "fp16x3"},
        # ... and the last block (amplitudes, then the sum over |a|^2), in the cheapest precision.
        {"name": "block2_30q_bf16x3", "kind": "contract", "family": "brick", "n": 30, "depth": 12, "b": 10, "search": 1000,
         "block": 2, "traj": 131, "draws": 244, "precision": "bf16x3"},
        # A small job end to end: 12 qubits, 64 error sets, 1000 shots each (latency, launches, host work).
        {"name": "sample_12q", "kind": "sample", "family": "brick", "n": 12, "depth": 8, "b": 10, "search": 100,
         "traj": 64, "shots": 1000, "per_traj": True, "precision": "fp32"},
        # One network of a middle block at the paper's 100 qubits / 600 gates: the latency of a single contraction, ...
        {"name": "block5_100q_1net", "kind": "contract", "family": "paper", "n": 100, "depth": 600, "b": 10, "search": 100,
         "block": 5, "traj": 1, "draws": 1, "precision": "fp32"},
        # ... and one network for each of 256 error sets.
        {"name": "block5_100q_256net", "kind": "contract", "family": "paper", "n": 100, "depth": 600, "b": 10, "search": 100,
         "block": 5, "traj": 256, "draws": 1, "precision": "fp16x3"},
        # The precision study's 16-qubit grid: its second block for 2048 error sets, a few prefixes each.
        {"name": "block1_grid16_fp32", "kind": "contract", "family": "grid", "n": 16, "depth": 10, "b": 10, "search": 100,
         "block": 1, "traj": 2048, "draws": 5, "precision": "fp32"},
        # Amplitudes of 300 error sets of the same grid (fidelities, observables the library does not have).
        {"name": "amps_grid16", "kind": "amps", "family": "grid", "n": 16, "depth": 10, "b": 10, "search": 100,
         "traj": 300, "precision": "fp32"},
        # A training step's gradient: 16-qubit ansatz, 6 layers, 192 angles, 1024 error sets, checkpointed.
        {"name": "expval_16q", "kind": "expval", "family": "hea", "n": 16, "depth": 6, "b": 10, "search": 100,
         "traj": 1024, "checkpoint": True},
        # Labelled data at the paper's 50 qubits / 200 gates: a 28-qubit final block harvested exhaustively.
        {"name": "nonprop_50q", "kind": "nonprop", "family": "paper", "n": 50, "depth": 200, "b": 10, "final": 28, "search": 100,
         "traj": 24, "threshold": 1e-6, "precision": "fp16x3"},
        # The sampling step of a caller that holds the marginals itself (a job sharded over processes).
        {"name": "draws_10bit", "kind": "draws", "b": 10, "parents": 150001, "traj": 701, "mean": 2.5},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["contract", "contract", "contract", "sample", "sample", "nonprop", "draws", "expval", "amps"])
    prec = rng.choice(sorted(PREC))
    if kind == "contract":
        family = rng.choice(["brick", "brick", "paper", "grid"])
        if family == "brick":
            n, b = rng.randint(20, 31), rng.randint(6, 11)
            return {"kind": kind, "family": family, "n": n, "depth": rng.randint(6, 12), "b": b, "search": 100,
                    "block": rng.randrange(-(-n // b)), "traj": _log(rng, 1, 400), "draws": _log(rng, 1, 200),
                    "precision": prec}
        if family == "paper":
            n = rng.randint(40, 120)
            return {"kind": kind, "family": family, "n": n, "depth": n * rng.randint(4, 6), "b": 10, "search": 100,
                    "block": rng.randrange(-(-n // 10)), "traj": _log(rng, 1, 1000), "draws": _log(rng, 1, 20),
                    "precision": prec}
        return {"kind": kind, "family": family, "n": 16, "depth": rng.randint(6, 10), "b": 10, "search": 100,
                "block": rng.randrange(2), "traj": _log(rng, 16, 2048), "draws": _log(rng, 1, 20), "precision": prec}
    if kind == "sample":
        per_traj = rng.random() < 0.5
        traj = _log(rng, 16, 2048)
        return {"kind": kind, "family": "brick", "n": rng.randint(8, 26), "depth": rng.randint(4, 10),
                "b": rng.randint(6, 10), "search": 100, "traj": traj,
                "shots": _log(rng, 2, 200) if per_traj else _log(rng, 1000, 200000), "per_traj": per_traj,
                "precision": prec}
    if kind == "nonprop":
        n = rng.randint(32, 50)
        return {"kind": kind, "family": "paper", "n": n, "depth": 4 * n, "b": 10, "final": rng.randint(16, 26),
                "search": 100, "traj": _log(rng, 2, 48), "threshold": 1e-6, "precision": prec}
    if kind == "draws":
        parents = _log(rng, 100, 150000)
        return {"kind": kind, "b": rng.randint(4, 12), "parents": parents, "traj": max(1, parents // rng.randint(1, 300)),
                "mean": rng.choice([1.5, 2.5, 20.0])}
    if kind == "expval":
        return {"kind": kind, "family": "hea", "n": rng.randint(8, 16), "depth": rng.randint(2, 6), "b": 8, "search": 100,
                "traj": _log(rng, 16, 1024), "checkpoint": rng.random() < 0.5}
    return {"kind": kind, "family": "brick", "n": rng.randint(9, 16), "depth": rng.randint(4, 10), "b": 8, "search": 100,
            "traj": _log(rng, 4, 300), "precision": prec}


# ------------------------------------------------------------------ inputs --

def _blocks(case):
    n, b = case["n"], case["b"]
    if "final" in case:
        n -= case["final"]
    sizes = [b] * (n // b) + ([n % b] if n % b else [])
    return sizes + ([case["final"]] if "final" in case else [])


def _circuit(case):
    n, depth = case["n"], case["depth"]
    rng = np.random.default_rng([n, depth])
    if case["family"] == "brick":
        return W.attach_noise(W.brickwork_1d(n, depth, rng), [W.depolarizing_kraus(0.005), W.amplitude_damping_kraus(0.002)])
    if case["family"] == "grid":
        return W.attach_noise(W.grid_4colour(4, n // 4, depth, rng), [W.depolarizing_kraus(0.003)])
    if case["family"] == "hea":
        return W.attach_noise(W.hea_ring(n, depth, rng.standard_normal(2 * n * depth)), [W.depolarizing_kraus(0.01)])
    return W.paper_random_circuit(n, depth, rng)


@functools.lru_cache(maxsize=1)
def _plan_of(items):
    case = dict(items)
    circ = _circuit(case)
    return circ, ptn.ptn_plan_path(circ, _blocks(case), hypersamples=case["search"], search_threads=8,
                                   est_traj=case["est_traj"], est_shots=case["est_shots"],
                                   mem_cap_bytes=80e9, grad_checkpoint=case["checkpoint"])


def _plan(case):
    """The circuit and its plan, as a program keeps them for all its calls (the benchmark's 30-qubit plan is made for 4096 error sets and 10^6 shots)."""
    big = case["search"] > 100
    per = case.get("draws", 1) if case["kind"] == "contract" else case.get("shots", 1) if case.get("per_traj") else 0
    shots = case["traj"] * per or case.get("shots", case["traj"])
    items = {k: case[k] for k in ("family", "n", "depth", "b", "final", "search") if k in case}
    items.update(est_traj=4096 if big else case["traj"], est_shots=1000000 if big else shots,
                 checkpoint=case.get("checkpoint", False))
    return _plan_of(tuple(sorted(items.items())))


def _seed(seed):
    """The Philox key of the error sets of one preparation."""
    return 0x5EED0000 + 7919 * int(seed)


def _kraus(circ, n_traj, key):
    """[n_traj, n_sites] Kraus indices: u = uniform53 of Philox4x32-10 (Salmon et al., SC'11) at counter
    (site, 0, trajectory, 1 << 24), the smallest k with u < q_0 + ... + q_k, q_k = Tr(K_k^dagger K_k) / d."""
    m32 = np.uint64(0xFFFFFFFF)
    site, traj = np.meshgrid(np.arange(circ.n_sites, dtype=np.uint64), np.arange(n_traj, dtype=np.uint64))
    c = [site, np.zeros_like(site), traj, np.full_like(site, 1 << 24)]
    k0, k1 = np.uint64(key & 0xFFFFFFFF), np.uint64(key >> 32)
    for _ in range(10):
        p0, p1 = np.uint64(0xD2511F53) * c[0], np.uint64(0xCD9E8D57) * c[2]
        c = [(p1 >> np.uint64(32)) ^ c[1] ^ k0, p1 & m32, (p0 >> np.uint64(32)) ^ c[3] ^ k1, p0 & m32]
        k0, k1 = (k0 + np.uint64(0x9E3779B9)) & m32, (k1 + np.uint64(0xBB67AE85)) & m32
    u = (((c[0] << np.uint64(32)) | c[1]) >> np.uint64(11)).astype(np.float64) * 2.0 ** -53
    out = np.empty((n_traj, circ.n_sites), np.int64)
    for s, st in enumerate(circ.sites):
        cdf = np.cumsum([np.sum(np.abs(k) ** 2) / k.shape[0] for k in circ.channels[st.channel].kraus])
        cdf[-1] = 1.0
        out[:, s] = np.searchsorted(cdf, u[:, s], side="right")
    return out


def _prefixes(case, circ, seed):
    """Distinct (trajectory, prefix) pairs below the case's block, in order: `draws` bitstrings sampled from every
    trajectory's own state (1D circuits), or uniform ones (the grid, whose outputs are close to uniform)."""
    start, n_traj, n_draw = sum(_blocks(case)[: case["block"]]), case["traj"], case["draws"]
    if start == 0:
        return torch.arange(n_traj), torch.zeros((n_traj, 0), dtype=torch.int64)
    gen = torch.Generator(device="cuda").manual_seed(int(seed))
    if case["family"] == "grid":
        bits = torch.randint(0, 2, (n_traj, n_draw, start), generator=gen, device="cuda")
    else:
        got = []
        kraus = _kraus(circ, n_traj, _seed(seed))
        for t0 in range(0, n_traj, 128):
            mps = _mps(circ, kraus[t0:t0 + 128])
            env = _right(mps)
            T, v, row = len(mps[0]), None, []
            for q in range(start):
                a = mps[q]
                v = v if v is not None else a.new_ones((T, n_draw, 1))
                both = torch.stack([v @ a[:, :, i] for i in range(2)])                     # [2, T, S, D]
                p = ((both @ env[q + 1]) * both.conj()).sum(-1).real
                one = torch.rand((T, n_draw), generator=gen, device="cuda", dtype=torch.float64) * p.sum(0) >= p[0]
                v = torch.where(one[..., None], both[1], both[0]) / torch.where(one, p[1], p[0]).sqrt()[..., None]
                row.append(one.to(torch.int64))
            got.append(torch.stack(row, -1))
        bits = torch.cat(got)
    traj = torch.arange(n_traj, device="cuda")[:, None, None].expand(n_traj, n_draw, 1)
    rows = torch.unique(torch.cat([traj, bits], -1).reshape(-1, 1 + start), dim=0).cpu()
    return rows[:, 0], rows[:, 1:]


def prepare(case, seed):
    kind = case["kind"]
    if kind == "draws":
        gen = torch.Generator(device="cuda").manual_seed(int(seed))
        n, b = case["parents"], case["b"]
        marg = torch.empty((n, 1 << b), device="cuda").exponential_(generator=gen)   # Porter-Thomas rows of many scales
        marg *= torch.exp(-12 * torch.rand((n, 1), generator=gen, device="cuda"))
        marg[torch.rand((n, 1 << b), generator=gen, device="cuda") < 0.1] = 0.0
        marg[:, 0] += 1e-6
        traj = (torch.arange(n, device="cuda") * case["traj"] // n).to(torch.int32)
        prefix = torch.arange(n, device="cuda", dtype=torch.int64) & 0x3FF
        u = torch.rand(n, generator=gen, device="cuda", dtype=torch.float64)
        count = 1 + torch.floor(torch.log1p(-u) / math.log1p(-1.0 / case["mean"])).to(torch.int64)
        return dict(case=case, marg=marg, traj=traj, prefix=prefix, count=count, seed=_seed(seed),
                    out=_buffers(int(1.25 * n * case["mean"]) + 4096, torch.int32, torch.int64, torch.int64))
    circ, plan = _plan(case)
    s = dict(case=case, plan=plan, seed=_seed(seed))
    if kind in ("contract", "amps", "expval"):
        s["traj"] = ptn.ptn_presample_trajectories(plan, s["seed"], case["traj"])
    if kind == "contract":
        traj, bits = _prefixes(case, circ, seed)
        words = ptn.words_of(case["n"])
        prefix = np.zeros((len(traj), words), np.uint64)
        for q in range(bits.shape[1]):
            prefix[:, q // 64] |= bits[:, q].numpy().astype(np.uint64) << np.uint64(q % 64)
        s["net_traj"] = traj.to("cuda", torch.int32)
        s["net_prefix"] = torch.from_numpy(prefix.view(np.int64)).cuda().reshape(-1)
        s["marg"] = torch.zeros((case["traj"] * case["draws"], 1 << _blocks(case)[case["block"]]), device="cuda")
        s["Z"] = torch.zeros(len(s["marg"]), dtype=torch.float64, device="cuda")
    elif kind == "amps":
        s["amp"] = torch.empty((case["traj"], 1 << case["n"]), dtype=torch.complex64, device="cuda")
    elif kind == "expval":
        n = case["n"]
        s["terms"] = [(1.0 / n, (1 << q) | (1 << (q + 1) % n)) for q in range(n)]
        s["theta"] = torch.from_numpy(_theta(case, seed)).cuda().requires_grad_()
    elif kind == "sample":
        s["out"] = _buffers(case["shots"] * (case["traj"] if case["per_traj"] else 1), torch.int32, torch.int64, torch.int64)
    elif kind == "nonprop":
        s["out"] = _buffers(int(case["traj"] / case["threshold"]), torch.int32, torch.int64, torch.int64, torch.float64)
    return s


def _buffers(n, *types):
    """The arrays that a program collects records in, as long as the largest number of records that it expects."""
    return [torch.zeros(n, dtype=t, device="cuda") for t in types]


def _keep(records, out):
    for r, o in zip(records, out):
        o[: len(r)].copy_(r)
    return [len(records[0])] + out


def _theta(case, seed):
    return np.random.default_rng(int(seed)).standard_normal(2 * case["n"] * case["depth"]).astype(np.float32)


# --------------------------------------------------------------------- run --

def run(s):
    case = s["case"]
    kind = case["kind"]
    if kind == "contract":
        ptn.ptn_contract_batch(s["plan"], s["traj"], case["block"], s["net_traj"], s["net_prefix"], s["marg"], s["Z"],
                               precision=PREC[case["precision"]])
        return s["marg"], s["Z"].float()   # Z is a sum of FP32 marginals: FP32 holds all that it says
    if kind == "draws":
        n = ptn.ptn_sample_block(s["marg"], case["b"], 10, s["traj"], s["prefix"], s["count"], s["seed"], 0, 1, *s["out"])
        return [n] + s["out"]
    if kind == "amps":
        ptn.ptn_trajectory_amplitudes(s["plan"], s["traj"], 0, case["traj"], s["amp"], precision=PREC[case["precision"]])
        return s["amp"]
    if kind == "expval":
        value = autograd.trajectory_expval(s["theta"], s["plan"], s["traj"], s["terms"])
        return value.detach(), torch.autograd.grad(value, s["theta"])[0]
    tr = ptn.ptn_presample_trajectories(s["plan"], s["seed"], case["traj"])
    if kind == "sample":
        shots = {"shots_per_traj" if case["per_traj"] else "total_shots": case["shots"]}
        got = ptn.ptn_sample_shots(s["plan"], tr, s["seed"] + 1, precision=PREC[case["precision"]], **shots)
        return _keep(got.to_torch(), s["out"]) + [tr.to_torch()[1]]
    got = ptn.ptn_sample_nonprop(s["plan"], tr, s["seed"] + 1, threshold=case["threshold"], precision=PREC[case["precision"]])
    return _keep(got.to_torch() + (got.probs(),), s["out"])


def work(case):
    """Bytes: what the call is given and what it returns.  Operations: the pairwise contractions of the circuit's path
    (8 per complex multiply-add), once per error set or per network as the path has them."""
    kind = case["kind"]
    if kind == "draws":
        return {"bytes": case["parents"] * (4.0 * (1 << case["b"]) + 20 + 20 * case["mean"]), "flops": 0.0}
    circ, plan = _plan(case)
    sets = case["traj"] * circ.n_sites
    if kind == "amps":
        return {"bytes": sets + 8.0 * case["traj"] * (1 << case["n"]), "flops": 8.0 * case["traj"] * len(circ.gates) * (1 << case["n"])}
    if kind == "expval":   # forward, adjoint of the state and of the angles
        return {"bytes": sets + 12.0 * len(circ.gates), "flops": 24.0 * case["traj"] * len(circ.gates) * (1 << case["n"])}
    macs, nets = 0.0, case["traj"]
    blocks = plan.describe()["blocks"]
    for j, blk in enumerate(blocks):
        if kind == "sample" and j:
            nets = min(case["traj"] << blk["start"], case["shots"] * (case["traj"] if case["per_traj"] else 1))
        if kind == "contract":
            nets = min(case["traj"] * case["draws"], case["traj"] << blk["start"])
        if kind != "contract" or j == case["block"]:
            macs += blk["macs_traj"] / blk["mult_traj"] * case["traj"] + blk["macs_net"] / blk["mult_net"] * nets
    if kind == "contract":
        out = nets * (4.0 * (1 << blocks[case["block"]]["b"]) + 8)
    else:
        out = (20.0 if kind == "sample" else 28.0) * (nets if kind == "sample" else nets * 1e4)
    return {"bytes": sets + out, "flops": 8.0 * macs}


# ------------------------------------------------------------------- exact --

def _ops(circ):
    """Per gate, its noise in order: (site, qubit or -1, the operators K_k / sqrt(q_k) as one tensor)."""
    per = [[] for _ in circ.gates]
    for s, st in enumerate(circ.sites):
        ks = [np.asarray(k) / np.sqrt(np.sum(np.abs(k) ** 2) / k.shape[0]) for k in circ.channels[st.channel].kraus]
        per[st.gate].append((s, st.qubit, np.stack(ks)))
    return per


def _product(ks):
    """Factors of operators that are tensor products (a two-qubit Pauli error): K = A (x) B."""
    a, b = [], []
    for k in ks:
        u, sv, vh = np.linalg.svd(k.reshape(2, 2, 2, 2).transpose(0, 2, 1, 3).reshape(4, 4))
        assert sv[1] < 1e-12 * sv[0]
        a.append((u[:, 0] * sv[0]).reshape(2, 2))
        b.append(vh[0].reshape(2, 2))
    return np.stack(a), np.stack(b)


def _mps(circ, kraus):
    """Matrix product states of the trajectories, [T, left, 2, right] per qubit, exact: every two-qubit gate multiplies
    its bond by the number of terms of its operator-Schmidt decomposition."""
    T = len(kraus)
    idx = torch.from_numpy(kraus).cuda()
    cuda = lambda x: torch.from_numpy(np.ascontiguousarray(x)).cuda()   # noqa: E731
    zero = torch.zeros((T, 1, 2, 1), dtype=torch.complex128, device="cuda")
    zero[:, :, 0] = 1
    t = [zero] * circ.n_qubits
    one = lambda q, m: torch.einsum("toi,tlir->tlor", m.expand(T, 2, 2), t[q])   # noqa: E731
    for g, noise in zip(circ.gates, _ops(circ)):
        if g.arity == 1:
            t[g.qubits[0]] = one(g.qubits[0], cuda(g.matrix))
        else:
            u, sv, vh = np.linalg.svd(g.matrix.reshape(2, 2, 2, 2).transpose(0, 2, 1, 3).reshape(4, 4))
            r = int(np.sum(sv > 1e-12 * sv[0]))
            for q, f in ((g.qubits[0], (u[:, :r] * sv[:r]).T), (g.qubits[1], vh[:r])):
                x = torch.einsum("koi,tlir->ktlor", cuda(f.reshape(r, 2, 2)), t[q])
                right = q == min(g.qubits)     # the new index joins this site's right bond, the other's left bond
                x = x.permute(1, 2, 3, 4, 0) if right else x.permute(1, 2, 0, 3, 4)
                t[q] = x.reshape(T, x.shape[1], 2, -1) if right else x.reshape(T, -1, 2, x.shape[4])
        for s, q, ks in noise:
            for qq, f in ((q, ks),) if q >= 0 else zip(g.qubits, _product(ks)):
                t[qq] = one(qq, cuda(f)[idx[:, s]])
    return t


def _right(mps):
    """env[q]: the trace over qubits q, q + 1, ... as a matrix on the bond left of q."""
    env = [None] * len(mps) + [mps[0].new_ones((len(mps[0]), 1, 1))]
    for q in range(len(mps) - 1, -1, -1):
        env[q] = sum(mps[q][:, :, i] @ env[q + 1] @ mps[q][:, :, i].mH for i in range(2))
    return env


def _states(circ, kraus, theta=None):
    """State vectors [T, 2^n] of the trajectories (qubit q is bit q)."""
    n, T = circ.n_qubits, len(kraus)
    idx = torch.from_numpy(kraus).cuda()
    psi = torch.zeros([T] + [2] * n, dtype=torch.complex128, device="cuda")
    psi.view(T, -1)[:, 0] = 1
    ax = lambda q: n - q   # noqa: E731

    def one(psi, q, m):
        m = m.expand(T, 2, 2).reshape([T, 2, 2] + [1] * (n - 1))
        x = psi.movedim(ax(q), 1)
        return (m[:, :, 0] * x[:, :1] + m[:, :, 1] * x[:, 1:]).movedim(1, ax(q))

    for g, noise in zip(circ.gates, _ops(circ)):
        if g.arity == 2:   # CZ on the grid and the ring
            assert np.allclose(g.matrix, np.diag([1, 1, 1, -1]))
            sign = torch.ones([1] + [2] * n, device="cuda", dtype=torch.float64)
            sign.movedim((ax(g.qubits[0]), ax(g.qubits[1])), (0, 1))[1, 1] = -1
            psi = psi * sign
            local = {q: torch.eye(2, dtype=torch.complex128, device="cuda") for q in g.qubits}
        else:
            m = torch.from_numpy(g.matrix).cuda()
            if theta is not None and g.param_kind != W.PARAM_NONE:
                h = theta[g.param_index] / 2
                c, s_, z = torch.cos(h), torch.sin(h), torch.zeros_like(h)
                m = (torch.stack([c, -s_, s_, c]).to(torch.complex128) if g.param_kind == W.PARAM_RY else
                     torch.stack([torch.complex(c, -s_), torch.complex(z, z), torch.complex(z, z), torch.complex(c, s_)])).reshape(2, 2)
            local = {g.qubits[0]: m}
        for s, q, ks in noise:
            local[q] = torch.from_numpy(ks).cuda()[idx[:, s]] @ local[q]
        for q, m in local.items():
            psi = one(psi, q, m)
    return psi.reshape(T, -1)


def exact(case, seed):
    kind, key = case["kind"], _seed(seed)
    if kind in ("draws", "nonprop"):
        return None
    circ = _circuit(case)
    kraus = _kraus(circ, case["traj"], key)
    if kind == "sample":   # the records are whole numbers; log q of every error set is computed
        logq = np.zeros(case["traj"])
        for s, st in enumerate(circ.sites):
            logq += np.log([np.sum(np.abs(k) ** 2) / k.shape[0] for k in circ.channels[st.channel].kraus])[kraus[:, s]]
        return [None, None, None, None, torch.from_numpy(logq)]
    if kind == "amps":
        return torch.cat([_states(circ, kraus[t:t + 64]) for t in range(0, len(kraus), 64)])
    if kind == "expval":
        theta = torch.from_numpy(_theta(case, seed)).double().cuda().requires_grad_()
        x = torch.arange(1 << case["n"], device="cuda")
        w = sum((1 - 2 * ((x >> q) & 1)) * (1 - 2 * ((x >> (q + 1) % case["n"]) & 1)) for q in range(case["n"])) / case["n"]
        value = 0.0
        for t in range(0, case["traj"], 16):
            v = (_states(circ, kraus[t:t + 16], theta).abs() ** 2 * w).sum() / case["traj"]
            v.backward()
            value += v.item()
        return torch.tensor(value, dtype=torch.float64), theta.grad
    traj, bits = (x.cuda() for x in _prefixes(case, circ, seed))
    start, b = sum(_blocks(case)[: case["block"]]), _blocks(case)[case["block"]]
    out = torch.zeros((case["traj"] * case["draws"], 1 << b), dtype=torch.float64, device="cuda")
    for t0 in range(0, case["traj"], 64):
        if case["family"] == "grid":
            p = (_states(circ, kraus[t0:t0 + 64]).abs() ** 2).reshape(-1, 1 << (case["n"] - start - b), 1 << b, 1 << start).sum(1)
        else:
            mps = _mps(circ, kraus[t0:t0 + 64])
            env = _right(mps)[start + b]
        for t in range(t0, min(t0 + 64, case["traj"])):
            rows = torch.nonzero(traj == t)[:, 0]
            if case["family"] == "grid":
                s = (bits[rows] << torch.arange(start, device="cuda")).sum(-1)
                out[rows] = p[t - t0][:, s].T
                continue
            v = torch.ones((len(rows), 1, 1), dtype=torch.complex128, device="cuda")
            for q in range(start):
                a = mps[q][t - t0]
                v = torch.where(bits[rows, q].bool()[:, None, None], v @ a[:, 1], v @ a[:, 0])
            for q in range(start, start + b):
                a = mps[q][t - t0]
                v = torch.cat([v @ a[:, 0], v @ a[:, 1]], 1)
            out[rows] = ((v @ env[t - t0]) * v.conj()).sum(-1).real
    return out, out.sum(1)
