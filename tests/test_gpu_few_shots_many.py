"""Calls of many parents, where parents of few shots draw in registers
(k_sample_few) and the others by a warp each: the draws must be those of the
exact-integer rule, and those of calls of at most 300 parents, which take a CTA
each.  Parent counts past the line between the two forms (304) that do not fill a
CTA, and enough for several parents per look of a warp; the rows of the few-shot
test, and rows with infinite entries; marginals off a 16-byte boundary."""
import numpy as np
import pytest

from oracle import sampling
from test_gpu_few_shots import rows_of

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2604_08467_gb300 import ptn  # noqa: E402

DRAWN = [0, 1, 2, 3, 15, 16, 17, 33, 200]


def case(n, b, infinite):
    base = rows_of(45, b, seed=b)
    rows = np.tile(base, (-(-n // 45), 1))[:n]
    if infinite:
        rows[7::45, 3] = np.inf
        rows[8::45, :: 3] = np.inf
    counts = np.resize(np.array(DRAWN, dtype=np.int64), n)
    counts[:7] = [5, 3, 16, 4, 16, 16, 1]
    return rows, counts, np.arange(n) // 3      # three parents of a trajectory


def sample(rows, counts, traj, b, shift):
    n = len(counts)
    buf = torch.empty((n << b) + shift, device="cuda")[shift:]
    buf.copy_(torch.from_numpy(np.ascontiguousarray(rows).reshape(-1)))
    cap = int(np.minimum(counts, 1 << b).sum())
    ct, cp, cc = (torch.full((cap,), -7, dtype=t, device="cuda") for t in (torch.int32, torch.int64, torch.int64))
    nc = ptn.ptn_sample_block(buf, b, 3, torch.tensor(traj, dtype=torch.int32, device="cuda"),
                              torch.arange(n, device="cuda") & 7, torch.tensor(counts, device="cuda"), 77, 2, 1,
                              ct, cp, cc)
    assert bool((cc[nc:] == -7).all())
    return [x[:nc].cpu().numpy() for x in (ct, cp, cc)]


@pytest.mark.parametrize("b", [6, 7, 8, 9, 10])
@pytest.mark.parametrize("shift", [0, 1])
@pytest.mark.parametrize("n", [305, 317])
def test_many_parents_match_the_rule(b, shift, n):
    rows, counts, traj = case(n, b, False)
    t, p, c = sample(rows, counts, traj, b, shift)
    clean = np.where(rows > 0, rows, 0).astype(np.float64)
    par, xs, cs = sampling.sample_block(clean, traj, counts, sampling.rank_offsets(traj, counts), 77, 1, circuit=2)
    assert np.array_equal(c, cs) and np.array_equal(t, traj[par])
    assert np.array_equal(p, (par & 7) | (xs << 3))


@pytest.mark.parametrize("b", [6, 7, 8, 9, 10])
@pytest.mark.parametrize("shift", [0, 1])
@pytest.mark.parametrize("n", [317, 5003])
def test_many_parents_equal_few(b, shift, n):
    rows, counts, traj = case(n, b, True)
    got = sample(rows, counts, traj, b, shift)
    parts = []
    for lo in range(0, n, 288):                  # whole trajectories; 288 % 8 == 0 keeps the prefixes
        s = slice(lo, min(lo + 288, n))
        parts.append(sample(rows[s], counts[s], traj[s], b, shift))
    for k, a in enumerate(got):
        assert np.array_equal(a, np.concatenate([x[k] for x in parts]))
