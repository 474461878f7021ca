"""Parents with few shots draw without a full CDF (k_sample_few); the draws must
be those of the exact-integer rule for every block size and row the warp
samplers take: shot counts around the line between the two kernels, rows with
zeros, negatives, NaN, subnormal and very large entries, one nonzero bin, and
marginals that do not start on a 16-byte boundary."""
import numpy as np
import pytest

import workloads as W
from oracle import sampling

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2604_08467_gb300 import ptn  # noqa: E402


def rows_of(n, b, seed):
    rows = W.synthetic_marginals(n, b, seed=seed)
    rng = np.random.default_rng(seed)
    rows[0] = 0.0                                    # zero-norm row: nothing is drawn
    rows[1] = 0.0
    rows[1, -1] = 1e-45                              # one subnormal bin
    rows[2] = -1.0
    rows[2, rng.integers(1 << b)] = 3.0e38           # one bin, the rest negative
    rows[3, :: 2] = np.nan
    rows[4] *= 1e-30
    rows[5] = np.exp(rng.uniform(-90, 80, 1 << b)).astype(np.float32)   # quantisation rounds most bins
    rows[6] = 1.0
    return rows


@pytest.mark.parametrize("b", [6, 7, 8, 9, 10])
@pytest.mark.parametrize("shift", [0, 1])
def test_few_shots_match_the_rule(b, shift):
    n = 45
    rows = rows_of(n, b, seed=b)
    counts = np.array([0, 1, 2, 3, 15, 16, 17, 33, 200][:9] * 5, dtype=np.int64)
    counts[:7] = [5, 3, 16, 4, 16, 16, 1]
    traj = np.arange(n) // 3
    prefix = np.arange(n, dtype=np.int64)
    buf = torch.empty(n << b, device="cuda") if not shift else torch.empty((n << b) + 1, device="cuda")[1:]
    buf.copy_(torch.from_numpy(rows.reshape(-1)))
    cap = int(np.minimum(counts, 1 << b).sum())
    ct, cp, cc = (torch.full((cap,), -7, dtype=t, device="cuda") for t in (torch.int32, torch.int64, torch.int64))
    nc = ptn.ptn_sample_block(buf, b, 3, torch.tensor(traj, dtype=torch.int32, device="cuda"),
                              torch.tensor(prefix & 7, device="cuda"), torch.tensor(counts, device="cuda"), 77, 2, 1,
                              ct, cp, cc)
    clean = np.where(rows > 0, rows, 0).astype(np.float32)
    par, xs, cs = sampling.sample_block(clean.astype(np.float64), traj, counts, sampling.rank_offsets(traj, counts), 77, 1,
                                        circuit=2)
    assert nc == len(cs)
    assert np.array_equal(cp[:nc].cpu().numpy(), (prefix[par] & 7) | (xs << 3))
    assert np.array_equal(cc[:nc].cpu().numpy(), cs)
    assert np.array_equal(ct[:nc].cpu().numpy(), traj[par])
    assert bool((cc[nc:] == -7).all())
