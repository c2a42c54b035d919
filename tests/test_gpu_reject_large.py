"""Rejection calls above the staged kernels' reach (a thread per sample, lanes
refilled as samples end): the whole accept set equals the set of distances at or
below eps, in every mode, below 2^62, between 2^62 and 2^63 and at the cap, on
series that died-out samples match, outgrow and undercut; the simulated days are
those of the staged kernels over the same indices. And trajectories of every mode
against the one-day kernel, day by day."""
import numpy as np
import pytest

import oracle
from tests import inputs

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_2012_14332_gb300 as abc  # noqa: E402
from paper_2012_14332_gb300 import build as _build  # noqa: E402

_build.build()

N, PART, SEED = 400_000, 20_000, 91     # three waves of staged blocks hold fewer than 320,000 samples
MODES = ["exact", "fast", "exact_literal", "fast_literal"]
TOP = float(np.sqrt(np.float64(2.0**63)))


def _series(kind):
    """(observed, population)"""
    if kind == "top":       # differences of 2^31: sums cross 2^62 and 2^63
        obs = np.zeros((3, 3))
        obs[:, 0] = [10**9, 0, 0]
        obs[:, 1:] = np.array([[0], [2 * 10**9], [10**9]])
        return obs, 2**31 - 1
    d = np.arange(50)
    if kind == "died_out":
        th = np.array([0.05, 2.0, 1.0, 0.5, 0.6, 0.1, 0.5, 1.0], dtype=np.float32)
        return oracle.simulate(th, [100, 0, 0], 49, 10**6, 3, 1, 0)[:, 2:5].T, 10**6
    if kind == "grows":
        return np.stack([100 + d ** 3, 20 * d * d, 3 * d]), 10**7
    return np.stack([np.maximum(100 - 3 * d, 0), 40 * (d % 3), np.maximum(30 - d, 0) * (d > 0)]), 10**6


@pytest.mark.parametrize("mode", MODES)
@pytest.mark.parametrize("kind", ["died_out", "grows", "falls", "top"])
def test_accept_sets_of_large_calls(kind, mode):
    obs, P = _series(kind)
    obs = np.ascontiguousarray(obs.astype(np.int32))
    d, th = abc.abc_distances(obs, P, N, SEED, mode=mode, want_theta=True)
    srt = torch.sort(d)[0]
    eps = [float(srt[k]) for k in (300, N // 100, N // 2)]
    if kind == "top":
        eps += [2.0**31 - 0.5, float(srt[3 * N // 4]), TOP]
        assert 2.0**31 < eps[-2] < TOP and float(srt[-1]) == TOP
    for e in eps:
        want = torch.nonzero(d <= e)[:, 0]
        theta, dist, idx, n = abc.abc_sample(obs, P, e, N, SEED, mode=mode, capacity=N)
        days = abc.abc_last_simulated_days()
        o = torch.argsort(idx)
        assert n == len(want) and torch.equal(idx[o], want), (kind, mode, e, n, len(want))
        assert torch.equal(dist[o], d[want]) and torch.equal(theta[o], th[want])
        staged = 0
        for first in range(0, N, PART):
            abc.abc_sample(obs, P, e, PART, SEED, mode=mode, first_index=first, capacity=PART)
            staged += abc.abc_last_simulated_days()
        assert days == staged, (kind, mode, e)


@pytest.mark.parametrize("mode", MODES)
@pytest.mark.parametrize("B", [33, 60_000])
def test_trajectories_are_chains_of_single_days(mode, B):
    """Every day of every trajectory is the one-day kernel's from the day before."""
    P, T = 10**6, 17
    th = torch.from_numpy(inputs.random_thetas(B, B)).cuda()
    idx = torch.arange(B, device="cuda") * 3 + 1
    tr = abc.abc_simulate(th, idx, [100, 3, 1], T, P, SEED, mode=mode)
    for day in range(1, T + 1):
        nxt, _ = abc.abc_step(th, tr[:, day - 1].contiguous(), idx,
                              torch.full((B,), day, dtype=torch.int32, device="cuda"), P, SEED, mode=mode)
        assert torch.equal(nxt, tr[:, day]), day
