"""Samples whose infected die out are dropped once they cannot be accepted: the
accept sets stay those of simulating every day, at thresholds that lie among
the died-out samples' distances, for series that such samples match, series
that outgrow them and series that fall."""
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

N, SEED = 3001, 77


def _series(kind, T, P):
    if kind == "died_out":      # a run whose infected died out
        th = np.array([0.05, 2.0, 1.0, 0.5, 0.6, 0.1, 0.5, 1.0], dtype=np.float32)
        return oracle.simulate(th, [100, 0, 0], T, P, 3, 1, 0)[:, 2:5].T
    d = np.arange(T + 1)
    if kind == "grows":
        return np.stack([100 + d ** 3, 20 * d * d, 3 * d])
    return np.stack([np.maximum(100 - 3 * d, 0), 40 * (d % 3), np.maximum(30 - d, 0) * (d > 0)])   # falls and jumps


@pytest.mark.parametrize("kind", ["died_out", "grows", "falls"])
@pytest.mark.parametrize("T", [1, 2, 3, 4, 5, 48, 49])
def test_accept_sets_are_those_of_every_day(kind, T):
    P = 10**6
    obs = np.ascontiguousarray(_series(kind, T, P).astype(np.int32))
    ref = oracle.abc(obs, P, 0.0, N, SEED, want_all=True, capacity=1)["dist_all"]
    srt = np.sort(ref)
    for k in (1, 2, 40, N // 4, N // 2, N - 1, N):
        for eps in (float(srt[k - 1]), float(np.nextafter(srt[k - 1], -np.inf))):
            if eps < 0:
                continue
            want = np.flatnonzero(ref <= eps)
            theta, dist, idx, n = abc.abc_sample(obs, P, eps, N, SEED, mode="exact", capacity=N)
            days = abc.abc_last_simulated_days()
            got = np.sort(idx.cpu().numpy())
            assert n == len(want) and np.array_equal(got, want), (k, n, len(want))
            assert np.array_equal(np.sort(dist.cpu().numpy()), np.sort(ref[want]))
            plan = abc.Plan([dict(observed=obs, N_pop=P, eps=eps, n_samples=N, stream=0, capacity=N),
                             dict(observed=obs, N_pop=P, eps=eps, n_samples=7, stream=0, capacity=N)], SEED, mode="exact")
            plan.run()
            _, _, pidx, pn, pdays = plan.results(0)
            assert pn == n and np.array_equal(np.sort(pidx.cpu().numpy()), want) and pdays == days
            plan.close()


def test_died_out_samples_are_dropped_and_fast_mode_keeps_its_accepts():
    """On a series that outgrows died-out samples most of their days are never
    simulated, and in fast mode too the accepts are those of the distances."""
    w = inputs.workload("region_6e7_T100")
    n = 1 << 16
    d = abc.abc_distances(w["observed"], w["P"], n, 5, mode="fast").cpu().numpy()
    eps = float(np.sort(d)[200])
    _, dist, idx, m = abc.abc_sample(w["observed"], w["P"], eps, n, 5, mode="fast", capacity=n)
    assert m == 201 and np.array_equal(np.sort(idx.cpu().numpy()), np.flatnonzero(d <= eps))
    # simulating every sample until its own sum passes eps^2 takes about 0.5 n T days
    assert abc.abc_last_simulated_days() < 0.35 * n * w["T"]
