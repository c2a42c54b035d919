"""Small calls run on the staged kernels, larger ones on a thread per sample:
both give the same distances, accept sets and (exact) trajectories, bit for bit,
at the edges of blocks, stages and horizons (fast trajectories are always staged:
calls of different sizes agree); bands are the order statistics of the
trajectories at the edges of their two block shapes."""
import numpy as np
import pytest

from tests import inputs

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_2012_14332_gb300 as abc  # noqa: E402
from paper_2012_14332_gb300 import build as _build  # noqa: E402

_build.build()

BIG = 120_000   # more than one wave of staged blocks


def _series(T):
    d = np.arange(T + 1)
    return np.ascontiguousarray(np.stack([100 + 9 * d, 5 * d, d // 2]).astype(np.int32))


@pytest.mark.parametrize("mode", ["exact", "fast", "exact_literal", "fast_literal"])
@pytest.mark.parametrize("T", [1, 2, 5, 6, 7, 12, 49, 2500])
def test_small_calls_equal_the_large_ones(mode, T):
    P, seed = 10**6, 11
    obs = _series(T)
    big = BIG if T < 100 else 50_000
    d, th = abc.abc_distances(obs, P, big, seed, mode=mode, want_theta=True)
    for n in (1, 31, 32, 33, 1000):
        ds, ths = abc.abc_distances(obs, P, n, seed, mode=mode, want_theta=True)
        assert torch.equal(ds, d[:n]) and torch.equal(ths, th[:n]), n
        eps = float(torch.sort(ds)[0][n // 2])
        tha, da, ia, m = abc.abc_sample(obs, P, eps, n, seed, mode=mode, capacity=n)
        days = abc.abc_last_simulated_days()
        o = torch.argsort(ia)
        want = torch.nonzero(ds <= eps)[:, 0]
        assert m == len(want) and torch.equal(ia[o], want) and torch.equal(da[o], ds[want])
        assert torch.equal(tha[o], ths[want])
        assert 0 < days <= n * T
    idx = torch.arange(big, device="cuda") * 7
    step = max(1, T // 50)
    tr = abc.abc_simulate(th, idx, obs[:, 0], T, P, seed, mode=mode)
    for n in (1, 31, 33, 1000):
        ts = abc.abc_simulate(th[big - n:], idx[big - n:], obs[:, 0], T, P, seed, mode=mode)
        assert torch.equal(ts[:, ::step], tr[big - n:, ::step]) and torch.equal(ts[:, -1], tr[big - n:, -1]), n
    assert int(tr.sum(2).min()) == P == int(tr.sum(2).max())


@pytest.mark.parametrize("B", [1, 2, 32, 511, 512, 513, 4097, 8192])
@pytest.mark.parametrize("T", [1, 7, 60])
def test_bands_are_the_trajectories_order_statistics(B, T):
    """Columns of one value, of few values, and heavy-tailed ones; few quantiles
    (passed with the launch) and many (through device memory)."""
    th = torch.from_numpy(inputs.random_thetas(B, B)).cuda()
    idx = torch.arange(B, device="cuda") + 3
    tr = torch.sort(abc.abc_simulate(th, idx, [100, 3, 0], T, 300_000_000, 5, mode="fast")[:, :, 2:5], dim=0)[0]
    for q in (np.array([0.05, 0.5, 0.95]), np.linspace(0, 1, 33)):
        bands = abc.abc_project(th, idx, [100, 3, 0], T, 300_000_000, 5, quantiles=q, mode="fast")
        want = torch.stack([tr[int(np.floor(x * (B - 1)))] for x in q]).float()
        assert torch.equal(bands, want)
