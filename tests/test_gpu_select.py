"""The k-th smallest distance and the samples at or below a distance, against
numpy: around the sample's size and the tile's, ordered and tied inputs,
brackets that miss (the radix select then answers), unaligned arrays."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_2012_14332_gb300 as abc  # noqa: E402
from paper_2012_14332_gb300 import build as _build  # noqa: E402

_build.build()

KINDS = ["epidemic", "uniform", "rising", "falling", "equal", "two_values", "tied_middle", "spike", "with_inf", "tiny"]


def _values(kind, n):
    g = np.random.default_rng(n)
    if kind == "epidemic":
        return np.sqrt(np.floor(np.exp(np.minimum(36 + 3.5 * g.standard_normal(n), 43))))
    if kind == "uniform":
        return g.random(n)
    if kind == "rising":
        return np.arange(n, dtype=np.float64)
    if kind == "falling":
        return np.arange(n, 0, -1, dtype=np.float64) ** 2
    if kind == "equal":
        return np.full(n, 3.25)
    if kind == "two_values":
        return np.where(g.random(n) < 0.5, 1.0, 2.0)
    if kind == "tied_middle":       # one value holds most of the keys, others lie around it
        return np.where(g.random(n) < 0.9, 5.0, 10 * g.random(n))
    if kind == "spike":             # nearly all keys within one bin of a wide bracket, but not equal
        return np.where(np.arange(n) % 50 == 0, 1e6 * g.random(n), 7.0 + 1e-9 * g.random(n))
    if kind == "with_inf":
        return np.where(g.random(n) < 0.3, np.inf, g.random(n))
    return 5e-324 * g.integers(0, 1000, n)


@pytest.mark.parametrize("kind", KINDS)
@pytest.mark.parametrize("n", [1, 2, 255, 2047, 2048, 2049, 4097, 65_536, 300_001])
def test_kth_smallest_is_numpys(kind, n):
    v = _values(kind, n + 1)
    dev = torch.from_numpy(v).cuda()
    for part, x in ((dev[:n], v[:n]), (dev[1:], v[1:])):    # 16-byte aligned, and 8 bytes off
        s = np.sort(x)
        for k in sorted({1, 2, n // 1000 + 1, n // 7 + 1, n // 2 + 1, n - 1, n} & set(range(1, n + 1))):
            assert abc.abc_kth_smallest(part, k) == s[k - 1], (kind, n, k)


@pytest.mark.parametrize("kind", ["epidemic", "tied_middle", "with_inf"])
@pytest.mark.parametrize("n", [1, 63, 64, 255, 256, 257, 100_003])
def test_select_below_is_numpys(kind, n):
    v = _values(kind, n + 1)
    dev = torch.from_numpy(v).cuda()
    theta = torch.arange(8 * n, device="cuda", dtype=torch.float32).reshape(n, 8)
    for part, x in ((dev[:n], v[:n]), (dev[1:], v[1:])):
        s = np.sort(x)
        for eps in (0.0, float(s[n // 3]), float(s[n - 1])):
            want = np.flatnonzero(x <= eps)
            th, d, i, m = abc.abc_select_below(part, eps, first_index=5, theta=theta, capacity=n)
            o = torch.argsort(i)
            assert m == len(want) and np.array_equal(i[o].cpu().numpy(), want + 5)
            assert np.array_equal(d[o].cpu().numpy(), x[want])
            assert np.array_equal(th[o].cpu().numpy(), theta.cpu().numpy()[want])
        if n > 2:
            with pytest.raises(abc.AbcError) as e:
                abc.abc_select_below(part, float(s[n - 1]), capacity=n - 1)
            assert e.value.status == abc.binding.ABC_ERR_CAPACITY


@pytest.mark.parametrize("n", [1000, 5000, 300_001])
@pytest.mark.parametrize("bad", [float("nan"), -1.0, -0.0])
def test_invalid_keys_are_counted_wherever_they_lie(n, bad):
    v = np.random.default_rng(n).random(n)
    for at in (0, n // 2, n - 1):
        x = v.copy()
        x[at] = bad
        with pytest.raises(abc.AbcError) as e:
            abc.abc_kth_smallest(torch.from_numpy(x).cuda(), n // 2)
        assert e.value.status == abc.binding.ABC_ERR_INVALID_ARG and "1 distances" in e.value.message


def _zeros(kind, n):
    """Distances of exactly 0 in tiles of their own (a tile is 2048 keys)."""
    rest = 1.0 + np.random.default_rng(n).random(n)
    if kind == "all":
        return np.zeros(n)
    if kind == "lone_last":
        rest[n - 1] = 0.0
        return rest
    if kind == "rising_after_one":      # sorted input: one 0, then rising
        return np.arange(n, dtype=np.float64)
    lead = {"2048_first": 2048, "4096_first": 4096, "half_first": n // 2}[kind]
    return np.concatenate([np.zeros(min(lead, n)), np.sort(rest[min(lead, n):])])


@pytest.mark.parametrize("kind", ["all", "lone_last", "rising_after_one", "2048_first", "4096_first", "half_first"])
@pytest.mark.parametrize("n", [2049, 3000, 4096, 4097, 6145, 65_536, 98_305, 2_000_000])
def test_distances_of_exactly_zero_count_like_any_other(kind, n):
    """A block whose only candidates are zeros, few candidates (finished by one
    block) and many (binned first), ranks among the zeros, at their end and above."""
    v = _zeros(kind, n)
    s, dev = np.sort(v), torch.from_numpy(v).cuda()
    zeros = int((v == 0).sum())
    for k in sorted({1, 2, 14, 1000, 2000, 2300, zeros - 1, zeros, zeros + 1, n // 2, n - 1, n} & set(range(1, n + 1))):
        assert abc.abc_kth_smallest(dev, k) == s[k - 1], (kind, n, k)


@pytest.mark.parametrize("A0,T,n", [(0, 5, 3000), (0, 5, 70_000), (1, 1, 2049), (1, 2, 70_000), (2, 1, 200_000)])
def test_quantile_of_runs_that_match_the_series_exactly(A0, T, n):
    """A series without infections (every distance 0) and short ones of a few
    cases, which many runs match exactly."""
    obs = np.ascontiguousarray(np.tile([[A0], [0], [0]], (1, T + 1)).astype(np.int32))
    d = abc.abc_distances(obs, 10**6, n, 3, mode="exact")
    x = d.cpu().numpy()
    zeros = int((x == 0).sum())
    assert zeros > 0
    for k in sorted({1, zeros, min(zeros + 1, n), n // 2, n}):
        want = np.sort(x)[k - 1]
        _, _, idx, m, eps = abc.abc_sample_quantile(obs, 10**6, n, k, 3, mode="exact", capacity=n)
        assert eps == want and m == int((x <= want).sum())
        assert np.array_equal(np.sort(idx.cpu().numpy()), np.flatnonzero(x <= want))
