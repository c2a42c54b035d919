"""The performance cases: the work a user of this framework has it do, through
the package's public entry points.

Each case names a family (``kind``) and its sizes. The families and what they
stand for in real use:

  sample    ABC rejection at a fixed tolerance (abc_sample): from a ten-thousand
            draw exploratory call to the 2^24-draw production launch
  quantile  ABC rejection at a distance quantile in one call (abc_sample_quantile)
  select    a tolerance picked from distances already on the device
            (abc_kth_smallest) and the samples at or below it (abc_select_below)
  simulate  trajectories of accepted samples replayed in full (abc_simulate)
  project   posterior-predictive bands over a 120-day horizon (abc_project): the
            paper's 100 accepted samples, and the largest call the ABI takes
  regions   several regions with their own population, horizon and tolerance in
            one persistent launch replayed from a CUDA graph (Plan)
  flow_*    the learned proposal: drawing proposals with their density (Flow.sample),
            the density at given points (Flow.log_q), and training steps
            (Flow.train, Flow.train_flows)
  pmc       population Monte Carlo importance weights (abc_pmc_weights)

Inputs come from the seed alone. Observed series are epidemics of the six
compartment model simulated here with numpy. A tolerance is a distance quantile
of the batch that will be sampled, so that every seed accepts the same number.
Sampling returns accepted samples in an unspecified order, so a pass sorts them
by sample index, as the interface advises for a canonical order.
"""
import math

import numpy as np
import torch

import paper_2012_14332_gb300 as abc

LO = np.zeros(8)
HI = np.array([1, 100, 2, 1, 1, 1, 1, 2], dtype=np.float64)   # the default prior box
A0 = 100            # detected cases on the first day
DAY_OPS = 144       # operations of one simulated day: random words, normals, hazards, transitions, distance


def listed():
    return [
        # an exploratory call on a small region: launch latency and one short wave
        dict(name="sample_small", kind="sample", n=10_000, P=10**6, T=49, mode="exact", q=1e-2),
        # the production launch: 2^24 prior draws of a country-sized region, about 1e-4 accepted
        dict(name="sample_large", kind="sample", n=1 << 24, P=6 * 10**7, T=100, mode="fast", q=1e-4),
        # 65,536 draws, tolerance at the 0.1 % quantile, bit-reproducible arithmetic
        dict(name="quantile", kind="quantile", n=65_536, P=10**6, T=49, mode="exact", q=1e-3),
        # a tolerance for distances kept from an earlier batch, ragged length
        dict(name="select", kind="select", n=20_000_003, q=1e-4),
        # every trajectory of a large accepted set, ragged length, default arithmetic
        dict(name="simulate", kind="simulate", B=100_003, P=6 * 10**7, T=90, mode="exact"),
        # the paper's projection: 100 accepted samples, 120 days, 5 / 50 / 95 % bands
        dict(name="project_small", kind="project", B=100, P=6 * 10**7, T=120, mode="fast"),
        # the largest projection the interface takes
        dict(name="project_large", kind="project", B=8192, P=6 * 10**7, T=120, mode="fast"),
        # three regions of 2^22 draws each, populations 1e7 to 3.3e8, horizons 60 to 120 days
        dict(name="regions", kind="regions", regions=3, n=1 << 22, P_min=10**7, P_max=330_000_000, T_min=60,
             T_max=120, mode="fast", q=1e-4),
        # a learned round's proposals: 90 % of 2^22 with their densities
        dict(name="flow_sample", kind="flow_sample", n=3_774_873, blocks=3, hidden=256, tau=1.25),
        # a learned round's defensive draws: the flow's density at 10 % of 2^22 points
        dict(name="flow_log_q", kind="flow_log_q", n=419_431, blocks=3, hidden=256, tau=1.25),
        # a round's training: Adam steps on batches of 4096 weighted accepted samples
        dict(name="flow_train", kind="flow_train", flows=1, points=20_001, blocks=3, hidden=256, batch=4096, steps=50),
        # weights of a population against the previous one, ragged sizes
        dict(name="pmc_weights", kind="pmc", n=12_289, m=8_195),
    ]


def _log_int(rng, lo, hi):
    """A whole number spread over the logarithm of [lo, hi]."""
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["sample", "sample", "quantile", "select", "simulate", "project", "project", "regions",
                       "flow_sample", "flow_log_q", "flow_train", "pmc"])
    P, T, mode = _log_int(rng, 10**6, 330_000_000), rng.randint(30, 180), rng.choice(["exact", "fast"])
    if kind == "sample":
        return dict(kind=kind, n=_log_int(rng, 4_000, 1 << 22 if mode == "fast" else 1 << 20), P=P, T=T, mode=mode,
                    q=math.exp(rng.uniform(math.log(1e-4), math.log(1e-2))))
    if kind == "quantile":
        return dict(kind=kind, n=_log_int(rng, 4_000, 1 << 21 if mode == "fast" else 1 << 19), P=P, T=T, mode=mode,
                    q=math.exp(rng.uniform(math.log(1e-3), math.log(1e-2))))
    if kind == "select":
        return dict(kind=kind, n=_log_int(rng, 10_000, 40_000_000), q=math.exp(rng.uniform(math.log(1e-5), math.log(0.1))))
    if kind == "simulate":
        return dict(kind=kind, B=_log_int(rng, 100, 200_000), P=P, T=T, mode=mode)
    if kind == "project":
        return dict(kind=kind, B=_log_int(rng, 20, 8192), P=P, T=T, mode=mode)
    if kind == "regions":
        return dict(kind=kind, regions=rng.randint(2, 16), n=_log_int(rng, 20_000, 500_000), P_min=10**6,
                    P_max=_log_int(rng, 10**7, 330_000_000), T_min=rng.randint(30, 90), T_max=rng.randint(91, 180),
                    mode=mode, q=1e-3)
    if kind == "pmc":
        return dict(kind=kind, n=_log_int(rng, 500, 40_000), m=_log_int(rng, 500, 40_000))
    blocks, hidden = rng.randint(2, 4), 16 * rng.randint(4, 16)
    if kind == "flow_sample":
        return dict(kind=kind, n=_log_int(rng, 2_000, 4_000_000), blocks=blocks, hidden=hidden,
                    tau=rng.choice([1.0, 1.25]))
    if kind == "flow_log_q":
        return dict(kind=kind, n=_log_int(rng, 2_000, 4_000_000), blocks=blocks, hidden=hidden,
                    tau=rng.choice([1.0, 1.25]))
    flows = rng.choice([1, 1, 4, 16])
    return dict(kind=kind, flows=flows, points=_log_int(rng, 500, 100_000), blocks=blocks, hidden=hidden,
                batch=_log_int(rng, 512, 4096 if flows == 1 else 2048), steps=rng.randint(10, 50 if flows < 16 else 30))


# ---------------------------------------------------------------------------
# Inputs
# ---------------------------------------------------------------------------
def _epidemic(g, P, T):
    """(theta, observed [3, T + 1]): a seeded epidemic of the model from A0 cases,
    the first of a block of prior draws that grows but leaves half the population."""
    while True:
        th = LO + (HI - LO) * g.random((256, 8))
        a0, a, n, beta, gamma, delta, eta, kappa = th.T
        I, A = np.floor(kappa * A0), np.full(256, float(A0))
        R, D, S = np.zeros(256), np.zeros(256), P - A0 - np.floor(kappa * A0)
        days = [np.stack([A, R, D])]
        for _ in range(T):
            g_rate = a0 + a / (1 + (A + R + D) ** n)
            h = np.stack([g_rate * S * I / P, gamma * I, beta * A, delta * A, beta * eta * I])
            x = np.maximum(np.floor(h + np.sqrt(h) * g.standard_normal((5, 256))), 0)
            si, ia = np.minimum(x[0], S), np.minimum(x[1], I)
            iu, ar = np.minimum(x[4], I - ia), np.minimum(x[2], A)
            ad = np.minimum(x[3], A - ar)
            S, I, A, R, D = S - si, I + si - ia - iu, A + ia - ar - ad, R + ar, D + ad
            days.append(np.stack([A, R, D]))
        final = A + R + D
        good = np.flatnonzero((final >= 10 * A0) & (final <= P // 2) & (S > 0))
        if good.size:
            return th[good[0]], np.ascontiguousarray(np.stack(days)[:, :, good[0]].T.astype(np.int32))


def _tolerance_of(observed, case, P, seed, stream=0):
    """The q-quantile of the distances of the case's own draws."""
    d = abc.abc_distances(observed, P, case["n"], seed, stream=stream, mode=case["mode"])
    return float(torch.sort(d)[0][math.ceil(case["q"] * case["n"]) - 1])


def _posterior_like(g, theta, B):
    """B parameter vectors around theta inside the box, as an accepted set is."""
    th = theta + 0.08 * (HI - LO) * g.standard_normal((B, 8))
    return torch.from_numpy(np.clip(th, LO, HI).astype(np.float32)).cuda()


def _population(g, m):
    """A weighted particle population inside the box: correlated, bounded."""
    mix = 0.25 * np.tril(g.standard_normal((8, 8))) + 0.6 * np.eye(8)
    z = g.standard_normal((m, 8)) @ mix.T
    return LO + (HI - LO) / (1 + np.exp(-(g.normal(0, 0.5, 8) + z)))


def _flow_params(g, blocks, hidden, flows=1):
    """Weights of the size training reaches, in the flow's parameter order."""
    v = []
    for _ in range(flows * blocks):
        v += [g.normal(0, 0.6 / math.sqrt(8), hidden * 8), g.normal(0, 0.2, hidden),
              g.normal(0, 0.6 / math.sqrt(hidden), 16 * hidden), g.normal(0, 0.1, 16)]
    return np.concatenate(v).astype(np.float32)


def _cuda_rng(seed):
    r = torch.Generator(device="cuda")
    r.manual_seed(seed)
    return r


def _regions_of(case):
    """(population, horizon) of each region: populations evenly spaced in their logarithm, horizons evenly."""
    f = [r / max(1, case["regions"] - 1) for r in range(case["regions"])]
    return [(int(round(case["P_min"] * (case["P_max"] / case["P_min"]) ** x)),
             int(round(case["T_min"] + (case["T_max"] - case["T_min"]) * x))) for x in f]


def prepare(case, seed):
    g, kind = np.random.default_rng(seed), case["kind"]
    s = dict(case=case, seed=int(seed) & 0x7FFFFFFF)
    if kind in ("sample", "quantile"):
        _, s["observed"] = _epidemic(g, case["P"], case["T"])
        if kind == "sample":
            s["eps"] = _tolerance_of(s["observed"], case, case["P"], s["seed"])
            s["capacity"] = max(1024, 2 * math.ceil(case["q"] * case["n"]))
        else:
            s["k"] = math.ceil(case["q"] * case["n"])
    elif kind == "select":
        # distances over several decades, as a prior batch of an epidemic gives: roots of whole squared sums
        r, n = _cuda_rng(s["seed"]), case["n"]
        x = torch.randn(n, generator=r, device="cuda", dtype=torch.float64)
        s["dist"] = (x * 3.5 + 36).exp_().clamp_(max=2.0**62).floor_().sqrt_()
        s["theta"] = torch.rand((n, 8), generator=r, device="cuda") * torch.tensor(HI, device="cuda").float()
        s["k"], s["capacity"] = math.ceil(case["q"] * n), 2 * math.ceil(case["q"] * n) + 1024
    elif kind in ("simulate", "project"):
        theta, s["observed"] = _epidemic(g, case["P"], case["T"])
        s["theta"] = _posterior_like(g, theta, case["B"])
        # the sample indices of a set accepted from a large batch: sparse, increasing
        s["index"] = torch.from_numpy(np.cumsum(g.integers(1, 20_000, case["B"]))).cuda()
    elif kind == "regions":
        regs = []
        for j, (P, T) in enumerate(_regions_of(case)):
            _, obs = _epidemic(g, P, T)
            regs.append(dict(observed=obs, N_pop=P, eps=_tolerance_of(obs, case, P, s["seed"], stream=j),
                             n_samples=case["n"], stream=j, capacity=max(1024, 2 * math.ceil(case["q"] * case["n"]))))
        s["plan"], s["stream"] = abc.Plan(regs, s["seed"], mode=case["mode"]), torch.cuda.Stream()
    elif kind in ("flow_sample", "flow_log_q", "flow_train"):
        flows = case.get("flows", 1)
        s["flow"] = abc.Flow(case["blocks"], case["hidden"], n_flows=flows)
        s["params"] = _flow_params(g, case["blocks"], case["hidden"], flows)
        s["flow"].set_params(s["params"])
        if kind == "flow_train":
            n = case["points"]
            s["thetas"] = [torch.from_numpy(_population(g, n).astype(np.float32)).cuda() for _ in range(flows)]
            s["weights"] = [torch.from_numpy(np.exp(0.5 * g.standard_normal(n)).astype(np.float32)).cuda()
                            for _ in range(flows)]
            s["stream"] = torch.cuda.Stream()
        else:
            s["flow"].set_proposal_scale(case["tau"])
        if kind == "flow_log_q":
            r = _cuda_rng(s["seed"])
            s["theta"] = torch.rand((case["n"], 8), generator=r, device="cuda") * torch.tensor(HI, device="cuda").float()
    elif kind == "pmc":
        old, new = _population(g, case["m"]), None
        w = np.exp(0.7 * g.standard_normal(case["m"]))
        w /= w.sum()
        mean = w @ old
        s["L"] = np.linalg.cholesky(2 * (old - mean).T @ (w[:, None] * (old - mean))).astype(np.float32)
        # the accepted part of a round's proposals: moved particles near the population's centre
        new = old[g.integers(0, case["m"], case["n"])] + 0.5 * g.standard_normal((case["n"], 8)) @ s["L"].T
        s["old"], s["w"] = torch.from_numpy(old.astype(np.float32)).cuda(), torch.from_numpy(w).cuda()
        s["new"] = torch.from_numpy(np.clip(new, LO, HI).astype(np.float32)).cuda()
    return s


# ---------------------------------------------------------------------------
# One pass
# ---------------------------------------------------------------------------
def _sorted(theta, dist, idx):
    order = torch.argsort(idx)
    return theta[order], dist[order], idx[order]


def run(s):
    case = s["case"]
    kind = case["kind"]
    if kind == "sample":
        theta, dist, idx, n = abc.abc_sample(s["observed"], case["P"], s["eps"], case["n"], s["seed"],
                                             mode=case["mode"], capacity=s["capacity"])
        return _sorted(theta, dist, idx) + (n,)
    if kind == "quantile":
        theta, dist, idx, n, eps = abc.abc_sample_quantile(s["observed"], case["P"], case["n"], s["k"], s["seed"],
                                                           mode=case["mode"])
        return _sorted(theta, dist, idx) + (n, eps)
    if kind == "select":
        eps = abc.abc_kth_smallest(s["dist"], s["k"])
        theta, dist, idx, n = abc.abc_select_below(s["dist"], eps, theta=s["theta"], capacity=s["capacity"])
        return _sorted(theta, dist, idx) + (n, eps)
    if kind == "simulate":
        return abc.abc_simulate(s["theta"], s["index"], s["observed"][:, 0], case["T"], case["P"], s["seed"],
                                mode=case["mode"])
    if kind == "project":
        return abc.abc_project(s["theta"], s["index"], s["observed"][:, 0], case["T"], case["P"], s["seed"],
                               mode=case["mode"])
    if kind == "regions":
        # the same chunk of every region from its first index; the plan's buffers cleared
        plan = s["plan"]
        with torch.cuda.stream(s["stream"]):
            for j in range(plan.n_regions):
                plan.set_region(j, None, 0)
            plan.reset()
            plan.run_graph(1)
            out = []
            for j in range(plan.n_regions):
                theta, dist, idx, n, _ = plan.results(j)    # the fifth is the work done, not a result
                out.append(_sorted(theta, dist, idx) + (n,))
        torch.cuda.current_stream().wait_stream(s["stream"])
        return out
    if kind == "flow_sample":
        return s["flow"].sample(case["n"], seed=s["seed"])
    if kind == "flow_log_q":
        return s["flow"].log_q(s["theta"])
    if kind == "flow_train":
        flow = s["flow"]
        flow.set_params(s["params"])
        if case["flows"] == 1:
            loss = flow.train(s["thetas"][0], s["weights"][0], n_steps=case["steps"], batch=case["batch"],
                              seed=s["seed"], cuda_stream=s["stream"])
        else:
            loss = flow.train_flows(s["thetas"], s["weights"], n_steps=case["steps"], batch=case["batch"],
                                    seed=s["seed"], cuda_stream=s["stream"])
        return loss, flow.get_params()
    return abc.abc_pmc_weights(s["new"], s["old"], s["w"], s["L"])


# ---------------------------------------------------------------------------
# What a pass cannot do without
# ---------------------------------------------------------------------------
def work(case):
    kind = case["kind"]
    if kind == "sample":
        # early rejection simulates about half of the days
        return {"bytes": 48 * case["q"] * case["n"], "flops": DAY_OPS * 0.5 * case["n"] * case["T"]}
    if kind == "quantile":
        return {"bytes": 48 * case["q"] * case["n"], "flops": DAY_OPS * case["n"] * case["T"]}
    if kind == "select":
        return {"bytes": 8 * case["n"] + 80 * case["q"] * case["n"], "flops": case["n"]}
    if kind == "simulate":
        return {"bytes": case["B"] * (40 + 24 * (case["T"] + 1)), "flops": DAY_OPS * case["B"] * case["T"]}
    if kind == "project":
        return {"bytes": 40 * case["B"] + 36 * (case["T"] + 1), "flops": DAY_OPS * case["B"] * case["T"]}
    if kind == "regions":
        days = sum(T for _, T in _regions_of(case)) * case["n"]
        return {"bytes": 48 * case["q"] * case["n"] * case["regions"], "flops": DAY_OPS * 0.3 * days}
    if kind == "pmc":
        return {"bytes": 40 * case["n"] + 40 * case["m"], "flops": 19.0 * case["n"] * case["m"]}
    # multiply-adds of the masked layers: unit l reads its degree's inputs and feeds the later outputs
    degree = [l % 7 + 1 for l in range(case["hidden"])]
    per_row = 2 * case["blocks"] * sum(d + 2 * (8 - d) for d in degree)
    params = 4 * case["blocks"] * (25 * case["hidden"] + 16)
    if kind == "flow_train":
        rows = case["flows"] * case["batch"] * case["steps"]
        return {"bytes": 36 * rows + 2 * case["flows"] * params, "flops": 3 * per_row * rows}
    return {"bytes": 36 * case["n"] + params, "flops": per_row * case["n"]}


def tolerance(case):
    kind = case["kind"]
    if kind == "select" or case.get("mode") == "exact":
        return "exact"      # whole arithmetic and IEEE operations in a fixed order: bit-reproducible by contract
    if "mode" in case:
        # approximate transcendentals move a count by one now and then: against the exact arithmetic 2e-6 of
        # the result's norm and 2e-4 of a single count
        return {"rel": 1e-5, "max": 1e-3, "differ": 0.01}
    if kind == "pmc":
        return {"rel": 1e-5, "max": 1e-3}       # sums of 32-bit exponentials: 1e-6 to 5e-6 off 64 bits
    if kind == "flow_train":
        # points moved by 1e-7 of themselves move the trained parameters by up to 4e-4 of their norm, one
        # parameter by up to 0.08 (an update's sign where the gradient is near zero)
        return {"rel": 1.5e-3, "max": 0.3}
    # BF16 operands: 2e-3 to 4e-3 (densities at given points) and 2e-2 (densities of draws) off 64 bits
    return {"rel": 8e-3 if kind == "flow_log_q" else 2e-2, "max": 0.5}


# ---------------------------------------------------------------------------
# The same in 64 bits
# ---------------------------------------------------------------------------
def _philox(c, seed):
    """Philox4x32-10 words (int64 tensors below 2^32) of counters c, a list of four such tensors."""
    mask = 0xFFFFFFFF
    k0, k1 = seed & mask, (seed >> 32) & mask
    for _ in range(10):
        p0, p1 = c[0] * 0xD2511F53, c[2] * 0xCD9E8D57
        c = [((p1 >> 32) & mask) ^ c[1] ^ k0, p1 & mask, ((p0 >> 32) & mask) ^ c[3] ^ k1, p0 & mask]
        k0, k1 = (k0 + 0x9E3779B9) & mask, (k1 + 0xBB67AE85) & mask
    return c


class _Flow64:
    """The masked autoregressive flow in float64."""

    def __init__(self, params, blocks, hidden, tau):
        d = torch.arange(hidden, device="cuda") % 7 + 1
        j = torch.arange(1, 9, device="cuda")
        m1, m2 = (d[:, None] >= j[None, :]).double(), (j[:, None] > d[None, :]).double().repeat(2, 1)
        v, at, self.tau, self.blocks = torch.from_numpy(params).cuda().double(), 0, tau, []
        for _ in range(blocks):
            part = []
            for shape in ((hidden, 8), (hidden,), (16, hidden), (16,)):
                n = math.prod(shape)
                part.append(v[at:at + n].reshape(shape))
                at += n
            self.blocks.append((part[0] * m1, part[1], part[2] * m2, part[3]))
        self.lo, self.width = torch.tensor(LO, device="cuda"), torch.tensor(HI - LO, device="cuda")

    @staticmethod
    def made(x, block):
        w1, b1, w2, b2 = block
        out = torch.relu(x @ w1.T + b1) @ w2.T + b2
        return out[:, :8], 6 * torch.tanh(out[:, 8:] / 6)

    def base(self, z):
        a = (z / self.tau).abs()
        return (-a - 2 * torch.log1p(torch.exp(-a)) - math.log(self.tau)).sum(1)

    def jacobian(self, y):
        return (torch.log(self.width) - torch.nn.functional.softplus(-y) - torch.nn.functional.softplus(y)).sum(1)

    def log_q(self, theta):
        u = ((theta.double() - self.lo) / self.width).clamp(2.0**-24, 1 - 2.0**-24)
        y = x = torch.log(u) - torch.log1p(-u)
        logdet = torch.zeros(len(x), device="cuda", dtype=torch.float64)
        for block in self.blocks:
            mu, al = self.made(x, block)
            x, logdet = ((x - mu) * torch.exp(-al)).flip(1), logdet - al.sum(1)
        return self.base(x) + logdet - self.jacobian(y)

    def sample(self, n, seed, first):
        i = torch.arange(first, first + n, device="cuda")
        zero = torch.zeros_like(i)
        words = [w for b in (0, 1) for w in _philox([i & 0xFFFFFFFF, i >> 32, zero, zero + b], seed)]
        u = (2 * (torch.stack(words, 1) & 0x7FFFFF) + 1).double() * 2.0**-24
        x = self.tau * (torch.log(u) - torch.log1p(-u))
        logq = self.base(x)
        for block in reversed(self.blocks):
            z, x = x.flip(1), torch.zeros_like(x)
            for j in range(8):
                mu, al = self.made(x, block)
                x[:, j] = z[:, j] * torch.exp(al[:, j]) + mu[:, j]
            logq = logq - al.sum(1)
        return self.lo + self.width * torch.sigmoid(x), logq - self.jacobian(x)


def exact(case, seed):
    kind = case["kind"]
    if kind == "select":
        s = prepare(case, seed)
        eps = torch.sort(s["dist"])[0][s["k"] - 1]
        idx = torch.nonzero(s["dist"] <= eps)[:, 0]
        return s["theta"][idx].double(), s["dist"][idx], idx, len(idx), float(eps)
    if kind in ("flow_sample", "flow_log_q"):
        s = prepare(case, seed)
        f, chunk, out = _Flow64(s["params"], case["blocks"], case["hidden"], case["tau"]), 1 << 18, []
        for at in range(0, case["n"], chunk):
            n = min(chunk, case["n"] - at)
            out.append(f.log_q(s["theta"][at:at + n]) if kind == "flow_log_q" else f.sample(n, s["seed"], at))
        if kind == "flow_log_q":
            return torch.cat(out)
        return torch.cat([o[0] for o in out]), torch.cat([o[1] for o in out])
    if kind == "pmc":
        s = prepare(case, seed)
        inv = torch.linalg.inv(torch.from_numpy(s["L"].astype(np.float64))).cuda()
        a, b, w, out = s["new"].double() @ inv.T, s["old"].double() @ inv.T, s["w"], []
        for at in range(0, len(a), 1024):
            d2 = ((a[at:at + 1024, None, :] - b[None, :, :]) ** 2).sum(2)
            out.append(1 / (torch.exp(-0.5 * d2) @ w))
        return torch.cat(out)
    # simulated counts are floors of random sums: they have no value in 64 bits to be near to, and
    # training's batches are the framework's own draws
    return None
