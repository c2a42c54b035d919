"""A flow's gradient and training run are pinned: digests of the parameters,
gradient and losses recorded on a GB300. A step's rounding travels through every
later one, so a change of launch shape, order of loads or overlap must not move a
bit of them (the oracle tests hold the arithmetic itself)."""
import hashlib

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_2012_14332_gb300 as abc  # noqa: E402
from paper_2012_14332_gb300 import build as _build  # noqa: E402

_build.build()
HI = np.array([1, 100, 2, 1, 1, 1, 1, 2.0])


def _sha(a):
    return hashlib.sha256(np.ascontiguousarray(a, dtype=np.float32).tobytes()).hexdigest()[:16]


def _data(n, seed):
    g = np.random.default_rng(seed)
    theta = (HI * g.uniform(0.02, 0.98, (n, 8))).astype(np.float32)
    return torch.from_numpy(theta).cuda(), torch.from_numpy(g.uniform(0.1, 2.0, n).astype(np.float32)).cuda()


def _params(K, H, R):
    g, v = np.random.default_rng(K + H), []
    for _ in range(K * R):
        v += [g.uniform(-0.4, 0.4, 8 * H), g.uniform(-0.4, 0.4, H), g.uniform(-0.08, 0.08, 16 * H),
              g.uniform(-0.2, 0.2, 16)]
    return np.concatenate(v).astype(np.float32)


# blocks, hidden units, flows, points, batch, steps: the paired, the narrow and
# the wide form of the gradient kernel; digests of the first flow's gradient,
# the parameters after the steps and their losses, and the held-out losses of an
# early-stopped run
CASES = [(3, 256, 1, 5000, 1024, 30, "4448535305c09cb9", "04a93cd66a029664", "b179fcefcf4d4635", "eecbc381cfecce29"),
         (3, 256, 1, 20001, 4096, 10, "41edbe162a9721a2", "62a54e2c595530a5", "6648d98a479ed9be", "9503bfafb004bf14"),
         (2, 64, 1, 3000, 512, 30, "d5776448f206874d", "48425465aa006aef", "6c18f45195ac71ef", "7eef96e32168988e"),
         (4, 160, 1, 3000, 768, 10, "3344d2772fa9977e", "3a562d764103e22a", "75baeb471f5c651c", "9c6d4daa74447b18"),
         (1, 16, 1, 500, 64, 30, "0d38e029eaea6222", "c0a2645bc4a2450d", "531d9c7a00df2edb", "507d14890f56e273"),
         (3, 256, 16, 2055, 2048, 5, "4ffb87c21e6e5397", "516afef2d3d00554", "fb985ce9cc673412", "7a2b9b0ceddd7a5c"),
         (3, 128, 4, 3000, 512, 30, "97ca04ffd95b477e", "ec048389b0368b12", "77e634ca9e622c65", "7138e9c92d03f4bd")]


@pytest.mark.parametrize("K,H,R,n,batch,steps,gradient,params,losses,held_out", CASES)
def test_training_results_are_pinned(K, H, R, n, batch, steps, gradient, params, losses, held_out):
    f, s = abc.Flow(K, H, n_flows=R), torch.cuda.Stream()
    f.set_params(_params(K, H, R))
    data = [_data(n - 7 * r, 100 + r) for r in range(R)]
    got_gradient = _sha(f.gradient(*data[0])[1])
    theta, weights = [t for t, _ in data], [w for _, w in data]
    got_losses = f.train_flows(theta, weights, n_steps=steps, batch=batch, seed=9, cuda_stream=s)
    assert (got_gradient, _sha(f.get_params()), _sha(got_losses)) == (gradient, params, losses)
    f.set_params(_params(K, H, R))
    got = f.train_flows(theta, weights, n_steps=100, batch=batch, seed=9, lr=3e-3, val_fraction=0.3, cuda_stream=s)
    assert _sha(got) == held_out
    f.close()
