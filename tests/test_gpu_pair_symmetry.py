"""FP32: the forces of a pair on its two particles are each other's negatives, bit
for bit: distance, support and powers round alike for both ends."""
import numpy as np
import pytest

import workloads as W
from parity_util import make_gpu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("gamma,kappa", [(2.0, 1.0), (2.0, 1.3), (1.4, 1.0)])
@pytest.mark.parametrize("dim", [2, 3])
def test_forces_of_lone_pairs_cancel(dim, gamma, kappa):
    m = 8
    p = W.Problem(dim=dim, lo=[0, 0, 0], hi=[1, 1, 1 if dim == 3 else 0], field_kind=W.FIELD_LINEAR_DISTANCE, a=0.006,
                  b=0.03, dist_shape=0, rho_scale=1.0, gamma=gamma, kappa=kappa, tau=2.0 / kappa, n_colors=2,
                  shapes=[W.Shape(W.SPHERE, False, [0.5, 0.5, 0.5 if dim == 3 else 0.0], [0.03, 0, 0])])
    rng = np.random.default_rng(3)
    g = (np.arange(m) + 0.5) / m  # an eighth apart; the largest support is 0.063, partners are 0.025 away at most
    x = np.stack(np.meshgrid(*[g] * dim, indexing="ij"), -1).reshape(-1, dim)
    u = rng.standard_normal(x.shape)
    u /= np.linalg.norm(u, axis=1)[:, None]
    h = 2.0 * (0.006 + 0.03 * np.abs(np.linalg.norm(x - 0.5, axis=1) - 0.03))
    pos = np.concatenate([x, x + u * (h * rng.uniform(0.2, 0.8, len(x)) * 0.5)[:, None]])
    r = make_gpu(p, pos, rng.integers(0, 2, len(pos)).astype(np.uint8), "fp32")
    r.step(1)
    assert r.stats()["force_pairs"] == len(x)
    a = r.field("acc")
    r.close()
    first, second = a[:len(x)], a[len(x):]
    assert np.abs(first).min() > 0.0
    assert np.array_equal(first, -second)
