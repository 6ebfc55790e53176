"""The pair passes at the edges of their list layout: particle counts around
whole warps and tiles, lists with every remainder of a quad of entries, list
capacities that are no multiple of four, a support factor other than one.
Every case is one step against the FP64 oracle at the step parity tolerances
(parity_util)."""
import numpy as np
import pytest

import workloads as W
from parity_util import compare_step, make_gpu

pytestmark = pytest.mark.gpu


def _cloud(dim, n, gamma, kappa):
    s = (1.0 / n) ** (1.0 / dim)
    p = W.Problem(dim=dim, lo=[0, 0, 0], hi=[1, 1, 1 if dim == 3 else 0], field_kind=W.FIELD_LINEAR_DISTANCE, a=s,
                  b=0.2 * s, dist_shape=0, gamma=gamma, kappa=kappa, tau=2.0 / kappa, n_colors=5,
                  shapes=[W.Shape(W.SPHERE, False, [0.5, 0.5, 0.5 if dim == 3 else 0.0], [0.05, 0, 0])])
    rng = np.random.default_rng(n * dim)
    pos = W.uniform_in_domain(p, n, rng)
    return p, pos, rng.integers(0, 5, n).astype(np.uint8)


@pytest.mark.parametrize("precision", ["fp32", "fp64"])
@pytest.mark.parametrize("dim,n,gamma,kappa,capacity", [
    (2, 200, 2.0, 1.0, 0), (2, 257, 1.4, 1.0, 0), (2, 319, 2.0, 1.3, 101), (2, 321, 2.0, 1.0, 103),
    (3, 1000, 2.0, 1.0, 0), (3, 1023, 1.4, 1.0, 301), (3, 1025, 2.0, 0.8, 302), (3, 2081, 2.0, 1.0, 303)])
def test_one_step_matches_the_oracle(precision, dim, n, gamma, kappa, capacity):
    p, pos, col = _cloud(dim, n, gamma, kappa)
    r = make_gpu(p, pos, col, precision, list_capacity=capacity)
    compare_step(p, pos, col, precision, gpu=r)
    if capacity:
        assert r.stats()["list_capacity"] == capacity
    r.close()
