"""Lists that fit at the common reach but not at the particles' own: a start a
few times denser than its target in one place, whose particles move fast there.
The run goes on (as one with a skin of its own does), and every step still finds
every pair."""
import numpy as np
import pytest

import workloads as W
from parity_util import compare_step, make_gpu

pytestmark = pytest.mark.gpu


def _dense_ball(n, factor, seed=1):
    """About n particles: jittered lattices, `factor` times the target density inside a ball."""
    s = n ** (-1.0 / 3.0)
    rng = np.random.default_rng(seed)

    def lattice(step):
        m = int(np.floor(1.0 / step))
        g = (np.arange(m) + 0.5) / m
        x = np.stack(np.meshgrid(g, g, g, indexing="ij"), -1).reshape(-1, 3)
        return x + 0.1 * step * (2.0 * rng.random(x.shape) - 1.0)

    inner, outer = lattice(s * factor ** (-1.0 / 3.0)), lattice(s)
    inside = lambda x: np.linalg.norm(x - 0.5, axis=1) < 0.3  # noqa: E731
    pos = np.concatenate([inner[inside(inner)], outer[~inside(outer)]])
    p = W.Problem(dim=3, lo=[0, 0, 0], hi=[1, 1, 1], field_kind=W.FIELD_UNIFORM, s0=s, rho_scale=1.0, tau=2.0,
                  kappa=1.0, n_colors=5)
    return p, pos, rng.integers(0, 5, len(pos)).astype(np.uint8)


# both list builders (groups of lanes up to 20,480 particles, one thread beyond)
@pytest.mark.parametrize("precision,n", [("fp32", 5000), ("fp64", 5000), ("fp32", 21000), ("fp64", 21000)])
def test_a_dense_start_runs_through_its_rebuilds(precision, n):
    p, pos, col = _dense_ball(n, 2.75)
    r = make_gpu(p, pos, col, precision)
    for _ in range(25):
        r.step(1)
        r.sync()
    st = r.stats()
    assert st["list_rebuilds"] >= 2 and st["list_max"] <= st["list_capacity"]
    r.close()


@pytest.mark.parametrize("precision", ["fp32", "fp64"])
def test_lists_cut_to_the_common_reach_hold_every_pair(precision):
    p, pos, col = _dense_ball(5000, 2.75)
    r = make_gpu(p, pos, col, precision)
    for at in range(14):
        compare_step(p, r.positions(), col, precision, step_index=at, gpu=r)
    r.close()
