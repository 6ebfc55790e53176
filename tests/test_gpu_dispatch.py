"""Particle counts on both sides of each launch rule of a step, lists at every
age between rebuilds, and lists that do not fit. Steps are checked against the
FP64 oracle at the step parity tolerances (parity_util)."""
import numpy as np
import pytest

import workloads as W
from parity_util import compare_step, make_gpu

pytestmark = pytest.mark.gpu


def _sampled(dim, n, gamma, seed):
    s = (1.0 / n) ** (1.0 / dim)
    p = W.Problem(dim=dim, lo=[0, 0, 0], hi=[1, 1, 1 if dim == 3 else 0], field_kind=W.FIELD_LINEAR_DISTANCE, a=s,
                  b=0.2 * s, dist_shape=0, gamma=gamma, kappa=1.0, tau=2.0, n_colors=5,
                  shapes=[W.Shape(W.SPHERE, False, [0.5, 0.5, 0.5 if dim == 3 else 0.0], [0.05, 0, 0])])
    rng = np.random.default_rng(seed)
    return p, W.uniform_in_domain(p, n, rng), rng.integers(0, 5, n).astype(np.uint8)


# the largest count with several lanes per particle, and the next: FP64 passes
# (8,192), FP32 pass B (16,384), list build (20,480, either precision)
@pytest.mark.parametrize("precision,dim,n,gamma", [
    ("fp64", 2, 8192, 1.4), ("fp64", 2, 8193, 1.4), ("fp64", 3, 8192, 2.0), ("fp64", 3, 8193, 2.0),
    ("fp32", 2, 16384, 2.0), ("fp32", 2, 16385, 2.0), ("fp32", 3, 16384, 1.4), ("fp32", 3, 16385, 1.4),
    ("fp32", 2, 20480, 2.0), ("fp32", 2, 20481, 2.0), ("fp64", 2, 20480, 2.0), ("fp64", 2, 20481, 2.0)])
def test_one_step_on_both_sides_of_a_launch_rule(precision, dim, n, gamma):
    p, pos, col = _sampled(dim, n, gamma, n + dim)
    r, _ = compare_step(p, pos, col, precision)
    r.close()


# a list holds each particle's reach: every step from the rebuild to the last one
# before the next finds all pairs, first while particles move fast, then slowly
@pytest.mark.parametrize("precision", ["fp32", "fp64"])
@pytest.mark.parametrize("dim,n", [(2, 1500), (3, 1500)])
def test_lists_hold_every_pair_until_they_are_rebuilt(precision, dim, n):
    p, pos, col = _sampled(dim, n, 2.0, 7 + dim)
    r = make_gpu(p, pos, col, precision)
    at = 0
    for skipped in (0, 30):
        r.step(skipped)
        at += skipped
        for _ in range(12):
            compare_step(p, r.positions(), col, precision, step_index=at, gpu=r)
            at += 1
    r.close()


@pytest.mark.parametrize("precision,n", [("fp32", 1000), ("fp64", 1000), ("fp32", 20481)])
def test_a_list_that_does_not_fit_is_an_error(precision, n):
    from paper_1906_07925_gb300 import SphError
    p, pos, col = _sampled(2, n, 2.0, 5)
    r = make_gpu(p, pos, col, precision, list_capacity=8)
    with pytest.raises(SphError, match="CELL_OVERFLOW"):
        r.step(1)
        r.sync()
    r.close()
