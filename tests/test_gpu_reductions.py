"""The step's global reductions (sph_stats) against sums over the recorded
fields, at particle counts around the edges of a warp, a block and a group of
blocks: one lane, ragged warps, one block, several groups."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", ["fp32", "fp64"])
@pytest.mark.parametrize("n", [1, 2, 31, 33, 255, 257, 32768, 32769, 70001])
def test_statistics_are_the_sums_over_the_fields(n, precision):
    """sum rho: the device adds the recorded values themselves (fixed-point or
    FP64), so only FP64 rounding of n terms separates it from numpy's sum. The
    density error also takes rho_t, which the device rounds to its working
    precision: a few ulp of rho / rho_t in each term."""
    from paper_1906_07925_gb300 import Relaxation
    # a spacing of at most 1/8: a coarser one leaves no cell grid
    p = W.uniform_square_2d(max(8, int(np.sqrt(n))), 3)
    rng = np.random.default_rng(n)
    pos, col = rng.random((n, 2)), rng.integers(0, 3, n).astype(np.uint8)
    r = Relaxation(p, n, 3, precision=precision, record_fields=True)
    r.set_state(pos, col)
    r.step(1)
    st, rho, acc = r.stats(), r.field("rho"), r.field("acc")
    r.close()
    eps = 2.0 ** -23 if precision == "fp32" else 2.0 ** -52
    assert abs(st["sum_rho"] - rho.sum()) <= 1e-13 * rho.sum()
    an = np.linalg.norm(acc, axis=1)
    assert abs(st["max_a"] - an.max()) <= 4 * eps * an.max()
    e = rho / (1.0 / p.s0 ** 2) - 1.0  # rho_t of the uniform field
    ulp = 8 * eps * (1.0 + np.abs(e))  # h, its powers and 1 / rho_t, each rounded once
    assert abs(st["err_max"] - np.abs(e).max()) <= ulp.max()
    assert abs(st["err_l2"] - (e * e).sum()) <= (2 * np.abs(e) * ulp + ulp ** 2).sum() + 1e-13 * (e * e).sum()
    if an.max() > 0:  # the support radius is kappa h = tau s0 everywhere
        m = p.tau * p.s0 / an.max()
        assert abs(st["min_rc_over_a"] - m) <= 16 * eps * m
        assert abs(st["dt1"] - 0.25 * np.sqrt(m)) <= 16 * eps * st["dt1"]
    else:
        assert np.isinf(st["min_rc_over_a"]) and st["dt1"] == 0.0
