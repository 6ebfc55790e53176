"""Neighbour lists between rebuilds, pair by pair, and the launch rules that
test_gpu_dispatch leaves out: the list builders and the FP64 blocks on both sides
of their lines in 3D and at large counts, and a grid whose scan takes two levels."""
import numpy as np
import pytest
from scipy.spatial import cKDTree

import oracle
import workloads as W
from parity_util import compare_step, h_all, make_gpu
from test_gpu_parity import check_cell_list

pytestmark = pytest.mark.gpu


def _steep(dim, b, n, seed):
    """n particles around a small ball, drawn from a density that falls off steeply
    (spacing a + b times the distance: smoothing lengths over several grid levels)."""
    r0, a = 0.05, 0.003
    c = [0.5, 0.5, 0.5 if dim == 3 else 0.0]
    p = W.Problem(dim=dim, lo=[0, 0, 0], hi=[1, 1, 1 if dim == 3 else 0], field_kind=W.FIELD_LINEAR_DISTANCE, a=a, b=b,
                  dist_shape=0, rho_scale=1.0, tau=2.0, n_colors=5, shapes=[W.Shape(W.SPHERE, False, c, [r0, 0, 0])])
    r = np.linspace(r0, 0.5, 20001)
    mass = r ** (dim - 1) / (a + b * (r - r0)) ** dim * (2 * np.pi if dim == 2 else 4 * np.pi)
    cum = np.concatenate([[0.0], np.cumsum(0.5 * (mass[1:] + mass[:-1]) * np.diff(r))])
    p.rho_scale = n / cum[-1]
    rng = np.random.default_rng(seed)
    u = rng.standard_normal((n, dim))
    u /= np.linalg.norm(u, axis=1)[:, None]
    rad = np.interp(rng.random(n) * cum[-1], cum, r)
    return p, np.array(c[:dim]) + rad[:, None] * u, rng.integers(0, 5, n).astype(np.uint8)


def _edge_pairs(p, x, rel):
    """Pairs whose distance is within rel of their support kappa (h_i + h_j) / 2."""
    h = h_all(p, x)
    order = np.argsort(h)
    xs, hs = x[order], h[order]
    tree = cKDTree(xs)
    found = 0
    for i, nb in enumerate(tree.query_ball_point(xs, p.kappa * hs * (1 + rel))):  # from the pair's larger h
        nb = np.asarray(nb)
        nb = nb[nb < i]
        H = 0.5 * p.kappa * (hs[i] + hs[nb])
        found += int((np.abs(np.linalg.norm(xs[nb] - xs[i], axis=1) - H) <= rel * H).sum())
    return found


# list builders: groups of lanes (3,000), one thread per particle (21,000); the
# FP64 pass with several lanes and the screened one. A missing pair near its edge
# changes no sum beyond rounding, so the pairs are counted: FP32 rounds a pair's
# distance and support to a few 2^-24 of themselves (1e-5 is far above that)
@pytest.mark.parametrize("precision", ["fp32", "fp64"])
@pytest.mark.parametrize("dim,b,n", [(2, 0.08, 3000), (3, 0.18, 3000), (3, 0.1, 21000)])
def test_aged_lists_hold_every_pair(precision, dim, b, n):
    p, pos, col = _steep(dim, b, n, 11 + dim)
    r = make_gpu(p, pos, col, precision)
    assert r.grid()["n_levels"] >= 3
    built = []
    for at in range(10):
        x = r.positions()
        r.step(1)
        st = r.stats()
        want = oracle.step(p, x, col, at)[1]["force_pairs"]
        slack = _edge_pairs(p, x, 1e-5) if precision == "fp32" else 0
        assert abs(st["force_pairs"] - want) <= slack, (at, st["force_pairs"], want, slack)
        built.append(st["list_rebuilds"])
    assert built[-1] < 10  # some of these steps ran on lists of an earlier one
    r.close()


@pytest.mark.parametrize("precision", ["fp32", "fp64"])
@pytest.mark.parametrize("n", [20480, 20481])
def test_both_list_builders_in_3d(precision, n):
    p, pos, col = _steep(3, 0.1, n, 5)
    r, _ = compare_step(p, pos, col, precision)
    r.close()


@pytest.mark.parametrize("n", [131072, 131073])
def test_fp64_step_at_the_block_rule(n):
    p = W.graded_hole_2d(n, 8)
    pos, col, _ = W.sample_density(p, n, 3)
    r, _ = compare_step(p, pos, col, "fp64")
    r.close()


# the reverse kernels follow the same rule; the oracle's reverse pass takes too
# long here, so FP64 against FP32 (other block sizes), whose gradients agree to
# 1e-4 of the largest in the oracle tests
@pytest.mark.parametrize("n", [131072, 131073])
def test_reverse_pass_at_the_block_rule(n):
    p = W.graded_hole_2d(n, 8)
    pos, col, _ = W.sample_density(p, n, 3)
    g = {}
    for precision in ("fp32", "fp64"):
        r = make_gpu(p, pos, col, precision)
        g[precision] = r.backward(2)
        r.close()
    a, b = g["fp32"], g["fp64"]
    assert abs(a["L"] - b["L"]) <= 1e-5 * abs(b["L"])
    assert np.abs(a["dpos0"] - b["dpos0"]).max() <= 1e-4 * np.abs(b["dpos0"]).max()


# FP32 pass B in other blocks from 524,288 on: against an FP64 step of the same
# state (the parity tests hold that to 1e-12)
@pytest.mark.parametrize("n", [524287, 524288])
def test_fp32_step_at_the_block_rule(n):
    p = W.graded_hole_2d(n, 8)
    pos, col, _ = W.sample_density(p, n, 3)
    out = {}
    for precision in ("fp32", "fp64"):
        r = make_gpu(p, pos, col, precision)
        r.step(1)
        out[precision] = r.field("rho"), r.field("acc"), r.positions()
        r.close()
    (r32, a32, x32), (r64, a64, x64) = out["fp32"], out["fp64"]
    assert (np.abs(r32 - r64) <= 1e-5 * r64).all()
    assert np.abs(a32 - a64).max() <= 1e-4 * np.abs(a64).max()
    assert np.abs(x32 - x64).max() <= 1e-4 * np.abs(x64 - pos).max() + 1.2e-7


@pytest.mark.parametrize("precision", ["fp32", "fp64"])
def test_a_grid_of_more_than_2048_scan_tiles(precision):
    p = W.uniform_square_2d(140, 5)
    pos, col, _ = W.lattice_jitter_2d(p, 140, 0.3, 1)
    x = []
    for factor in (0.0174, 1.0):
        r = make_gpu(p, pos, col, precision, cell_factor=factor)
        if factor < 1:
            assert r.grid()["base"][-1] > 2048 * 4096
            check_cell_list(p, r, precision)
        r.step(4)
        x.append(r.positions())
        r.close()
    # another cell order: sums in another order, rounding only
    assert np.abs(x[0] - x[1]).max() <= (2e-6 if precision == "fp32" else 1e-13)
