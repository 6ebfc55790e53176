"""The block size of the pair passes changes no position by a bit, in either
precision, on both sides of the launch rules that it overrides."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision,n", [("fp64", 8192), ("fp64", 8193), ("fp64", 131072), ("fp64", 131073),
                                         ("fp32", 524287), ("fp32", 524288)])
def test_positions_do_not_depend_on_the_block_size(precision, n):
    from paper_1906_07925_gb300 import Relaxation
    p = W.graded_hole_2d(n, 8)
    out = []
    for threads in (0, 128, 256):
        r = Relaxation(p, n, 8, precision=precision, seed=4)
        r.set_tuning(pass_threads=threads)
        assert r.tuning()["pass_threads"] == (threads or 256)
        r.step(3)
        out.append(r.positions())
        r.close()
    assert np.array_equal(out[0], out[1]) and np.array_equal(out[0], out[2])
