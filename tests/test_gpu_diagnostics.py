"""The neighbour diagnostics name the pairs that the step itself uses."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu


# support factors that are no powers of two: rounding then tells apart two ways
# of computing the support of a pair; some 10^7 pairs, so that pairs lie within
# a rounding of their edge
@pytest.mark.parametrize("kappa", [0.7, 1.1, 1.3])
@pytest.mark.parametrize("dim", [2, 3])
def test_force_sets_are_the_pairs_of_the_step(dim, kappa):
    from paper_1906_07925_gb300 import Relaxation
    n = 700_000
    p = (W.graded_hole_2d if dim == 2 else W.graded_inclusion_3d)(n, 8).copy(kappa=kappa, tau=2.0 / kappa)
    r = Relaxation(p, n, 8, precision="fp32", seed=2)
    r.step(2)
    sets = r.neighbor_sets()
    r.step(1)
    assert int(sets["force_count"].astype(np.int64).sum()) == 2 * r.stats()["force_pairs"]
    r.close()
