"""A particle's smoothing length goes into the FP32 view with one rounding and
comes out of it with none, whatever the support factor."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu

f = np.float32


# a lone particle's density is alpha / (kappa h)^2 and so shows its h; here in
# numpy's FP32, each operation rounded once, as the device computes it (the self
# term, 1 to a rounding, may differ by an ulp, and so the result)
@pytest.mark.parametrize("kappa", [0.7, 1.0, 1.1, 1.3])
def test_the_density_of_a_lone_particle(kappa):
    from paper_1906_07925_gb300 import Relaxation
    for s0 in np.linspace(0.021, 0.12, 40):
        p = W.uniform_square_2d(8, 1).copy(s0=float(s0), kappa=kappa, tau=2.0)
        r = Relaxation(p, 1, 1, precision="fp32", record_fields=True)
        r.set_state(np.array([[0.4, 0.6]]), np.zeros(1, np.uint8))
        r.step(1)
        rho, c0 = f(r.field("rho")[0]), r.grid()["cell"][0]
        r.close()
        h = f(2.0) * f(s0)
        hv = h * f(1.0 / c0)
        H = f(kappa) * hv * f(c0)
        want = f(7.0 / np.pi) / (H * H)
        assert abs(int(rho.view(np.int32)) - int(want.view(np.int32))) <= 2, (s0, rho, want)
