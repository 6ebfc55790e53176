"""Device memory of a taped step of the reverse pass against the figure that
the C header gives (include/sphmesh.h, sensitivities)."""
import pytest

import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision,base", [("fp32", 100), ("fp64", 156)])
@pytest.mark.parametrize("gamma", [2.0, 1.4])
def test_a_tape_slot_takes_what_the_header_says(precision, base, gamma):
    import torch
    from paper_1906_07925_gb300 import Relaxation
    n = 32 * 640
    p = W.graded_inclusion_3d(n, 4).copy(gamma=gamma)
    used = []
    r = Relaxation(p, n, 4, precision=precision, seed=1)
    for slots in (2, 8):
        r.backward(8, ckpt_every=slots)
        used.append(torch.cuda.memory_stats()["requested_bytes.all.current"])  # not the allocator's blocks
    cap = r.stats()["list_capacity"]
    r.close()
    # 8 checkpoints of the positions shrink to none: allocated by the first run, with more of them
    lists = 4 * cap + (4 * cap + 4 if gamma != 2.0 else 0)
    assert (used[1] - used[0]) / 6 <= (base + lists) * n + 16 * 512
