"""CUDA tensors that the caller's stream has still to write: the handle works on
a stream of its own and has to wait for them (positions and colours given to
set_state, the seed and the outputs of backward, the output of positions)."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu

N = 3000


def _handle(precision="fp32"):
    from paper_1906_07925_gb300 import Relaxation
    p = W.adjoint_poly_2d(n=N, n_colors=8, seed=3)
    pos, col, _ = W.sample_density(p, N, seed=5)
    return Relaxation(p, N, int(col.max()) + 1, precision=precision), pos, col


def _busy():
    """Some tens of milliseconds of work on the current stream (a bounded spin)."""
    import torch
    torch.cuda._sleep(100_000_000)


@pytest.mark.parametrize("dtype", ["float32", "float64"])
def test_set_state_waits_for_its_inputs(dtype):
    import torch
    r, pos, col = _handle()
    t = getattr(torch, dtype)
    want = torch.tensor(pos, dtype=t, device="cuda")
    c = torch.tensor(col, device="cuda")
    x, k = torch.full_like(want, 0.1), torch.zeros_like(c)  # what must not be read
    spare = x.double()  # the conversion's kernel and memory are at hand: nothing else waits for the device
    torch.cuda.synchronize()
    del spare
    _busy()
    x.copy_(want)
    k.copy_(c)
    r.set_state(x, k)
    assert np.abs(r.positions() - want.double().cpu().numpy()).max() <= 1e-15
    assert np.array_equal(r.colors(), col)
    r.close()


def test_positions_overwrite_what_the_stream_still_writes():
    import torch
    r, pos, col = _handle()
    r.set_state(pos, col)
    out = torch.empty((N, 2), dtype=torch.float64, device="cuda")
    torch.cuda.synchronize()
    _busy()
    out.fill_(-1.0)
    r.positions(out=out)
    assert np.array_equal(out.cpu().numpy(), r.positions())
    r.close()


def test_backward_waits_for_its_seed_and_returns_its_step_sizes():
    import torch
    r, pos, col = _handle("fp64")
    rng = np.random.default_rng(0)
    seed = torch.tensor(rng.standard_normal((N, 2)), device="cuda")
    r.set_state(pos, col)
    ref = torch.empty_like(seed)
    r.backward(4, seed=seed, out=ref)
    r.close()
    r, pos, col = _handle("fp64")
    r.set_state(pos, col)
    late, out = torch.zeros_like(seed), torch.empty_like(seed)
    torch.cuda.synchronize()
    _busy()
    late.copy_(seed)
    out.fill_(float("nan"))
    res = r.backward(4, seed=late, out=out)
    torch.cuda.synchronize()
    assert torch.equal(out, ref)
    assert bool((res["dt"] > 0).all())
    r.close()
