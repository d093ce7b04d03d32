"""CP-ALS in tight memory: the slices of the tensor-core products (200 MB here) are
optional, so that a call whose own arrays fit goes through (needs a GB300)."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


def test_call_goes_through_without_room_for_slices():
    import __graft_entry__ as g
    g.build()
    from paper_2111_11473_gb300 import binding
    o, v, N, W = 20, 100, 1500, 1500
    r = np.random.default_rng(1)
    yo, yv, tau = (r.standard_normal((m, W)) for m in (o, v, N))
    U = (yo[:, None, :] * yv[None, :, :]).reshape(o * v, W) @ tau.T
    U += 0.05 * U.std() * r.standard_normal(U.shape)
    eps = np.linspace(1.0, 0.3, N)
    start = [a + 0.1 * r.standard_normal(a.shape) for a in (yo, yv, tau)]
    # (eigenvalues over decades take the CUDA cores: every kernel is loaded then)
    w = 10.0 ** (-6.0 * np.arange(N) / N)
    binding.cp_als(U / w, w, *start, iters=1)
    ref = binding.cp_als(U, eps, *start, iters=1)[3]
    own = 8 * (3 * W * W + 2 * o * v * W + N * W + N * W + o * v * N + (1 << 22)    # work
               + o * v * N + (o + v + N) * W)                                      # inputs
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    free = torch.cuda.mem_get_info()[0]
    hold = torch.empty(free - own - (90 << 20), dtype=torch.uint8, device="cuda")
    try:
        got = binding.cp_als(U, eps, *start, iters=1)[3]
    finally:
        del hold
        torch.cuda.empty_cache()
    assert np.allclose(got, ref, rtol=1e-9)
