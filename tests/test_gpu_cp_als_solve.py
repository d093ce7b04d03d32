"""The normal equations of CP-ALS at ranks around the 32-column panels and with
fewer and more right-hand sides than SMs, and the large products on the tensor
cores, against the float64 oracle (needs a GB300).

Bounds: those of the other CP-ALS test (1e-9 of the objective and of the
reconstruction)."""
import numpy as np
import pytest

from oracle import cp_als
from tests.test_gpu_cp_als import _case

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__ as g
    g.build()


@pytest.mark.parametrize("shape", [(5, 9, 31, 1, 1), (9, 33, 200, 31, 2), (8, 31, 170, 32, 3),
                                   (11, 30, 160, 33, 4), (13, 40, 310, 64, 5),
                                   (20, 61, 650, 97, 6), (30, 100, 301, 130, 7)],
                         ids=lambda s: "x".join(map(str, s)))
def test_matches_oracle(shape):
    from paper_2111_11473_gb300 import binding
    o, v, N, W, seed = shape
    U, eps, start = _case(o, v, N, W, seed, noise=0.05)
    yo, yv, tau, hist = binding.cp_als(U, eps, *start, iters=3)
    ryo, ryv, rtau, rhist = cp_als.als(U, eps, *start, 3)
    assert np.allclose(hist, rhist, rtol=1e-9, atol=1e-12)
    rec = (yo[:, None, :] * yv[None, :, :]).reshape(o * v, W) @ tau.T
    rrec = (ryo[:, None, :] * ryv[None, :, :]).reshape(o * v, W) @ rtau.T
    assert np.abs(rec - rrec).max() < 1e-9 * max(1.0, np.abs(rrec).max())


def test_singular_normal_equations_are_refused():
    import paper_2111_11473_gb300 as pkg
    U, eps, start = _case(4, 9, 50, 40, 1, noise=0.0)
    with pytest.raises(pkg.ThcError, match="singular"):
        pkg.binding.cp_als(U, eps, *[0.0 * a for a in start], iters=1)
