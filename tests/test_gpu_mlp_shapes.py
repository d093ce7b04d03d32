"""The network's fused passes and float32 products at ragged batches and
widths, against the float64 reference (needs a GB300).

Bounds: those of the other float32 test (1e-5 of the loss and of the outputs,
1e-4 of the largest gradient entry)."""
import numpy as np
import pytest

from oracle import mlp as omlp
from tests.test_gpu_mlp import F, _data, _params

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__ as g
    g.build()


@pytest.mark.parametrize("n,H", [(1, 32), (3, 64), (5, 256), (609, 32), (2433, 128), (4097, 64),
                                 (5000, 256), (33, 16), (1000, 48), (300, 512)])
def test_gradient_matches_reference(n, H):
    import paper_2111_11473_gb300 as pkg
    th = _params(H, 3).astype(np.float32)
    X, j, t = _data(n, 4)
    net = pkg.Mlp(hidden=H, bf16=False)
    net.set_params(th)
    L, g = net.loss_grad(X, j, t)
    y = net.predict(X)
    net.close()
    Lr, gr = omlp.grad(th.astype(np.float64), X.astype(np.float64), j.astype(np.float64),
                       t.astype(np.float64), F, H)
    yr, _ = omlp.forward(th.astype(np.float64), X.astype(np.float64), F, H)
    assert abs(L - Lr) < 1e-5 * max(Lr, 1e-3)
    assert np.abs(g - gr).max() < 1e-4 * np.abs(gr).max()
    assert np.abs(y - yr).max() < 1e-5 * max(1.0, np.abs(yr).max())
