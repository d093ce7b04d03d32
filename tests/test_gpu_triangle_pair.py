"""The float32 triangle over X pairs at every remainder of P modulo 4 (rows
padded to the pitch), odd numbers of rows X, X blocks and grid chunks, against
the float64 residual (needs a GB300).

Bound: float32 FMA chains (tc_products = 0), 2e-5 of the largest entry."""
import numpy as np
import pytest

from synth import make_system, random_amplitudes
from tests.gpu_util import context

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__ as g
    g.build()


@pytest.mark.parametrize("size", [(2, 5, 1, 9, 3), (3, 5, 33, 50, 9), (2, 7, 34, 61, 6),
                                  (4, 9, 63, 96, 12), (3, 6, 64, 67, 5), (2, 4, 97, 40, 8)],
                         ids=lambda s: "x".join(map(str, s)))
@pytest.mark.parametrize("kw", [dict(), dict(i_chunk=7), dict(x_block6=5),
                                dict(workspace_bytes=1 << 20)],
                         ids=["auto", "i_chunk7", "x6_5", "rebuilt_g"])
def test_matches_float64(size, kw):
    import paper_2111_11473_gb300 as pkg
    o, v, P, G, K = size
    s = make_system(o, v, P, G, K, 3)
    Zc, t1 = random_amplitudes(P, o, v, seed=4, t1_scale=0.05, t2_scale=0.5)
    out = []
    for prec in (dict(), dict(precision=pkg.THC_PREC_MIXED, tc_products=0, **kw)):
        with context(s, **prec) as ctx:
            out.append(ctx.residual(Zc, t1))
    scale = max(np.abs(out[0][0]).max(), np.abs(out[0][1]).max())
    assert np.abs(out[1][0] - out[0][0]).max() < 2e-5 * scale
    assert np.abs(out[1][1] - out[0][1]).max() < 2e-5 * scale
