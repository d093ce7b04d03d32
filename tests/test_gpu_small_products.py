"""Float64 products on the CUDA cores at the sizes where the one-output-per-
thread kernel can go wrong (tile remainders, single rows, K shorter and longer
than its unrolled group, batches that are reduced), through residuals against
the oracle (needs a GB300)."""
import numpy as np
import pytest

from tests.gpu_util import context, oracle_case

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__ as g
    g.build()


# o, v, P, G, K, seed: 1-wide, one below and above the 4 x 8 tile and the
# groups of 8 K indices, and a K split over the warps of a block
CASES = [(1, 2, 3, 4, 2, 1), (1, 8, 9, 17, 1, 2), (3, 4, 8, 8, 5, 3), (4, 9, 31, 33, 16, 4),
         (5, 7, 33, 40, 3, 5), (9, 17, 63, 65, 65, 6)]


@pytest.mark.parametrize("case", CASES, ids=lambda c: "x".join(map(str, c)))
@pytest.mark.parametrize("kw", [dict(), dict(k_slab=1), dict(t2sq_route=2), dict(alg7_route=1)],
                         ids=["auto", "slab1", "algs45", "alg7_blocked"])
def test_residual_matches_oracle(case, kw):
    s, Zc, t1, sig_ref, r1_ref, E_ref = oracle_case(*case)
    with context(s, **kw) as ctx:
        sig, sig1, E = ctx.residual(Zc, t1)
    # float64 sums of products: 1e-13 of the largest entry at these sizes
    assert np.abs(sig - sig_ref).max() < 1e-13 * max(1.0, np.abs(sig_ref).max())
    assert np.abs(sig1 - r1_ref).max() < 1e-13 * max(1.0, np.abs(r1_ref).max())
    assert abs(E - E_ref) < 1e-13 * max(1.0, abs(E_ref))
