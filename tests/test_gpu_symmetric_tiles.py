"""Symmetric 16- and 32-wide tiles of the float64 triangle and of the symmetry
check of the amplitudes, around their edges (needs a GB300).

Bound: float64 sums, 1e-10 as for the other float64 residuals."""
import numpy as np
import pytest

from tests.gpu_util import context, oracle_case

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__ as g
    g.build()


@pytest.mark.parametrize("P", [15, 16, 17, 31, 32, 33, 47, 65])
@pytest.mark.parametrize("kw", [dict(), dict(x_block6=5, i_chunk=7)], ids=["auto", "blocked"])
def test_residual_at_tile_edges(P, kw):
    s, Zc, t1, sig_ref, r1_ref, E_ref = oracle_case(3, 6, P, 19, 7, P)
    with context(s, **kw) as ctx:
        sig, sig1, E = ctx.residual(Zc, t1)
    assert np.abs(sig - sig_ref).max() < 1e-10
    assert np.abs(sig1 - r1_ref).max() < 1e-10
    assert abs(E - E_ref) < 1e-9


@pytest.mark.parametrize("P", [1, 31, 32, 33, 70])
@pytest.mark.parametrize("bad", ["asymmetric", "nan", "inf"])
def test_symmetry_check_refuses(P, bad):
    import paper_2111_11473_gb300 as pkg
    if P == 1 and bad == "asymmetric":
        pytest.skip("1 x 1 is symmetric")
    s, Zc, t1 = oracle_case(2, 4, P, 9, 5, 1)[:3]
    Zc = Zc.copy()
    r, c = P - 1, 0                   # corner of the last tile row
    if bad == "asymmetric":
        Zc[r, c] += 1e-3 * max(1.0, np.abs(Zc).max())
    else:
        Zc[r, c] = Zc[c, r] = np.nan if bad == "nan" else -np.inf
    with context(s) as ctx:
        with pytest.raises(pkg.ThcError):
            ctx.residual(Zc, t1)
