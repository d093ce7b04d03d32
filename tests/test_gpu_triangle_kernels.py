"""The triangle kernels alone on given operands (needs a GB300).

Float pairs: operands of one scale, spread over many binades and decaying over
the grid, for tiles of both forms in one launch.  Bound: a term is stated to
carry an error of about 2^-45 of |E F G|; the errors of different terms and
outputs are independent, so that their rms over W = sum_I |E F G| is at most
2^-45, and 2^-44 with the float32 low words that collect them.

Float32 (paired and unpaired): three roundings per term and one per addition,
(nI + 4) 2^-24 of W at worst."""
import ctypes as C

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__ as g
    g.build()


def _triangle(kind, E, F, G):
    import paper_2111_11473_gb300 as pkg
    nI, nX, P = E.shape
    H = np.zeros((nX, P, P))
    tiles, uneven = C.c_int(0), C.c_int(0)
    lib = pkg.load_library()
    lib.thc_diag_triangle.restype = C.c_int
    args = [np.ascontiguousarray(a, dtype=np.float64) for a in (E, F, G)] + [H]
    st = lib.thc_diag_triangle(kind, P, nX, nI, *[C.c_void_p(a.ctypes.data) for a in args],
                               C.byref(tiles), C.byref(uneven), C.c_void_p(0))
    assert st == 0
    return H, tiles.value, uneven.value


def _operands(kind, P, nX, nI, seed=1):
    r = np.random.default_rng(seed)
    E, F, G = (r.standard_normal(s) for s in ((nI, nX, P), (nI, nX, P), (nI, P, P)))
    if kind.startswith("decay"):
        w = np.exp(-np.arange(nI) / float(kind[5:]))[:, None, None]
        E, F, G = E * w, F * w, G * w
    elif kind.startswith("spread"):
        E, F, G = (a * 2.0 ** r.integers(-int(kind[6:]), 1, size=a.shape) for a in (E, F, G))
    elif kind == "mirror":      # G^ZY (Z > Y) far below G^YZ
        G = np.where(np.arange(P)[:, None] > np.arange(P), G * 2.0 ** -20, G)
    elif kind == "half":        # the columns of the upper half are spread
        h = P // 32 * 16
        for a in (E, F):
            a[:, :, h:] *= 2.0 ** r.integers(-40, 1, size=a[:, :, h:].shape)
    return E, F, G


def _reference(E, F, G):
    """H and W = sum |E F G| (long double)."""
    L = np.longdouble
    H, W = 0, 0
    for e, f, g in zip(E.astype(L), F.astype(L), G.astype(L)):
        p = e[:, :, None] * f[:, None, :]
        H = H + (p + p.transpose(0, 2, 1)) * g
        p = abs(p.astype(np.float64))
        W = W + (p + p.transpose(0, 2, 1)) * abs(g.astype(np.float64))
    return H, W


@pytest.mark.parametrize("kind", ["one_scale", "mirror", "spread40", "decay2", "decay4", "half"])
@pytest.mark.parametrize("size", [(40, 5, 600), (33, 9, 613), (64, 8, 512), (17, 3, 511)],
                         ids=lambda s: "x".join(map(str, s)))
def test_float_pairs(kind, size):
    P, nX, nI = size
    E, F, G = _operands(kind, P, nX, nI)
    H, tiles, uneven = _triangle(1, E, F, G)
    ref, W = _reference(E, F, G)
    rms = np.sqrt(np.mean((np.asarray(H - ref, dtype=np.float64) / W) ** 2))
    print(f"{kind} {size}: rms 2^{np.log2(rms):.2f} of sum |E F G|, {uneven} of {tiles} tiles uneven")
    assert rms < 2.0 ** -44
    if nI < 512:
        assert uneven == 0       # (not looked at: every tile takes the TwoSum form)
    elif kind == "half":
        assert 0 < uneven < tiles
    else:
        assert uneven == (0 if kind in ("one_scale", "mirror") else tiles)


def test_float_pairs_not_finite():
    for value in (np.inf, np.nan):
        E, F, G = _operands("one_scale", 20, 3, 520)
        E[77, 1, 4] = value
        H = _triangle(1, E, F, G)[0]
        assert not np.isfinite(H[1, 4, :]).any() and not np.isfinite(H[1, :, 4]).any()
        assert np.isfinite(H[0]).all() and np.isfinite(H[2]).all()


@pytest.mark.parametrize("kind", [0, 2, 3], ids=["float64", "paired", "unpaired"])
@pytest.mark.parametrize("size", [(1, 1, 1), (5, 3, 7), (33, 9, 65), (70, 33, 31), (64, 64, 40)],
                         ids=lambda s: "x".join(map(str, s)))
def test_plain_kernels(kind, size):
    P, nX, nI = size
    E, F, G = _operands("one_scale", P, nX, nI)
    if kind:
        E, F, G = (a.astype(np.float32).astype(np.float64) for a in (E, F, G))
    H = _triangle(kind, E, F, G)[0]
    ref, W = _reference(E, F, G)
    bound = (nI + 4) * 2.0 ** (-24 if kind else -53)
    assert (np.abs(np.asarray(H - ref, dtype=np.float64)) <= bound * W).all()
