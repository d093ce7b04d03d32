"""The float-pair triangle with bounds (512 grid points or more): the residual
with only the triangle in float pairs against the float64 triangle, at odd
sizes, grid chunks that are and are not whole bound chunks, X blocks and a
large spread of magnitudes (needs a GB300).

Bound: with |term| <= b (the product of the largest |E|, |F|, |G| of 16 grid
points, twice), a term is off by at most 2^-45 b (remainder, low products and
their float32 sum of 16), against b <= 64 rms on these Gaussian-like operands:
2^-39 = 2e-12 of the rms term, summed over G terms and projected; 1e-11 of the
largest residual entry leaves room for cancellation between the terms."""
import numpy as np
import pytest

from synth import make_system, random_amplitudes
from tests.gpu_util import context

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__ as g
    g.build()


@pytest.mark.parametrize("size", [(3, 5, 35, 513, 9), (2, 7, 33, 541, 6), (4, 9, 64, 512, 12),
                                  (3, 6, 1, 600, 5)], ids=lambda s: "x".join(map(str, s)))
@pytest.mark.parametrize("kw", [dict(), dict(i_chunk=48), dict(i_chunk=37), dict(x_block6=7),
                                dict(workspace_bytes=1 << 20)],
                         ids=["auto", "whole_chunks", "ragged_chunks", "x6_7", "rebuilt_g"])
def test_matches_float64_triangle(size, kw):
    o, v, P, G, K = size
    s = make_system(o, v, P, G, K, 3)
    Zc, t1 = random_amplitudes(P, o, v, seed=4, t1_scale=0.05, t2_scale=0.5)
    out = []
    for pol in ("fp64", "fp64tc"):
        with context(s, policy={"triangle": pol}, t2sq_route=1, **kw) as ctx:
            out.append(ctx.residual(Zc, t1))
    scale = np.abs(out[0][0]).max()
    assert np.abs(out[1][0] - out[0][0]).max() < 1e-11 * scale


def test_spread_of_magnitudes_and_zeros():
    """Amplitude columns over 2^-20 .. 1, some of them zero."""
    o, v, P, G, K = 3, 6, 34, 530, 8
    s = make_system(o, v, P, G, K, 5)
    rng = np.random.default_rng(6)
    w = np.exp2(-rng.integers(0, 21, P)) * (rng.random(P) > 0.2)
    Zc, t1 = random_amplitudes(P, o, v, seed=7, t1_scale=0.05, t2_scale=0.5)
    Zc = Zc * w[:, None] * w[None, :]
    out = []
    for pol in ("fp64", "fp64tc"):
        with context(s, policy={"triangle": pol}, t2sq_route=1) as ctx:
            out.append(ctx.residual(Zc, t1))
    scale = np.abs(out[0][0]).max()
    assert np.abs(out[1][0] - out[0][0]).max() < 1e-11 * scale
