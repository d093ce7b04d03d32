"""CPU model of the float-pair triangle with bounds and of the rule that chooses
it tile by tile, in numpy float32 (the kernels' operations one for one; the
constants are read from the kernels' source).

Bounded sums hold t G relative to a bound per output and chunk of grid points.
Their rms error is close to 2^-46.5 sqrt(16 sum_c b_c^2); an output that is accepted
has sqrt(16 sum_c b_c^2) <= 10 W (W = sum_I |E F G|, bounded from below by geometric
means), hence at most 2^-43.2 of W.  On the operands that are accepted here W is at
least twice that lower bound (3.4 times on Gaussian entries), so 2^-44.2 and, for the
largest of a few dozen outputs, 2^-42, the bound that the TwoSum form is held to.
Operands that vary over the grid points of a chunk, or are large at different
ones, have to be refused."""
import os
import re

import numpy as np
import pytest

from tests.test_df_model import exact, fma, max_scaled_error, split

f32 = np.float32
CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_2111_11473_gb300", "csrc")


def _constant(name, source):
    with open(os.path.join(CSRC, source)) as f:
        return float(re.search(r"constexpr \w+ %s = ([0-9.]+)f?;" % name, f.read()).group(1))


BC = int(_constant("kBiasChunk", "kernels.cuh"))
MIN_POINTS = int(_constant("kBiasMinPoints", "kernels.cuh"))
EVEN = _constant("kEven", "triangle_df.cu")


def bias_of(b):
    e = np.minimum((b * f32(1.001)).view(np.uint32) & np.uint32(0x7F800000), np.uint32(0x7D800000))
    return (e + np.uint32(0x01400000)).view(f32)


def bounded(E1, F2, E2, F1, G):
    """sum_I (E1 F2 + E2 F1) G by the kernel's sums."""
    nI, n = G.shape
    total = np.zeros(n)
    for lo in range(0, nI, BC):
        c = slice(lo, min(nI, lo + BC))
        mx = [np.abs(a[c].astype(f32)).max(0) for a in (E1, F2, E2, F1, G)]
        p1, p2 = mx[0] * mx[1], mx[2] * mx[3]
        s, cb = bias_of(np.maximum(p1, p2)), bias_of((p1 + p2) * mx[4])
        units, low = np.zeros(n), np.zeros(n, f32)
        for I in range(c.start, c.stop):
            (aH, aL), (bH, bL), (cH, cL), (dH, dL), (gH, gL) = (
                split(a[I]) for a in (E1, F2, E2, F1, G))
            z1, z2 = s - fma(aH, bH, s), s - fma(dH, cH, s)
            r1, r2 = fma(aH, bH, z1), fma(dH, cH, z2)
            r1, r2 = fma(aH, bL, r1), fma(dH, cL, r2)
            r1, r2 = fma(aL, bH, r1), fma(dL, cH, r2)
            th, tl = -(z1 + z2), r1 + r2
            h = fma(th, gH, cb)
            p = fma(tl, gH, fma(th, gL, fma(th, gH, cb - h)))
            units += h.astype(np.float64) - cb.astype(np.float64)   # exact: the integer sum
            low = low + p
        total += units + low
    return total


def chunk_stats(a):
    """Largest |a| (bf16, rounded up) and geometric mean (bf16, rounded down) of every chunk."""
    a = np.abs(a.astype(f32))
    chunks = [a[lo:lo + BC] for lo in range(0, len(a), BC)]
    m = np.array([c.max(0) for c in chunks])
    with np.errstate(divide="ignore"):
        g = np.array([np.exp2(np.log2(c).mean(0, dtype=f32)) for c in chunks], dtype=f32)
    up = ((m.view(np.uint32) + np.uint32(0xFFFF)) & np.uint32(0xFFFF0000)).view(f32)
    return up, (g.view(np.uint32) & np.uint32(0xFFFF0000)).view(f32)


def uneven(EY, EZ, FY, FZ, G1, G2):
    """The rule of k_bias_check for 32 X and one tile: E, F (nI, 32, 16) of both sides, G^YZ
    and G^ZY (nI, 16, 16), both indexed [Y, Z]."""
    Y, Z = np.meshgrid(np.arange(16), np.arange(16), indexing="ij")
    stats = [chunk_stats(a) for a in (EY, EZ, FY, FZ, G1, G2)]
    n = np.array([min(BC, len(G1) - lo) for lo in range(0, len(G1), BC)])[:, None, None]
    for lane in (0, 1):
        X = 2 * ((Y + Z) % 16) + lane
        (mEY, gEY), (mEZ, gEZ), (mFY, gFY), (mFZ, gFZ) = (
            [a[:, X, i] for a in s] for s, i in zip(stats, (Y, Z, Y, Z)))
        for mG, gG in stats[4:]:
            b = (mEY * mFZ + mFY * mEZ) * mG
            v = ((gEY * gFZ + gFY * gEZ) * gG * n).sum(0) * (EVEN / 4)
            sb, mb = b.sum(0), b.max(0)
            with np.errstate(divide="ignore", invalid="ignore", over="ignore"):
                good = (mb > 2.0 ** -100) & (mb < 2.0 ** 120) & (mb / v * (sb / v) <= 1.0)
            if not np.all((mb == 0) | good):
                return True
    return False


def operands(kind, nI, seed, nX=32, T=16):
    """E, F of both sides and both G of one tile."""
    r = np.random.default_rng(seed)
    I = np.arange(nI)
    out = []
    for shape in [(nI, nX, T)] * 4 + [(nI, T, T)] * 2:
        x = r.standard_normal(shape)
        name, _, arg = kind.partition("_")
        if name == "spread":          # magnitudes over 2^-arg .. 1
            x *= 2.0 ** r.integers(-int(arg), 1, size=shape)
        elif name == "decay":         # exp(-I / arg)
            x *= np.exp(-I / float(arg))[:, None, None]
        elif name == "apart":         # a maximum of width arg at a grid point of its own
            x *= np.exp(-np.abs(I[:, None, None] - r.integers(0, nI, (1,) + shape[1:])) / float(arg))
        elif name == "point":         # one grid point stands out
            x *= np.where(I == int(arg), 1.0, 1e-4)[:, None, None]
        elif name == "halves":        # large at even or at odd grid points
            odd = (I[:, None, None] + r.integers(0, 2, (1,) + shape[1:])) % 2
            x *= np.where(odd, 1.0, 2.0 ** -int(arg))
        elif name == "element" and len(out) == int(arg):    # one element at one grid point
            x[5, shape[1] // 2 + 1, 9] *= 1e5
        out.append(x)
    return out


UNEVEN = ["spread_4", "spread_40", "decay_2", "decay_8", "decay_32", "apart_8", "apart_32",
          "point_0", "point_8", "point_13", "halves_12", "element_0", "element_3", "element_4"]


@pytest.mark.parametrize("nI", [MIN_POINTS, 601, 1200])
@pytest.mark.parametrize("kind", ["gauss", "zeros"] + UNEVEN)
def test_choice_and_accuracy(kind, nI):
    ops = operands(kind, nI, 3)
    if kind == "zeros":
        for a in ops[:4]:
            a[:] = 0.0
    refused = uneven(*ops)
    assert refused == (kind in UNEVEN)
    if refused or kind == "zeros":
        return
    r = np.random.default_rng(4)
    x, y, z = r.integers(0, 8, 24), r.integers(0, 16, 24), r.integers(0, 16, 24)
    EY, EZ, FY, FZ, G1, G2 = ops
    o = EY[:, x, y], FZ[:, x, z], EZ[:, x, z], FY[:, x, y], G1[:, y, z]
    err = max_scaled_error(bounded(*o), exact(*o), *o)
    print(f"{kind} {nI}: {err:.2e} of sum |E F G| (2^-42 = {2.0 ** -42:.2e})")
    assert err < 2.0 ** -42


def test_bounded_sums_would_miss_the_bound_on_uneven_operands():
    """What the rule is for: entries spread over 2^-40 .. 1."""
    EY, EZ, FY, FZ, G1, G2 = operands("spread_40", 600, 5)
    i = np.arange(16)
    o = EY[:, 0, :], FZ[:, 0, :], EZ[:, 0, :], FY[:, 0, :], G1[:, i, i]
    assert max_scaled_error(bounded(*o), exact(*o), *o) > 2.0 ** -40
