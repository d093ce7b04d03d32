"""The balanced 8-bit slices of the float64 tensor-core products: a CPU model
of the scheme (csrc/gemm_tc.cu) against exact rational arithmetic, and the
kernel at the edges of its tiles, K steps and drain periods (needs a GB300)."""
from fractions import Fraction

import numpy as np
import pytest

SLICES, LMAX = 7, 8


def digits(x, e):
    """7 balanced base-256 digits of x 2^(55 - e), |x| < 2^e, most significant first."""
    v = Fraction(x) * Fraction(2) ** (55 - e)
    V = int(abs(v) + Fraction(1, 2)) * (1 if x >= 0 else -1)     # round half up
    out = []
    for _ in range(SLICES - 1):
        d = ((V + 128) & 255) - 128
        out.append(d)
        V = (V - d) >> 8
    return [V] + out[::-1]


def row_exponent(a):
    m = np.abs(a).max()
    return 0 if m == 0 else int(np.frexp(m)[1])


@pytest.mark.parametrize("spread", [0, 12, 60])
def test_digits_and_products_within_derived_bounds(spread):
    rng = np.random.default_rng(spread)
    K = 40
    a = rng.standard_normal(K) * np.exp2(-rng.integers(0, spread + 1, K))
    b = rng.standard_normal(K) * np.exp2(-rng.integers(0, spread + 1, K))
    ea, eb = row_exponent(a), row_exponent(b)
    da, db = [digits(x, ea) for x in a], [digits(x, eb) for x in b]
    for x, e, d in [(x, ea, d) for x, d in zip(a, da)] + [(x, eb, d) for x, d in zip(b, db)]:
        assert all(-128 <= q <= 128 for q in d)          # exact in bf16
        value = sum(Fraction(q) * Fraction(2) ** (1 - 8 * (t + 1)) for t, q in enumerate(d))
        assert abs(Fraction(x) / Fraction(2) ** e - value) <= Fraction(1, 2 ** 56)
    total = Fraction(0)
    for l in range(2, LMAX + 1):
        S = sum(da[k][t] * db[k][l - 2 - t] for k in range(K)
                for t in range(SLICES) if 0 <= l - 2 - t < SLICES)
        total += Fraction(S) * Fraction(2) ** (2 - 8 * l)
    exact = sum(Fraction(x) * Fraction(y) for x, y in zip(a, b)) / Fraction(2) ** (ea + eb)
    # pairs left out: 6 at level 9 (at most 2^14 2^-70 each) and less than one
    # more from the levels beyond; two remainders of 2^-56
    assert abs(total - exact) <= K * Fraction(9, 2 ** 56)


@pytest.mark.parametrize("value", [1.0, np.nextafter(1.0, 0.0), -0.5, 2.0 ** -55, 2.0 ** -57, 0.0])
def test_extreme_digits(value):
    e = 1 if value == 1.0 else 0
    d = digits(value, e)
    assert all(-128 <= q <= 128 for q in d)


# Level q = l - 2 sums (q + 1) pairs; drained every PERIOD[q] steps of 64.
PERIOD = [16, 8, 4, 4, 2, 4, 8]


def test_level_sums_stay_exact_between_drains():
    for q in range(5):
        assert (q + 1) * 64 * PERIOD[q] * 128 * 128 <= 2 ** 24
    # the levels that start afresh at step i, as the kernel's table has them
    table = 0x7F7E3C1000
    for i in range(64):
        tz = (i | 16) & -(i | 16)
        fresh = (table >> (8 * (tz.bit_length() - 1))) & 0x7F
        assert fresh == sum(1 << q for q in range(7) if i % PERIOD[q] == 0)


@pytest.mark.gpu
@pytest.mark.parametrize("seed", [11, 12, 13, 14])
def test_kernel_at_tile_edges(seed):
    """Every fourth case has M, N, K at the edges (1, 16, 17, 63 .. 129, K up
    to 1025); all within 1e-15 (K + 1) of the CUDA-core product."""
    import __graft_entry__ as g
    g.build()
    import paper_2111_11473_gb300 as pkg
    status, max_rel, failures = pkg.binding.selftest_gemm_f64(cases=96, seed=seed)
    assert status == "THC_OK" and failures == 0
    assert max_rel < 1e-13
