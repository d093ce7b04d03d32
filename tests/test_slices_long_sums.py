"""Float64 products by slices whose sums come near the ends of their fixed-point
range: the constants of the kernel's source against the range of a level's float32
sum and of the 64-bit sums, and a product of 65536 K indices in one tile with
entries of one sign just below a power of two (needs a GB300)."""
import os
import re

import numpy as np
import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_2111_11473_gb300", "csrc")
with open(os.path.join(CSRC, "gemm_tc.cu")) as f:
    SOURCE = f.read()


def _int(pattern):
    return int(re.search(pattern, SOURCE).group(1), 0)


SLICES = _int(r"constexpr int kSlices = (\d+);")
LEVELS = _int(r"constexpr int kLevels = (\d+);")
STEPS = _int(r"constexpr int kMaxSteps = (\d+);")
TABLE = _int(r"\((0x[0-9A-Fa-f]+)ULL >> \(8 \* \(__ffs\(i \| 16\) - 1\)\)\)")


def _fresh(i):
    """Levels that K step i starts afresh, from the kernel's table."""
    return TABLE >> (8 * ((i | 16) & -(i | 16)).bit_length() - 8) & 0x7F


def test_exact_levels_are_drained_before_2_to_24():
    assert (SLICES, LEVELS) == (7, 7)
    for q in range(LEVELS):
        starts = [i for i in range(256) if _fresh(i) >> q & 1]
        assert starts[0] == 0
        steps = max(b - a for a, b in zip(starts, starts[1:] + [256]))
        largest = (q + 1) * 64 * steps * 128 * 128
        # levels 0 - 4 are exact; 5 and 6 pass 2^24 by less than a factor of 4 (units of 1, 2)
        assert largest <= 2 ** 24 if q <= 4 else largest < 2 ** 26


def test_64_bit_sums_hold_the_longest_tile():
    """H counts 2^-46 of the scale, a K index adds at most 2^46 (two entries of 1), and
    `hshift` more bits are kept only where 2^62 is not passed."""
    for steps in (1, 2, 3, 15, 16, 1000, STEPS):
        kmax = steps * 64
        hshift = max(0, min(16, 16 - (kmax - 1).bit_length()))
        assert kmax * 2 ** 46 * 2 ** hshift <= 2 ** 62


@pytest.mark.gpu
def test_longest_sum_of_one_sign():
    """M = U te of CP-ALS with 65536 projectors in 80 tiles (K is then not split), entries
    of U and te in 0.9 .. 1.  y_o = R S^-1 with R_i^X = sum_a M_ia^X y_a^X is backward
    stable: y_o S differs from R by a modest multiple of 2^-53 of |y_o| |S|, for which
    1e-13 leaves a factor of 1000."""
    import __graft_entry__ as g
    g.build()
    from paper_2111_11473_gb300 import binding
    o, v, N, W = 8, 152, 65536, 512
    r = np.random.default_rng(3)
    yo, yv = (r.standard_normal((m, W)) for m in (o, v))
    U, tau = (1.0 - 0.1 * r.random(s) for s in ((o * v, N), (N, W)))
    got = binding.cp_als(U, np.ones(N), yo, yv, tau, iters=1)[0].astype(np.longdouble)
    S = ((yv.T @ yv) * (tau.T @ tau)).astype(np.longdouble)
    for i, X in ((0, 0), (3, 77), (7, 511)):
        M = [(U[i * v + a].astype(np.longdouble) * tau[:, X]).sum() for a in range(v)]
        R = (np.array(M) * yv[:, X]).sum()
        bound = 1e-13 * (np.abs(got[i]) @ np.abs(S[:, X]))
        print(f"y_o S - R: {float(got[i] @ S[:, X] - R):.2e} (R {float(R):.2e}, bound {float(bound):.2e})")
        assert bound < 1e-3 * abs(R) and abs(got[i] @ S[:, X] - R) < bound
