"""CP-ALS products where the large entries of one operand meet small ones of the
other: eigenvalues over decades and U large where they are small.

The products may run as integer slices only if every output's sum |a b| reaches
the scale 2^(e_i + e_j) that its slices are cut at: K terms by slices are then off
by at most K 2^-53 sum |a b|, as float64 sums are.  On the CPU: the rule (a lower
bound of the sum from the first digits) on a model of the slices.  On the GPU:
y_o after one sweep against products formed in long double."""
import numpy as np
import pytest


def _slices(A):
    """Digits (7, R, K) and exponents (R,) of the rows of A."""
    m = np.abs(A).max(1)
    e = np.where(m > 0, np.frexp(m)[1], 0)
    V = np.rint(np.ldexp(A.astype(np.longdouble), (55 - e)[:, None])).astype(np.int64)
    d = []
    for _ in range(6):
        low = ((V + 128) & 255) - 128
        d.append(low)
        V = (V - low) >> 8
    return np.array(([V] + d[::-1])), e


def _product(A, B):
    """A B^T by slices, and the rule's word for it."""
    (a, ea), (b, eb) = _slices(A), _slices(B)
    total = 0
    for l in range(2, 9):
        S = sum(a[t - 1].astype(float) @ b[l - t - 1].astype(float).T
                for t in range(1, 8) if 1 <= l - t <= 7)
        total = total + S.astype(np.longdouble) * np.longdouble(2.0) ** (2 - 8 * l)
    first = [np.maximum(2 * np.abs(d[0]) - 1, 0) for d in (a, b)]
    assert max(f.max() for f in first) <= 255           # bytes
    uneven = bool((first[0] @ first[1].T < 66200).any())
    return np.ldexp(total, ea[:, None] + eb[None, :]), uneven


def _operands(kind, K, seed, n=24):
    r = np.random.default_rng(seed)
    A, B = r.standard_normal((n, K)), r.standard_normal((n, K))
    w = 10.0 ** (-6.0 * np.arange(K) / K)
    if kind == "opposed":             # A grows where B falls
        A, B = A / w, B * w * w
    elif kind == "one_entry":         # one large entry of a row meets nothing large
        A[3, 7] *= 1e9
    elif kind == "both_fall":
        A, B = A * w ** 0.05, B * w ** 0.05
    elif kind == "products":          # heavy tails, as Khatri-Rao rows have
        A, B = A * r.standard_normal((n, K)), B * r.standard_normal((n, K))
    return A, B


@pytest.mark.parametrize("kind,K,uneven", [("gauss", 100, False), ("gauss", 300, False),
                                           ("both_fall", 300, False), ("products", 2000, False),
                                           ("opposed", 300, True), ("one_entry", 300, True),
                                           ("gauss", 2, True)])
def test_rule_keeps_the_bound_of_float64_sums(kind, K, uneven):
    A, B = _operands(kind, K, 5)
    C, refused = _product(A, B)
    assert refused == uneven
    exact = A.astype(np.longdouble) @ B.astype(np.longdouble).T
    W = np.abs(A) @ np.abs(B).T
    err = float((np.abs(C - exact) / W).max())
    print(f"{kind} K={K}: {err:.2e} of sum |a b| (K 2^-53 = {K * 2.0 ** -53:.2e})")
    if not uneven:
        assert err <= K * 2.0 ** -53
    if kind == "opposed":
        assert err > 2.0 ** -43       # what the rule is for


@pytest.mark.gpu
@pytest.mark.parametrize("decades", [0, 3, 6])
def test_eigenvalues_over_decades(decades):
    """Bound: the sums of M = U te have at most K 2^-53 of sum |a b|, carried through
    the reduction and the solve by the condition number of S; a factor 4 for sum |a b|
    over the entries themselves."""
    import __graft_entry__ as g
    g.build()
    from paper_2111_11473_gb300 import binding
    o, v, N, W = 12, 60, 300, 100
    r = np.random.default_rng(1)
    yo, yv, tau = (r.standard_normal((m, W)) for m in (o, v, N))
    eps = 10.0 ** (-decades * np.arange(N) / N)
    U = (yo[:, None, :] * yv[None, :, :]).reshape(o * v, W) @ (tau / np.sqrt(W)).T / eps
    yo, yv, tau = (a + 0.1 * r.standard_normal(a.shape) for a in (yo, yv, tau))
    got = binding.cp_als(U, eps, yo, yv, tau, iters=1)[0]
    te = eps[:, None] ** 2 * tau
    M = U.astype(np.longdouble) @ te.astype(np.longdouble)
    R = (M.reshape(o, v, W) * yv[None]).sum(1).astype(np.float64)
    S = (yv.T @ yv) * (tau.T @ te)
    ref = np.linalg.solve(S, R.T).T
    err = np.abs(got - ref).max() / np.abs(ref).max()
    bound = 4 * N * np.linalg.cond(S) * 2.0 ** -53
    print(f"{decades} decades: y_o off by {err:.2e} of its largest entry (bound {bound:.2e})")
    assert err < bound
