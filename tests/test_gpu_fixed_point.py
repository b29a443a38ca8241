"""The FP64 kernels' fixed-point column scaling and products at the edges of
their range: column bounds met exactly, columns of extreme or zero scale,
entries that are not finite, and both lane splits of the minors.

Tolerance: entries are rounded once at 2^-62 of a column's bound S_j = sum
M (|Re a| + |Im a|), a pair of columns loses at most a few units of 2^-50 of
the bounds' product in the worst case (column sums of sqrt(2n) below their
bound, 2^-64 products of them), so K columns stay within K 2^-50 of the
modulus sum of the addends (oracle.perm_mult_abs), far inside 1e-12 of it."""
import math

import numpy as np
import pytest

import oracle
import synthetic as S

pytestmark = pytest.mark.gpu

REL = 1e-12  # of the modulus sum of the addends


def _minors_ref(a, M, N):
    """Each minor as a permanent with multiplicities of the other columns."""
    K = a.shape[1]
    keep = [[j for j in range(K) if j != l] for l in range(K)]
    return np.array([sum(oracle.perm_mult(a[:, k], M, N[k])) for k in keep])


@pytest.mark.parametrize("n", [1, 2, 3, 4, 8, 12, 16])
def test_column_sums_at_their_bound(ctx, n):
    """All-ones matrices: the largest column sum is the column bound itself, a
    power of two at n = 1, 2, 4, 8, 16.  Up to n = 8 every addend is an integer
    below 2^24, and permanents and minors are exact; above, within REL of the
    modulus sum."""
    ones = np.ones(n, np.int32)
    J = np.ones((n, n))
    p, q = ctx.perm(J, ones, ones), ctx.perm(-1j * J, ones, ones)
    f = math.factorial(n)
    m = ctx.laplace_minors(J[1:], ones[1:], ones) if n > 1 else np.ones(1)
    if n <= 8:
        assert p == f and q == (-1j) ** n * f
        assert np.array_equal(m, np.full(n, math.factorial(n - 1), np.complex128))
    else:
        tol = REL * oracle.perm_mult_abs(J, ones, ones)
        assert abs(p - f) <= tol and abs(q - (-1j) ** n * f) <= tol
        assert np.all(np.abs(m - math.factorial(n - 1)) <= REL * oracle.perm_mult_abs(J[1:, 1:], ones[1:], ones[1:]))


@pytest.mark.parametrize("K", [5, 12, 33, 36])
@pytest.mark.parametrize("scales", ["huge", "tiny", "mixed"])
def test_extreme_column_scales(ctx, K, scales):
    """Columns scaled by powers of two far apart: the result scales exactly."""
    M = np.ones(K, np.int32) if K <= 12 else np.array([K // 3] * 2 + [K - 2 * (K // 3)], np.int32)
    a = S.random_complex(len(M), K, 60 + K)
    ex = {"huge": np.full(K, 20), "tiny": np.full(K, -20), "mixed": np.where(np.arange(K) % 2, 300, -300)}[scales]
    if K % 2 and scales == "mixed":
        ex = ex.copy()
        ex[-1] = 0
    b = a * np.exp2(ex.astype(float))[None, :]
    N = np.ones(K, np.int32)
    p, q = ctx.perm(a, M, N), ctx.perm(b, M, N)
    assert q == complex(math.ldexp(p.real, int(ex.sum())), math.ldexp(p.imag, int(ex.sum())))
    M2 = M.copy()
    M2[0] -= 1
    keep = M2 > 0
    m, w = ctx.laplace_minors(a[keep], M2[keep], N), ctx.laplace_minors(b[keep], M2[keep], N)
    for l in range(K):
        e = int(ex.sum() - ex[l])
        assert w[l] == complex(math.ldexp(m[l].real, e), math.ldexp(m[l].imag, e)), l


@pytest.mark.parametrize("K", [2, 3, 7, 31, 35])
def test_zero_columns_and_structured_zeros(ctx, K):
    """A zero column makes the permanent and every minor but its own exactly
    zero; that minor matches the oracle."""
    rows = K - 1 if K <= 7 else 4
    M = np.full(rows, (K - 1) // rows, np.int32)
    M[0] += K - 1 - M.sum()
    a = S.random_complex(rows, K, 90 + K)
    a[:, K // 2] = 0
    N = np.ones(K, np.int32)
    got = ctx.laplace_minors(a, M, N)
    ref = _minors_ref(a, M, N)
    others = np.arange(K) != K // 2
    assert np.all(got[others] == 0)
    keep = [j for j in range(K) if j != K // 2]
    assert abs(got[K // 2] - ref[K // 2]) <= REL * oracle.perm_mult_abs(a[:, keep], M, N[keep])


@pytest.mark.parametrize("bad", [np.nan, np.inf, -np.inf])
@pytest.mark.parametrize("K", [2, 6, 13])
def test_entries_that_are_not_finite(ctx, bad, K):
    """Such an entry gives NaN wherever its column enters the product; the
    minor without that column stays a number."""
    ones = np.ones(K, np.int32)
    a = S.random_complex(K, K, 110 + K)
    a[0, 1] = bad
    v = ctx.perm(a, ones, ones)
    assert math.isnan(v.real) and math.isnan(v.imag)
    got = ctx.laplace_minors(a[:K - 1], ones[1:], ones)
    assert np.all(np.isnan(got[np.arange(K) != 1]))
    clean = a[:K - 1].copy()
    clean[0, 1] = 0
    ref = _minors_ref(clean, ones[1:], ones)[1]
    keep = [j for j in range(K) if j != 1]
    assert abs(got[1] - ref) <= REL * oracle.perm_mult_abs(clean[:, keep], ones[1:], ones[1:])
    assert ctx.perm(np.array([[1.5 + 0.5j]]), [1], [1]) == 1.5 + 0.5j


@pytest.mark.parametrize("M", [[1] * 9, [2] * 5, [3, 1, 2, 2, 1, 1], [9], [1, 1, 7], [4, 4, 1], [1, 2, 1, 4, 1],
                               [1, 1, 1, 1, 2, 3], [1, 1, 1, 1, 1, 4]])
def test_minors_runs_end_where_the_weight_changes(ctx, M):
    """Integer runs of the minors: rows of every kind (no, one, two, three and
    more binary digits before the repeated ones), odd and even widths."""
    M = np.array(M, np.int32)
    K = int(M.sum()) + 1
    a = S.random_complex(len(M), K, 130 + K)
    N = np.ones(K, np.int32)
    got, ref = ctx.laplace_minors(a, M, N), _minors_ref(a, M, N)
    for l in range(K):
        keep = [j for j in range(K) if j != l]
        assert abs(got[l] - ref[l]) <= REL * oracle.perm_mult_abs(a[:, keep], M, N[keep]), l
