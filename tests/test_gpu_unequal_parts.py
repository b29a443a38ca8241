"""FP64 results where real and imaginary parts differ by orders of magnitude:
each part keeps its own relative accuracy, as with products of doubles (a
derivative by a small imaginary step comes out of the imaginary part).

Reference: the addends in rational arithmetic.  Tolerance: a part of an addend
is a sum of products with one factor of every column; S sums, over the addends,
the moduli of those products that belong to the part.  Products of doubles err
by 2^-52 each in every product, K of them, and their sum, the weight and the
scaled sums once more: 2 (K + 2) 2^-52 S.  Columns whose parts' bounds are
within 1/8 of one another are rounded at the larger one's scale instead, K
pairs by 2^-53 of the moduli, at most 8 S: 8 (K + 2) 2^-52 S covers both."""
import itertools
from fractions import Fraction

import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu


def addends(a, keep):
    """Exact permanent (re, im) of columns `keep` of a (distinct rows), and S
    of both parts, by the Glynn sum."""
    n = len(keep)
    cols = [[(Fraction(float(z.real)), Fraction(float(z.imag))) for z in a[:, j]] for j in keep]
    re = im = Fraction(0)
    sre = sim = 0.0
    for signs in itertools.product((1, -1), repeat=n - 1):
        d = (1,) + signs
        x, y = Fraction(1), Fraction(0)
        ax, ay = 1.0, 0.0
        for col in cols:
            p = sum(s * z[0] for s, z in zip(d, col))
            q = sum(s * z[1] for s, z in zip(d, col))
            x, y = x * p - y * q, x * q + y * p
            fp, fq = float(abs(p)), float(abs(q))
            ax, ay = ax * fp + ay * fq, ax * fq + ay * fp
        w = -1 if signs.count(-1) % 2 else 1
        re, im = re + w * x, im + w * y
        sre, sim = sre + ax, sim + ay
    f = Fraction(1, 2 ** (n - 1))
    return re * f, im * f, sre * float(f), sim * float(f)


def check(got, a, keep):
    re, im, sre, sim = addends(a, keep)
    tol = 8.0 * (len(keep) + 2) * 2.0 ** -52
    assert abs(float(Fraction(got.real) - re)) <= tol * sre
    assert abs(float(Fraction(got.imag) - im)) <= tol * sim


def matrix(R, K, h, seed):
    g = np.random.Generator(np.random.PCG64(seed))
    return g.standard_normal((R, K)) + 1j * h * g.standard_normal((R, K))


H = [0.5, 0.1, 1e-2, 1e-6, 1e-9, 1e-12, 1e-20, 1e-200, 1e12]


@pytest.mark.parametrize("h", H)
@pytest.mark.parametrize("K", [1, 2, 3, 5, 8])
def test_small_parts(ctx, K, h):
    ones = np.ones(K, np.int32)
    a = matrix(K, K, h, 7 * K)
    for mode in (0, 2):
        check(ctx.perm(a, ones, ones, mode=mode), a, range(K))
    r = matrix(K, K + 1, h, 7 * K + 1)
    got = ctx.laplace_minors(r, ones, np.ones(K + 1, np.int32))
    for l in range(K + 1):
        check(got[l], r, [j for j in range(K + 1) if j != l])


@pytest.mark.parametrize("f", ["ryser", "nw"])
@pytest.mark.parametrize("h", [1e-2, 1e-9, 1e-20])
def test_small_parts_of_formulas(ctx, f, h):
    """Their sums and addends differ: ten times the bound of the Glynn sum's."""
    for K in (1, 2, 5):
        a = matrix(K, K, h, K)
        re, im, sre, sim = addends(a, range(K))
        got = ctx.perm_formula(a, f)
        tol = 80.0 * (K + 2) * 2.0 ** -52
        assert abs(float(Fraction(got.real) - re)) <= tol * sre and abs(float(Fraction(got.imag) - im)) <= tol * sim


@pytest.mark.parametrize("K,R", [(13, 4), (29, 3), (34, 3), (47, 2)])
def test_step_of_one_column(ctx, K, R):
    """Wide jobs with repeated rows: an imaginary step of 1e-30 in one column of
    a real matrix, proportional to it, gives 1e-30 times the permanent in the
    imaginary part.  Products of doubles: 4 (K + 2) 2^-52 of the modulus sum of
    the addends, in both parts (the step's part has one term)."""
    M = np.full(R, K // R, np.int32)
    M[: K - int(M.sum())] += 1
    N = np.ones(K, np.int32)
    g = np.random.Generator(np.random.PCG64(K))
    a = np.abs(g.standard_normal((R, K))).astype(complex)
    tol = 4.0 * (K + 2) * 2.0 ** -52

    def check_real(got, x, mult, cols, step):
        ref = sum(oracle.perm_mult(x, mult, cols)).real
        lim = tol * oracle.perm_mult_abs(x, mult, cols)
        assert abs(got.real - ref) <= lim
        assert abs(got.imag * 1e30 - ref) <= lim if step else got.imag == 0.0

    M2 = M.copy()
    M2[0] -= 1
    for col in (0, K - 1):
        b = a.copy()
        b[:, col] += 1e-30j * a[:, col]
        check_real(ctx.perm(b, M, N), a, M, N, True)
        got = ctx.laplace_minors(b, M2, N)
        for l in (0, K // 2, K - 1):
            keep = [j for j in range(K) if j != l]
            check_real(got[l], a[:, keep], M2, N[keep], l != col)


def test_sampling_a_matrix_with_small_parts(ctx):
    """Jobs of both kinds in one launch: a real interferometer with small
    phases gives the samples of the oracle."""
    g = np.random.Generator(np.random.PCG64(3))
    q, _ = np.linalg.qr(g.standard_normal((12, 12)))
    u = q * np.exp(1j * np.where(np.arange(12) % 3 == 0, 1e-9, 0.7 * np.arange(12)))[:, None]
    occ = np.array([1] * 6 + [0] * 6, np.int32)
    got = ctx.sample(u, occ, 24, seed=5)
    exp, margin, _ = oracle.cc_sample(u, occ, 24, seed=5)
    assert all(np.array_equal(got[s], exp[s]) or margin[s] < 1e-9 for s in range(24))
