"""FP64 results on matrices whose column sums cancel: every addend keeps its own
relative accuracy, so results stay within a few K^2 2^-49 of the modulus sum of
the addends however small the products are against the column bounds.

Inputs: diagonal blocks [[B, B], [B + 1, -B]], exactly representable.  In each
block one column sum is zero or 1 where the other is 2 B + 1 or 2 B, so every
nonzero addend has a sum 2^-log2(2 B) below its bound per block, and all of
them have the same value: the modulus sum is the permanent itself.

Tolerance: two lanes form at most K / 2 + 2 pairs of columns; each may err by
two units (2^1.5 with both components) of 2^(12 + log2 K - 61) before its addend
is formed again in double: (K / 2 + 2) 2^1.5 K 2^-49, 3 K^2 2^-49 for K >= 4,
and as much again for addends that are compared with the largest one."""
from fractions import Fraction
from functools import lru_cache

import numpy as np
import pytest

import oracle
import synthetic as S

pytestmark = pytest.mark.gpu


def perm_exact(a):
    """Permanent of a real matrix of doubles in rational arithmetic."""
    rows = [[Fraction(float(x)) for x in r] for r in np.asarray(a).real]

    @lru_cache(maxsize=None)
    def rec(i, used):
        if i == len(rows):
            return Fraction(1)
        return sum((x * rec(i + 1, used | 1 << j) for j, x in enumerate(rows[i]) if x and not used >> j & 1), Fraction(0))

    return rec(0, 0)


def blocks(nb, B):
    return np.kron(np.eye(nb), np.array([[B, B], [B + 1, -B]]))


def tol(K):
    return 6.0 * K * K * 2.0 ** -49


def orders(K, seed):
    """Column orders: as they are, the blocks' columns in different pairs, and
    at random."""
    g = np.random.Generator(np.random.PCG64(seed))
    return [np.arange(K), np.argsort(np.arange(K) % 2, kind="stable"), g.permutation(K)]


@pytest.mark.parametrize("nb,B", [(1, 3.0 ** 25), (2, 789.0), (2, 3.0 ** 25), (4, 808037.0), (4, 3.0 ** 25), (5, 2.0 ** 50),
                                  (7, 3.0 ** 20), (9, 3.0 ** 25), (10, 3.0 ** 12)])
def test_permanents_of_cancelling_blocks(ctx, nb, B):
    K = 2 * nb
    a, ones = blocks(nb, B), np.ones(2 * nb, np.int32)
    exact = perm_exact(a)
    for order in orders(K, nb):
        for mode in (0, 2):
            got = ctx.perm(a[:, order], ones, ones, mode=mode)
            assert got.imag == 0.0
            assert abs(float((Fraction(got.real) - exact) / exact)) <= tol(K), (order, mode)
    # rotated by a phase that is not a multiple of 90 degrees: 3 + 4i per column
    got = ctx.perm(a * (3 + 4j), ones, ones)
    want = complex(float(exact)) * (3 + 4j) ** K
    assert abs(got - want) <= (tol(K) + K * 2.0 ** -50) * abs(want)


@pytest.mark.parametrize("f", ["ryser", "nw"])
def test_formulas_of_cancelling_blocks(ctx, f):
    a = blocks(4, 3.0 ** 20)
    exact = float(perm_exact(a))
    got = ctx.perm_formula(a[:, orders(8, 3)[1]], f)
    assert abs(got - exact) <= tol(8) * oracle.formula_abs(f, a)


@pytest.mark.parametrize("K", [8, 15, 24])
def test_permanents_of_noise_and_zeros(ctx, K):
    """Sums that vanish exactly (signs) or up to the rounding of the entries
    (roots of unity) beside ordinary ones."""
    R = min(K, 10)
    M = np.full(R, K // R, np.int32)
    M[: K - int(M.sum())] += 1
    N = np.ones(K, np.int32)
    g = np.random.Generator(np.random.PCG64(K))
    signs = g.choice([-1.0, 1.0], size=(R, K))
    roots = np.exp(2j * np.pi * np.outer(np.arange(R), np.arange(K)) / 12)
    for a in (signs, roots, signs * (1 + 2.0 ** -40 * g.standard_normal((R, K)))):
        got = ctx.perm(a, M, N)
        assert abs(got - sum(oracle.perm_mult(a, M, N))) <= tol(K) * oracle.perm_mult_abs(a, M, N)


# Minors: products of normalised sums err by 2^-55 (K + 1 of them enter an
# addend), an addend's place in its run's integer sum by 3 units of 2^-54 of the
# run's largest addend of that column (8 in a run), the sums of runs in double
# by 2^-53 in at most 256 additions before they are folded.
TOL_MINORS = (48 + 1) * 2.0 ** -55 + 8 * 3 * 2.0 ** -54 + 256 * 2.0 ** -53 + 2.0 ** -50


@pytest.mark.parametrize("nb,B,seed", [(1, 3.0 ** 25, 1), (2, 789.0, 2), (2, 3.0 ** 20, 3), (3, 3.0 ** 25, 4), (4, 789.0, 5),
                                       (4, 3.0 ** 25, 6), (5, 3.0 ** 31, 7), (6, 808037.0, 8)])
def test_minors_of_cancelling_blocks(ctx, nb, B, seed):
    K = 2 * nb + 1
    g = np.random.Generator(np.random.PCG64(seed))
    a = np.concatenate([blocks(nb, B), g.standard_normal((K - 1, 1))], axis=1)
    ones, cols = np.ones(K - 1, np.int32), np.ones(K, np.int32)
    exact = [float(perm_exact(np.delete(a, l, 1))) for l in range(K)]
    for order in orders(K, seed):
        got = ctx.laplace_minors(a[:, order], ones, cols)
        for i, l in enumerate(order):
            bound = oracle.perm_mult_abs(np.delete(a, l, 1), ones, ones)
            assert got[i].imag == 0.0 and abs(got[i].real - exact[l]) <= TOL_MINORS * bound, (order, i)


@pytest.mark.parametrize("K", [9, 14, 27, 34])
def test_minors_of_noise_and_zeros(ctx, K):
    R = min(K - 1, 6)
    M = np.full(R, (K - 1) // R, np.int32)
    M[: K - 1 - int(M.sum())] += 1
    N = np.ones(K, np.int32)
    g = np.random.Generator(np.random.PCG64(K))
    signs = g.choice([-1.0, 1.0], size=(R, K))
    roots = np.exp(2j * np.pi * np.outer(np.arange(R), np.arange(K)) / 12)
    for a in (signs, roots, signs * (1 + 2.0 ** -40 * g.standard_normal((R, K)))):
        got = ctx.laplace_minors(a, M, N)
        for l in (0, K // 2, K - 1):
            keep = [j for j in range(K) if j != l]
            ref = sum(oracle.perm_mult(a[:, keep], M, N[keep]))
            assert abs(got[l] - ref) <= TOL_MINORS * oracle.perm_mult_abs(a[:, keep], M, N[keep]), l
