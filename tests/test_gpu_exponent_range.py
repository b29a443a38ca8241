"""FP64 results at the ends of the exponent range: subnormal columns, columns
whose moduli add up to more than a double holds, one part that is not finite,
and addends far below the product of the column bounds."""
import math

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def one(n):
    return np.ones(n, np.int32)


@pytest.mark.parametrize("mode", [0, 2])
def test_subnormal_columns(ctx, mode):
    tiny = 5e-324
    assert ctx.perm(np.array([[tiny]]), [1], [1], mode=mode) == tiny
    assert ctx.perm(np.array([[complex(3 * tiny, tiny)]]), [1], [1], mode=mode) == complex(3 * tiny, tiny)
    a = np.array([[tiny, 0.0, 0.0], [0.0, 2.0, 0.0], [0.0, 0.0, 1j]])
    assert ctx.perm(a, one(3), one(3), mode=mode) == complex(0.0, 2 * tiny)
    b = np.array([[1e-310, 2.0], [1e-312, 1.0]])          # 1e-310 + 2e-312, a sum of subnormals
    assert ctx.perm(b, one(2), one(2), mode=mode) == 1e-310 + 2.0 * 1e-312
    # scaled back up by another column: exact
    c = np.array([[tiny, 0.0], [0.0, 2.0 ** 1000]])
    assert ctx.perm(c, one(2), one(2), mode=mode) == math.ldexp(tiny, 1000)
    assert np.array_equal(ctx.laplace_minors(np.array([[tiny, 3.0]]), [1], one(2), mode=mode), [3.0, tiny])


def test_finite_columns_whose_moduli_overflow(ctx):
    a = np.array([[1.7e308 + 1.7e308j]])
    assert ctx.perm(a, [1], [1]) == a[0, 0]
    big = 2.0 ** 1023
    b = np.array([[big, 0.5], [big, 0.25]])                # big (1/4 + 1/2)
    assert ctx.perm(b, one(2), one(2)) == 0.75 * big
    assert ctx.perm(b * [1, -1j], one(2), one(2)) == -0.75j * big
    c = np.array([[big, 0.5, 0.0], [big, 0.25, 0.0], [big, 0.0, 1.0]])
    assert ctx.perm(c, one(3), one(3)) == 0.75 * big
    assert np.array_equal(ctx.laplace_minors(np.array([[big, 0.5]]), [1], one(2)), [0.5, big])


def test_one_part_that_is_not_finite(ctx):
    for bad in (np.inf, -np.inf, np.nan):
        v = ctx.perm(np.array([[complex(bad, 3.0)]]), [1], [1])
        assert math.isnan(v.real) and v.imag == 3.0
        v = ctx.perm(np.array([[complex(-2.0, bad)]]), [1], [1])
        assert math.isnan(v.imag) and v.real == -2.0
        m = ctx.laplace_minors(np.array([[complex(bad, 3.0), 5.0]]), [1], one(2))
        assert m[0] == 5.0 and math.isnan(m[1].real) and m[1].imag == 3.0


def test_addends_far_below_the_column_bounds(ctx):
    """Sixteen blocks [[B, B], [B + 1, -B]], B = 2^52: every nonzero addend is
    2^-848 of the product of the column bounds, and the permanent is B^16.
    Tolerance: K^2 2^-47 of the modulus sum, which is the permanent."""
    B, nb = 2.0 ** 52, 16
    K = 2 * nb
    a = np.kron(np.eye(nb), np.array([[B, B], [B + 1, -B]]))
    got = ctx.perm(a, one(K), one(K))
    assert got.imag == 0.0 and abs(got.real / B ** nb - 1.0) <= K * K * 2.0 ** -47
    r = np.concatenate([a[:28, :28], np.ones((28, 1))], axis=1)
    m = ctx.laplace_minors(r, one(28), one(29))
    assert m[28].imag == 0.0 and abs(m[28].real / B ** 14 - 1.0) <= K * K * 2.0 ** -47
