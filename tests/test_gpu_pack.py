"""Packing of FP32 and double-float jobs (eight lanes per column, start sums in
128-bit integers) at the edges of its lanes and rounds: 1 to 47 digit rows,
1 to 48 columns.  A power-of-two scale of a column changes nothing but the
exponent, so results must scale exactly; an entry that is not finite gives
NaN exactly where its column enters the product."""
import math

import numpy as np
import pytest

import synthetic as S

pytestmark = pytest.mark.gpu

MIXED, DF64 = 1, 2
# photons of the distinct rows of a (K - 1)-photon minors job
ROWS = [[1], [1] * 7, [1] * 8, [1] * 9, [2] * 8 + [1], [1] * 16 + [5], [3, 2] * 8 + [1], [12, 12, 12, 11], [1, 46]]


@pytest.mark.parametrize("mode", [MIXED, DF64])
@pytest.mark.parametrize("M", ROWS, ids=lambda m: "%dx%d" % (len(m), sum(m)))
def test_scaled_columns_scale_the_result_exactly(bslib, mode, M):
    ctx = bslib.Context(0)
    ctx.set_mixed_tolerance(1e300)  # MIXED: the FP32 kernels
    M = np.array(M, np.int32)
    K = int(M.sum()) + 1
    a = S.random_complex(len(M), K, 700 + K)
    ex = np.where(np.arange(K) % 2, 18, -18)
    ex[0] = -1000 if K == 2 else 5
    b = a * np.exp2(ex.astype(float))[None, :]
    N = np.ones(K, np.int32)
    m, w = ctx.laplace_minors(a, M, N, mode=mode), ctx.laplace_minors(b, M, N, mode=mode)
    for l in range(K):
        e = int(ex.sum() - ex[l])
        assert w[l] == complex(math.ldexp(m[l].real, e), math.ldexp(m[l].imag, e)), l
    ctx.close()


@pytest.mark.parametrize("mode", [MIXED, DF64])
@pytest.mark.parametrize("bad", [np.nan, np.inf])
@pytest.mark.parametrize("K", [3, 10, 18])
def test_entries_that_are_not_finite(bslib, mode, bad, K):
    ctx = bslib.Context(0)
    ctx.set_mixed_tolerance(1e300)
    M, N = np.ones(K - 1, np.int32), np.ones(K, np.int32)
    a = S.random_complex(K - 1, K, 800 + K)
    clean = ctx.laplace_minors(a, M, N, mode=mode)
    a[K - 2, 1] = bad
    got = ctx.laplace_minors(a, M, N, mode=mode)
    assert np.all(np.isnan(got[np.arange(K) != 1])) and np.isfinite(got[1])
    assert got[1] == clean[1]  # a minor never reads its own column
    ctx.close()


def test_sources_on_both_sides_of_the_direct_limit(ctx):
    """Up to 16 KB of matrices are read in place from pinned memory, more are
    uploaded; either way a batch gives the bits of single calls, also when a
    captured call repeats after the pinned block has grown."""
    one = np.ones(8, np.int32)
    items = [(S.random_complex(8, 8, 900 + i), one, one) for i in range(300)]
    ref = np.array([ctx.perm(*it) for it in items[:17]])
    for count in (1, 15, 16, 17, 300, 16, 1):
        got = ctx.perm_batch(items[:count])
        assert np.array_equal(got[:17], ref[:count])
        for _ in range(3):
            assert ctx.perm(*items[3]) == ref[3]
