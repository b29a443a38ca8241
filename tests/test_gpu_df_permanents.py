"""Double-float permanents run in the FP64 kernels' fixed point: the bucket
edges of the two layouts (rows padded to four columns there, to eight in the
double-float minors), and the same bits from a call, a batch that mixes widths
and an FP64-mode call.

Tolerance: the fixed-point products lose at most K 2^-50 of the modulus sum of
the addends (oracle.perm_mult_abs), far inside 1e-12 of it."""
import numpy as np
import pytest

import oracle
import synthetic as S

pytestmark = pytest.mark.gpu

DF64 = 2
REL = 1e-12


def _job(K):
    """Distinct rows up to 12 columns; above, a few rows of high multiplicity."""
    R = K if K <= 12 else 5
    M = np.full(R, K // R, np.int32)
    M[: K - int(M.sum())] += 1
    return S.random_complex(R, K, 500 + K), M, np.ones(K, np.int32)


WIDTHS = [1, 2, 4, 5, 8, 9, 12, 13, 16, 17, 24, 25, 32, 33, 40, 41, 48]


@pytest.mark.parametrize("K", WIDTHS)
def test_permanent_at_bucket_edges(ctx, K):
    a, M, N = _job(K)
    got = ctx.perm(a, M, N, mode=DF64)
    assert abs(got - sum(oracle.perm_mult(a, M, N))) <= REL * oracle.perm_mult_abs(a, M, N)


def test_batch_and_fp64_mode_give_the_call_bits(ctx):
    jobs = [_job(K) for K in WIDTHS]
    one = np.array([ctx.perm(*j, mode=DF64) for j in jobs])
    assert np.array_equal(one, ctx.perm_batch(jobs, mode=DF64))
    assert np.array_equal(one, ctx.perm_batch(jobs[::-1], mode=DF64)[::-1])
    assert np.array_equal(one, np.array([ctx.perm(*j) for j in jobs]))
