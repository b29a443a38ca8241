"""Chunk lengths of sampler calls with few chains and of served requests: a
chain's counts do not depend on how many tasks its jobs are cut into (exact
column sums; the sums differ only in their last rounding)."""
import numpy as np
import pytest

import synthetic as S

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("mode", [0, 2])
@pytest.mark.parametrize("n", [3, 11, 18])
def test_few_chains_equal_many(ctx, bslib, mode, n):
    u, occ = S.config_cc(n=n, m=2 * n, seed=40 + n)
    many = ctx.sample(u, occ, 160, seed=71, mode=mode)          # 64 tasks per job
    for few in (1, 3, 20):                                      # up to 1024
        assert np.array_equal(ctx.sample(u, occ, few, seed=71, mode=mode), many[:few]), few
    small = bslib.Context(0, mem_budget_bytes=4 << 20)          # falls back to 64
    try:
        assert np.array_equal(small.sample(u, occ, 3, seed=71, mode=mode), many[:3])
    finally:
        small.close()


@pytest.mark.parametrize("mode", [0, 2])
@pytest.mark.parametrize("budget,slots", [(64 << 20, 4), (1 << 20, 64)])
def test_served_chains_at_both_targets(ctx, bslib, mode, budget, slots):
    u, occ = S.config_cc(n=16, m=32, seed=55)
    ref = ctx.sample(u, occ, 4, seed=73, mode=mode)
    a = u[:15, :15]
    ones = np.ones(15, np.int32)
    with bslib.Server(0, mem_budget_bytes=budget, max_active=slots, tick_tasks=512, mode=mode) as srv:
        tickets = [srv.submit_sample(u, occ, 73, s) for s in range(4)]
        p = srv.submit(0, a, ones, ones)
        assert np.array_equal(np.array([srv.wait_sample(t)[0] for t in tickets]), ref)
        v = srv.wait(p)[0][0]
    d = ctx.perm(a, ones, ones, mode=mode)
    assert abs(v - d) <= 1e-11 * np.prod(np.sqrt((np.abs(a) ** 2).sum(axis=0)))
