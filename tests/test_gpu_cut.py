"""How a job is cut into tasks, and the order in which their partials are
summed, depend on the job alone: memory budgets, what a context did before, the
number of chains and the server's size change no bit of a result."""
import numpy as np
import pytest

import synthetic as S

pytestmark = pytest.mark.gpu


def _minors_job(K, R, seed):
    M = np.full(R, (K - 1) // R, np.int32)
    M[: K - 1 - int(M.sum())] += 1
    return S.random_complex(R, K, seed), M, np.ones(K, np.int32)


@pytest.mark.parametrize("mode", [0, 2])
@pytest.mark.parametrize("K,R", [(12, 11), (16, 15), (20, 19), (23, 22), (26, 20), (34, 9)])
def test_minors_do_not_depend_on_the_budget(ctx, bslib, mode, K, R):
    job = _minors_job(K, R, 7 * K)
    want = ctx.laplace_minors(*job, mode=mode)
    u, occ = S.config_cc(n=14, m=28, seed=3)
    ran = 0
    for kib in (256, 512, 1024, 1536, 2048, 3072, 4096, 8192, 16384, 32768):
        c = bslib.Context(0, mem_budget_bytes=kib << 10)
        try:
            for other in (False, True):
                if other:
                    c.sample(u, occ, 50, seed=1, mode=mode)
                got = c.laplace_minors(*job, mode=mode)
                assert np.array_equal(got, want), (kib, other)
                ran += 1
        except bslib.BsError as e:
            assert "BS_ENOMEM" in str(e)        # (what the smallest budgets refuse)
        finally:
            c.close()
    assert ran >= 6


@pytest.mark.parametrize("mode", [0, 2])
def test_served_results_do_not_depend_on_the_server(bslib, mode):
    jobs = [(0, S.random_complex(k, k, k), np.ones(k, np.int32), np.ones(k, np.int32)) for k in (9, 15, 21, 24)]
    jobs += [(1,) + _minors_job(k, r, 3 * k) for k, r in ((10, 9), (17, 16), (21, 20), (24, 16), (34, 9))]
    results = []
    for budget, slots, tick in ((256 << 20, 4, 512), (8 << 20, 64, 512), (64 << 20, 64, 64), (2 << 20, 2, 2000)):
        with bslib.Server(0, mem_budget_bytes=budget, max_active=slots, tick_tasks=tick, mode=mode) as srv:
            tickets = [srv.submit(*j) for j in jobs]
            results.append([srv.wait(t)[0] for t in tickets])
    for other in results[1:]:
        for a, b in zip(results[0], other):
            assert np.array_equal(np.asarray(a), np.asarray(b))


@pytest.mark.parametrize("mode", [0, 2])
def test_samples_do_not_depend_on_their_number(ctx, bslib, mode):
    """Counts of a prefix, with a slot per task and per group of tasks."""
    u, occ = S.config_cc(n=19, m=38, seed=9)
    many = ctx.sample(u, occ, 200, seed=4, mode=mode)
    assert np.array_equal(ctx.sample(u, occ, 2, seed=4, mode=mode), many[:2])
    small = bslib.Context(0, mem_budget_bytes=1 << 20)
    try:
        assert np.array_equal(small.sample(u, occ, 12, seed=4, mode=mode), many[:12])
    finally:
        small.close()
