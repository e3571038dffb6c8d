"""The sliced-storage kernel of lane groups (sell_lane.cu) against the lock-step scheduler with
the same rows per item: the same bits for every iterate, penalty step and whole solve, at the
edges of its slices (32 rows), blocks (256 rows on one CTA), groups and launches, and with
slices that stay in L2 because they do not fit in shared memory."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ub():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    import paper_2408_04875_gb300 as m
    return m


def _one_block(n):
    rb = 32
    while rb < n:
        rb *= 2
    return rb if n <= 256 else 32


def _same(a, b, keys=("inner_steps", "inner_iters", "outer_steps", "lobpcg_iters", "jacobi_iters", "floor_steps")):
    for x, y in zip(a[0], b[0]):
        assert np.array_equal(x, y)
    assert np.array_equal(np.asarray(a[1]), np.asarray(b[1]))
    assert {k: a[2][k] for k in keys} == {k: b[2][k] for k in keys}


@pytest.mark.parametrize("budget", [0, 7])
@pytest.mark.parametrize("n", [1, 2, 31, 32, 33, 64, 65, 129, 255, 256, 257, 289, 500, 1030, 2500])
def test_single_lane_matches_lock_step(ub, n, budget):
    from paper_2408_04875_gb300 import instances as I
    Q, b = I.random_ubqp(n, 0.15, 11, b_range=(-20, 20))
    mu = I.perturbation(Q, 11)
    kw = dict(max_outer=5, max_inner=40, sparse_storage=1)
    got = ub.solve_batched([Q], [b], [mu], lane_budget=budget, **kw)
    ref = ub.solve_batched([Q], [b], [mu], gemv_kernel=1, rows_per_item=_one_block(n), **kw)
    assert got[2]["gemv_kernel"] == 3 and got[2]["storage"] == 2
    _same(got, ref)


@pytest.mark.parametrize("n,density", [(40, 0.3), (250, 0.05), (300, 0.1), (1000, 0.1), (700, 0.33), (1500, 0.02)])
def test_iterates_and_penalty_step_match_lock_step(ub, n, density):
    from paper_2408_04875_gb300 import instances as I
    Q, b = I.random_ubqp(n, density, 5)
    mu = I.perturbation(Q, 5)
    Qm = Q + mu
    gam = 2 * np.abs(Qm).sum(1) + np.abs(b) + 1
    Qp, bp = Qm + np.diag(gam), b - gam
    x0, _ = ub.initial_point(Q, b, mu)
    z = x0 - x0 * x0
    p = 1.3 * np.min(np.diag(Qp) / z) * z
    rb = _one_block(n)
    for method in (ub.PABB, ub.PPA):
        kw = dict(trace_len=50, max_inner=200, method=method, sparse_storage=1)
        got = ub.inner_run(Qp, bp, p, x0, **kw)
        ref = ub.inner_run(Qp, bp, p, x0, gemv_kernel=1, rows_per_item=rb, **kw)
        assert (got["steps"], got["exit"]) == (ref["steps"], ref["exit"])
        for k in ("trace_x", "trace_alpha", "x"):
            assert np.array_equal(got[k], ref[k]), k
    assert ub.penalty_probe(Qp, bp, 0.4 * p, x0, sparse_storage=1) == \
        ub.penalty_probe(Qp, bp, 0.4 * p, x0, sparse_storage=1, gemv_kernel=1, rows_per_item=rb)


@pytest.mark.parametrize("sizes,density", [
    ((30, 33, 250, 257, 500, 511, 900), 0.1),
    ((2500, 2500, 2500, 1000, 1000, 250, 250), 0.1),          # several slices per CTA, all in shared memory
    ((1500, 1400, 1300, 1500, 1200, 1500, 1450, 1350), 0.3),  # slices that stay in L2
    (tuple([1100] * 24), 0.1),                                # two CTAs per SM
])
def test_lane_groups_match_lock_step(ub, sizes, density):
    from paper_2408_04875_gb300 import instances as I
    Qs = [I.random_ubqp(n, density, k)[0] for k, n in enumerate(sizes)]
    mus = [I.perturbation(Q, k) for k, Q in enumerate(Qs)]
    kw = dict(max_outer=3, max_inner=30, sparse_storage=1)
    got = ub.solve_batched(Qs, None, mus, lane_budget=50, gemv_kernel=3, **kw)
    _same(got, ub.solve_batched(Qs, None, mus, gemv_kernel=1, rows_per_item=32, **kw))
