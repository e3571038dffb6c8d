"""The symmetric-tile kernel of lane groups (sym_lane.cu) against the lane loop, which runs the
same tiles: the same bits for whole solves at the edges of its tiles (128 rows), groups and
launches, with tiles that stay in L2, for Alg. 2 and Alg. 1."""
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


@pytest.mark.parametrize("kw", [dict(max_inner=60), dict(max_inner=60, lane_budget=7), dict(max_inner=40, method=1)])
@pytest.mark.parametrize("sizes", [
    (1, 2, 127, 128),                    # one tile each
    (129, 256, 257, 384),                # two and three row blocks
    (700, 1000, 511, 640, 90, 1300),
    (2200, 2000, 1500, 1800),            # more tiles per CTA than fit in shared memory
    tuple([300] * 30),                   # many small groups
])
def test_groups_match_the_lane_loop(ub, sizes, kw):
    from paper_2408_04875_gb300 import instances as I
    pairs = [I.random_ubqp(n, 0.7, k, b_range=(-9, 9)) if k % 2 == 0 else I.maxcut_ubqp(n, 0.6, k)
             for k, n in enumerate(sizes)]
    Qs, bs = [q for q, _ in pairs], [b for _, b in pairs]
    mus = [I.perturbation(Q, k) for k, Q in enumerate(Qs)]
    kw = dict(max_outer=3, sparse_storage=2, **kw)
    x, f, st = ub.solve_batched(Qs, bs, mus, **kw)
    y, h, ref = ub.solve_batched(Qs, bs, mus, gemv_kernel=2, **kw)
    assert (st["gemv_kernel"], ref["gemv_kernel"]) == (3, 2) and st["storage"] == ref["storage"] == 1
    assert all(np.array_equal(a, b) for a, b in zip(x, y)) and np.array_equal(f, h)
    for k in ("inner_steps", "inner_iters", "outer_steps", "lobpcg_iters", "jacobi_iters", "floor_steps"):
        assert st[k] == ref[k], k


def test_batches_beyond_the_groups_run_on_the_lane_loop(ub):
    from paper_2408_04875_gb300 import instances as I
    Qs = [I.random_ubqp(1000, 0.7, k)[0] for k in range(24)]   # 24 x 8 row blocks exceed one CTA per SM
    _, _, st = ub.solve_batched(Qs, None, max_outer=1, max_inner=5)
    assert st["gemv_kernel"] == 2 and st["storage"] == 1
