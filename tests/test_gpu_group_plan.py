"""Which kernel runs the lane groups, and with which plan: ubqp_profile_groups after calls whose
results other tests compare (the kernels give the same bits, so a call that silently ran another one
would pass those)."""
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ub():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    import paper_2408_04875_gb300 as m
    return m


def _plan(ub, sizes, density, **kw):
    from paper_2408_04875_gb300 import instances as I
    Qs = [I.random_ubqp(n, density, k)[0] for k, n in enumerate(sizes)]
    _, _, st = ub.solve_batched(Qs, None, max_outer=2, max_inner=20, seed=1, **kw)
    assert st["gemv_kernel"] == 3
    return ub.lane_groups(), [int((Q != 0).sum(1).max()) for Q in Qs]


def test_one_sparse_lane(ub):
    for n, ctas in ((40, 1), (256, 1), (257, 9), (2500, 79)):
        g, width = _plan(ub, (n,), 0.1)
        assert (g["kernel"], g["ctas_per_sm"], g["blocks_per_cta"], g["ctas"]) == ("sell_lane_kernel", 1, 1, ctas)
        assert g["smem_bytes"] > 0


def test_slices_that_fit_and_slices_that_do_not(ub):
    # 192 bytes (32 entries of six) per column of a slice's widest row
    g, width = _plan(ub, (2500, 2500, 2500, 1000, 1000, 250, 250), 0.1)
    assert g["kernel"] == "sell_lane_kernel" and g["blocks_per_cta"] > 1
    assert g["smem_bytes"] >= 192 * (max(width) - 1)
    g, width = _plan(ub, (1500, 1400, 1300, 1500, 1200, 1500, 1450, 1350), 0.3)
    assert g["kernel"] == "sell_lane_kernel"
    assert g["smem_bytes"] < g["blocks_per_cta"] * 192 * (max(width) - 1)


def test_two_ctas_per_sm(ub):
    g, width = _plan(ub, (1100,) * 24, 0.15)
    assert (g["kernel"], g["ctas_per_sm"], g["blocks_per_cta"]) == ("sell_lane_kernel", 2, 3)
    assert g["smem_bytes"] < 3 * 192 * (max(width) - 1)   # not all of a CTA's slices
    g, _ = _plan(ub, (600,) * 20, 0.1)
    assert (g["kernel"], g["ctas_per_sm"]) == ("sell_lane_kernel", 1)


def test_dense_lanes(ub):
    g, _ = _plan(ub, (1000, 900, 1000, 800), 0.7)
    assert g["kernel"] == "sym_lane_kernel" and g["smem_bytes"] == g["blocks_per_cta"] * 65536
    g, _ = _plan(ub, (1000,), 0.7)
    assert g["kernel"] == "solo_lane_kernel"
    g, _ = _plan(ub, (1000,), 0.1, rows_per_item=64)
    assert g["kernel"] == "solo_lane_kernel"


# two CTAs on an SM hold two vectors of up to 12,416 entries: three lanes of 11,600 and 12,320 need more than five
# slices per CTA with one CTA per SM, and run on the sliced kernel with two, with the bits of the lock-step
# scheduler; a lane of one block (20 variables) rides along
@pytest.mark.parametrize("n,method", [(11600, 0), (12320, 0), (12320, 1)])
def test_long_vectors_on_two_ctas_per_sm(ub, n, method):
    import torch
    Qs = []
    for k in range(3):
        g = torch.Generator(device="cuda").manual_seed(k)
        v = torch.randint(-100, 101, (n, n), generator=g, device="cuda").double()
        v *= torch.rand(n, n, generator=g, device="cuda") < 0.002
        u = torch.triu(v)
        Qs.append((u + torch.triu(v, 1).T).contiguous())
        del v, u
    Qs.append(Qs[0][:20, :20] + 7 * torch.eye(20, device="cuda", dtype=torch.float64))
    Qs[-1][3, 11] = Qs[-1][11, 3] = -40
    kw = dict(max_outer=2, max_inner=30, seed=1, method=method)
    xs, f, st = ub.solve_batched(Qs, None, lane_budget=40, **kw)
    g = ub.lane_groups()
    assert st["gemv_kernel"] == 3
    assert (g["kernel"], g["ctas_per_sm"], g["blocks_per_cta"]) == ("sell_lane_kernel", 2, 4)
    ys, h, ref = ub.solve_batched(Qs, None, gemv_kernel=1, rows_per_item=32, **kw)
    assert (f == h).all() and all((x == y).all() for x, y in zip(xs, ys))
    for k in ("inner_steps", "inner_iters", "outer_steps", "lobpcg_iters", "jacobi_iters", "floor_steps"):
        assert st[k] == ref[k], k
