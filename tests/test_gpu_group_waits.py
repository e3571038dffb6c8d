"""Bounded waits of the lane-group kernels: a limit of one microsecond runs out, the call returns
UBQP_ETIMEOUT with the kernel's name and the limit, and the same context then solves the same batch as
if nothing had happened.  (Each wait gives up by itself; nothing is in flight that a CTA waits for.)"""
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


# sizes, density, options: sliced rows (one lane, several groups, two CTAs per SM), symmetric tiles, and
# the group-barrier kernel on dense rows and on sliced rows of 64
CASES = {
    "sell_lane_kernel": [((2500,), 0.1, {}), ((700, 900, 500), 0.1, {}), ((1100,) * 24, 0.1, {})],
    "sym_lane_kernel": [((1000, 900, 1000, 800), 0.7, {}), ((300,) * 30, 0.7, {})],
    "solo_lane_kernel": [((2000,), 0.7, {}), ((2500,), 0.1, dict(rows_per_item=64))],
}


@pytest.mark.parametrize("kernel,case", [(k, c) for k in CASES for c in range(len(CASES[k]))])
def test_wait_limit_runs_out(ub, kernel, case):
    from paper_2408_04875_gb300 import instances as I
    sizes, density, kw = CASES[kernel][case]
    Qs = [I.random_ubqp(n, density, k)[0] for k, n in enumerate(sizes)]
    kw = dict(kw, max_outer=3, max_inner=40, seed=5)
    xs, f, _ = ub.solve_batched(Qs, None, **kw)
    with pytest.raises(ub.UBQPError) as e:
        ub.solve_batched(Qs, None, wait_limit_us=1, **kw)
    assert e.value.status == -6 and kernel in str(e.value) and "limit 1 us" in str(e.value)
    ys, h, _ = ub.solve_batched(Qs, None, **kw)
    assert ub.lane_groups()["kernel"] == kernel
    assert np.array_equal(f, h) and all(np.array_equal(x, y) for x, y in zip(xs, ys))
