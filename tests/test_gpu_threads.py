"""Two host threads in the library at once, one with a large problem in many launches and one with
small ones: the results of each alone, for every kind of launch that asks for dynamic shared
memory by the size of its problem."""
import threading

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


# large sizes, small sizes, density, options
CASES = {
    "sliced": ((2500,), (300,), 0.1, dict(sparse_storage=1)),
    "sliced batch": ((1500, 1400, 1300), (300, 250, 200), 0.1, dict(sparse_storage=1)),
    "tiles": ((1000, 900, 1000, 800), (200, 150, 200, 100), 0.7, dict(sparse_storage=2)),
    "dense rows": ((2000,), (300,), 0.7, dict(sparse_storage=2)),
    "lock-step": ((6000,), (300,), 0.02, dict(gemv_kernel=1)),
    "split-K": ((600,), (130,), 0.3, dict(precision=1, restarts=64, tc_cluster=2)),
    "many tiles": ((500,) * 40, (130,) * 160, 0.3, dict(precision=1, restarts=4, tc_cluster=1)),
}


@pytest.mark.parametrize("name", CASES)
def test_two_threads(ub, name):
    from paper_2408_04875_gb300 import instances as I
    large, small, density, kw = CASES[name]
    kw = dict(kw, max_outer=3, max_inner=60, lane_budget=5, max_ticks_per_sync=8, seed=3)
    data = [[I.random_ubqp(n, density, k)[0] for k, n in enumerate(sizes)] for sizes in (large, small)]
    alone = [ub.solve_batched(Qs, None, **kw) for Qs in data]
    results, errors = [[], []], []
    done = threading.Event()

    def work(side, times):
        try:
            for _ in range(times):
                results[side].append(ub.solve_batched(data[side], None, **kw))
                if side == 1 and done.is_set():
                    break
        except Exception as e:   # noqa: BLE001
            errors.append((side, str(e)))
        finally:
            if side == 0:
                done.set()

    threads = [threading.Thread(target=work, args=(0, 4)), threading.Thread(target=work, args=(1, 400))]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors
    for side in (0, 1):
        for xs, f, _ in results[side]:
            assert np.array_equal(f, alone[side][1])
            assert all(np.array_equal(x, y) for x, y in zip(xs, alone[side][0]))
