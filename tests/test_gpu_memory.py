"""Device memory after a call: what the library keeps between calls is bounded, and everything beyond
that is back with the device when the call returns (no synchronization by the caller)."""
import ctypes

import pytest

pytestmark = pytest.mark.gpu

KEPT = 128 << 20


@pytest.fixture(scope="module")
def ub():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    import paper_2408_04875_gb300 as m
    return m


def _free(torch):
    return torch.cuda.mem_get_info()[0]


@pytest.mark.parametrize("kw", [dict(), dict(sparse_storage=2), dict(precision=1, restarts=8, tc_cluster=1)])
def test_large_workspace_is_given_back(ub, kw):
    import torch
    n = 8000   # about 0.8 GB of FP32 and evaluation rows, or 0.13 GB of BF16 beside 1 GB of host Q
    g = torch.Generator(device="cuda").manual_seed(1)
    v = torch.randint(-100, 101, (n, n), generator=g, device="cuda").double() * \
        (torch.rand(n, n, generator=g, device="cuda") < 0.01)
    Q = torch.triu(v) + torch.triu(v, 1).T
    del v
    if "precision" in kw:
        Q = Q.cpu().numpy()   # staged in the workspace
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    kw = dict(kw, max_outer=1, max_inner=5, seed=1)
    ub.solve(Q[:300, :300], None, **kw)   # kernels loaded
    torch.cuda.synchronize()
    before = _free(torch)
    for _ in range(2):
        ub.solve(Q, None, **kw)
        after = _free(torch)
        assert before - after <= KEPT + (64 << 20), (before - after) >> 20


def test_objective_scratch_is_given_back(ub):
    import torch
    n, batch = 2048, 400000   # 64 row tiles: 205 MB of shares of h
    x = torch.rand(batch, n, device="cuda")
    Q = torch.rand(n, n, device="cuda")
    b = torch.rand(n, device="cuda")
    ub.penalized_eval(Q, b, None, x[:8])
    out = torch.empty(batch, device="cuda")
    torch.cuda.synchronize()
    before = _free(torch)
    vp = ctypes.c_void_p
    rc = ub.lib().ubqp_penalized_eval(vp(Q.data_ptr()), vp(b.data_ptr()), None, vp(x.data_ptr()), n, batch, 0,
                                      vp(out.data_ptr()), None, vp(torch.cuda.current_stream().cuda_stream))
    assert rc == 0 and before - _free(torch) <= KEPT + (64 << 20)
    assert torch.isfinite(out).all()
