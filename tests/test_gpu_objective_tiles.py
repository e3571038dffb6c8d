"""The penalized objective's tiled kernel at the edges of its tiles: 32 rows, chunks of 128 (FP32)
or 64 (FP64) columns, 1 to 8 points per CTA, one CTA per point group up to four row tiles; rows
off the 16-byte boundary; infinities; and the backward's 64-point chunks of 16 columns."""
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


def _inputs(n, batch, dt, torch, seed=3):
    g = torch.Generator(device="cuda").manual_seed(seed)
    r = lambda *s: torch.rand(*s, generator=g, device="cuda", dtype=torch.float64)
    Q = (200 * r(n, n) - 100).to(dt)
    return Q, (100 * r(n) - 50).to(dt), (100 * r(n)).to(dt), r(batch, n).to(dt)


# FP32: every product is within 2^-24, a chain of four within 4 of those, the compensated sum adds
# nothing: 5 * 2^-24 of the sum of |terms|, and the result's own rounding.  FP64: at most
# 8 + 4 + ceil(chunks / 4) + 4 roundings of 2^-53 in one chain.
@pytest.mark.parametrize("dtype", ["float32", "float64"])
@pytest.mark.parametrize("n", [1, 31, 32, 33, 64, 65, 127, 128, 129, 130, 255, 260, 1030])
@pytest.mark.parametrize("batch", [1, 2, 3, 8, 17, 70])
def test_objective_and_gradient(ub, n, batch, dtype):
    import torch
    dt = getattr(torch, dtype)
    Q, b, p, x = _inputs(n, batch, dt, torch)
    h, g = ub.penalized_eval(Q, b, p, x)
    Qd, bd, pd, xd = (t.double() for t in (Q, b, p, x))
    v = xd @ Qd.T
    a = v + bd + pd - pd * xd
    size = xd.abs() @ Qd.abs().T + bd.abs() + 2 * pd.abs()
    tol = 8 * 2.0 ** -24 if dtype == "float32" else (24 + n / 256) * 2.0 ** -53
    assert ((g.double() - (2 * a - bd - pd)).abs() <= 2 * tol * size).all()
    assert ((h.double() - (xd * a).sum(1)).abs() <= tol * (xd * size).sum(1)).all()
    assert torch.equal(ub.penalized_eval(Q, b, p, x, want_g=False)[0], h)
    assert torch.equal(ub.penalized_eval(Q, b, p, x, want_h=False)[1], g)
    h0, g0 = ub.penalized_eval(Q, None, None, x)
    assert ((g0.double() - 2 * v).abs() <= 2 * tol * size).all() and torch.isfinite(h0).all()


@pytest.mark.parametrize("offset", [1, 2, 3])
def test_rows_off_the_16_byte_boundary(ub, offset):
    import torch
    n, batch = 132, 5
    Q, b, p, x = _inputs(n, batch, torch.float32, torch)
    ref = ub.penalized_eval(Q, b, p, x)
    Qs = torch.zeros(n * n + 4, device="cuda")[offset:offset + n * n].view(n, n).copy_(Q)
    xs = torch.zeros(n * batch + 4, device="cuda")[offset:offset + n * batch].view(batch, n).copy_(x)
    got = ub.penalized_eval(Qs, b, p, xs)
    assert torch.equal(got[0], ref[0]) and torch.equal(got[1], ref[1])


@pytest.mark.parametrize("dtype", ["float32", "float64"])
def test_infinite_linear_term_stays_infinite(ub, dtype):
    import torch
    dt = getattr(torch, dtype)
    Q, b, p, x = _inputs(200, 3, dt, torch)
    b[7] = float("inf")
    h, g = ub.penalized_eval(Q, b, p, x)
    assert torch.isinf(h).all() and torch.isinf(g[:, 7]).all()
    assert torch.isfinite(g[:, :7]).all() and torch.isfinite(g[:, 8:]).all()


@pytest.mark.parametrize("dtype", ["float32", "float64"])
@pytest.mark.parametrize("n,batch", [(1, 1), (15, 63), (16, 64), (17, 65), (33, 129), (1000, 200)])
def test_backward(ub, n, batch, dtype):
    import torch
    dt = getattr(torch, dtype)
    _, _, _, x = _inputs(n, batch, dt, torch)
    g = torch.randn(batch, n, device="cuda", dtype=dt)
    w = torch.randn(batch, device="cuda", dtype=dt)
    gx, gp, gb = ub.penalized_vjp(x, g, w, True, True, True)
    assert torch.equal(gx, w[:, None] * g)
    xd, wd = x.double(), w.double()
    eps = (2.0 ** -24 if dtype == "float32" else 0.0) + (batch + 3) * 2.0 ** -53
    size = wd.abs() @ xd
    assert ((gb.double() - wd @ xd).abs() <= eps * size).all()
    assert ((gp.double() - wd @ (xd - xd * xd)).abs() <= eps * 2 * size).all()
    assert torch.equal(ub.penalized_vjp(x, g, w, True, False, False)[0], gx)
    assert torch.equal(ub.penalized_vjp(x, g, w, False, True, False)[1], gp)
