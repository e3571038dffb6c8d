"""The penalized objective at the ends of its range: FP32 shares of h whose sums leave FP32's range
on the way or in the end, and infinite or undefined entries of Q, x, b and p."""
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ub():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    import paper_2408_04875_gb300 as m
    return m


# every row of x = 1 has the share Q_ii of h, exactly: h is their sum in FP64, rounded to FP32 once
# (the sum of shares of one size is exact, so the two roundings are one)
@pytest.mark.parametrize("n", [4, 32, 33, 200])
@pytest.mark.parametrize("signs", ["+-", "++--", "+", "-", "+0"])
def test_shares_whose_sums_overflow(ub, n, signs):
    import torch
    size = {"+": 1.0, "-": -1.0, "0": 0.0}
    d = torch.tensor([size[signs[i % len(signs)]] for i in range(n)], device="cuda") * 3e38
    x = torch.ones(3, n, device="cuda")
    h, g = ub.penalized_eval(torch.diag(d), None, None, x)
    want = d.double().sum().to(torch.float32)
    assert torch.equal(h, want.expand(3)), (h, want)
    assert torch.equal(g, (2 * d.double()).to(torch.float32).expand(3, n))


def _kind(t):
    import torch
    return torch.where(torch.isnan(t), 2, torch.where(torch.isinf(t), torch.sign(t).nan_to_num(), torch.zeros_like(t)))


# FP64: infinities and NaN travel as in the formula itself.  FP32 sums are compensated, and an infinite
# product leaves a NaN in its row there; the other rows and points stay finite
@pytest.mark.parametrize("dtype", ["float64", "float32"])
@pytest.mark.parametrize("value", [float("inf"), -float("inf"), float("nan")])
@pytest.mark.parametrize("where", ["Q", "x", "b", "p"])
@pytest.mark.parametrize("n", [5, 129, 300])
def test_entries_that_are_not_finite(ub, n, where, value, dtype):
    import torch
    dt = getattr(torch, dtype)
    gen = torch.Generator(device="cuda").manual_seed(n)
    r = lambda *s: (0.25 + 0.5 * torch.rand(*s, generator=gen, device="cuda", dtype=torch.float64)).to(dt)
    t = dict(Q=r(n, n), x=r(3, n), b=r(n), p=r(n))
    i = n // 2
    if where == "Q":
        t["Q"][i, 1] = value
    elif where == "x":
        t["x"][1, i] = value
    else:
        t[where][i] = value
    h, g = ub.penalized_eval(t["Q"], t["b"], t["p"], t["x"])
    Q, b, p, x = (t[k].double() for k in "Qbpx")
    v = x @ Q.T
    eh, eg = (x * v).sum(1) + x @ b + (x - x * x) @ p, 2 * v - 2 * p * x + b + p
    if dtype == "float64":
        assert torch.equal(_kind(g), _kind(eg))
        assert torch.equal(torch.isfinite(h), torch.isfinite(eh))
    else:
        assert torch.equal(torch.isfinite(g), torch.isfinite(eg))
        assert torch.equal(torch.isfinite(h), torch.isfinite(eh))
