"""The split-K contraction's epilogue at the cluster sizes each of its forms serves: two and four CTAs
(sixteen warps), five and eight (eight warps).  Whole solves against the oracle's stored best of the
same starts, the eigen-solver against a dense one, and the update run by the epilogue against the
separate kernel, bit for bit."""
import json
import os

import numpy as np
import pytest

import oracle as O
from paper_2408_04875_gb300 import instances as I

pytestmark = pytest.mark.gpu
GOLD = os.path.join(os.path.dirname(__file__), "golden", "oracle_objectives.json")
SIZES = [2, 4, 5, 8]


@pytest.fixture(scope="module")
def ub():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    import paper_2408_04875_gb300 as m
    return m


@pytest.mark.parametrize("S", SIZES)
def test_restart_batch_within_a_tenth_percent_of_the_oracle(ub, S):
    n, seed, R = 1000, 2, 32
    with open(GOLD) as fh:
        gold = json.load(fh)["cases"]
    best = min(gold[f"c4:n={n}:seed={seed}:start={r}"]["f"] for r in range(R))
    Q, _ = I.c4_instance(n, seed)
    mu = np.diag(np.diag(I.perturbation(Q, seed)))
    x, f, st = ub.solve(Q, None, mu=mu, starts=I.random_starts(n, R - 1, seed), restarts=R, precision=ub.BF16X2_TC,
                        tc_cluster=S)
    assert (st["tc_kernel"], st["cluster_size"]) == (1, S)
    assert f == O.objective(Q, None, x) and f - best <= 1e-3 * abs(best)


# the bar of the tensor-core eigen-solver elsewhere: 2e-3
@pytest.mark.parametrize("S", SIZES)
@pytest.mark.parametrize("n", [300, 700])
def test_lambda_min(ub, n, S):
    Q, b = I.random_ubqp(n, 0.1, 3)
    Qm = Q + np.diag(np.diag(I.perturbation(Q, 3)))
    gamma = 2 * np.abs(Qm).sum(1) + np.abs(b) + 1
    Qp, bp = Qm + np.diag(gamma), b - gamma
    x, _ = ub.initial_point(Q, b, np.diag(np.diag(I.perturbation(Q, 3))))
    z = x - x * x
    p = 0.5 * np.min(np.diag(Qp) / z) * z
    s = 1 / np.sqrt(z)
    lam = np.linalg.eigvalsh(s[:, None] * (Qp - np.diag(p)) * s)[0]
    got = ub.penalty_probe(Qp, bp, p, x, precision=ub.BF16X2_TC, tc_cluster=S)
    assert got["n_active"] == n and abs(got["lambda"] - lam) <= 2e-3 * abs(lam)


@pytest.mark.parametrize("S", SIZES)
@pytest.mark.parametrize("n,R", [(1100, 1), (1100, 43), (600, 150)])
def test_fused_update_matches_the_separate_one(ub, n, R, S):
    Q, _ = I.random_ubqp(n, 0.1, 81)
    kw = dict(restarts=R, precision=ub.BF16X2_TC, max_outer=3, max_inner=80, seed=4, tc_cluster=S)
    xa, fa, a = ub.solve(Q, None, tc_fuse=1, **kw)
    xb, fb, b = ub.solve(Q, None, tc_fuse=0, **kw)
    assert a["cluster_size"] == b["cluster_size"] == S
    assert fa == fb == O.objective(Q, None, xa) and np.array_equal(xa, xb)
    for key in ("inner_iters", "outer_steps", "lobpcg_iters", "jacobi_iters"):
        assert a[key] == b[key], key
