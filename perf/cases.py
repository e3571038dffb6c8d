"""The work a user of this package has it do, as cases that can be timed and compared.

Three paths, each through the package's public entry points:

* ``objective``: the penalized objective of problem (p) with its backward,
  ``PenalizedObjective`` under autograd: h for a batch of box points sharing Q, b, p, and
  the gradients with respect to the points, p and b.
* ``penalty``: ``penalty_probe``, one lambda_min and penalty step of Lemma 3.1.
* ``solve``: ``solve_batched``, Alg. 3 on one instance or a batch, on FP32 lanes or on the
  BF16 tensor-core lanes of a restart batch.

Instances follow the laws of ``paper_2408_04875_gb300.instances`` (integers in [-100, 100]
at a density, Max-Cut with +-1 weights, dense data), drawn here on the GPU from the seed.
The tensor-core cases name their launch form (``tc_cluster``), as a program does that
wants the same result from every process: the measured choice may differ from run to run
and with it the order of the partial sums.
"""
import math

import numpy as np
import torch

import paper_2408_04875_gb300 as ub

DEVICE = "cuda"


def listed():
    return [
        # one point of the smallest instance in FP64: a gradient check or a line search, where
        # the call's latency is everything
        dict(name="objective_one_point", path="objective", n=50, batch=1, dtype="f64"),
        # the differentiable-objective workload: a dense instance and 64 box points
        dict(name="objective_batch", path="objective", n=1000, batch=64, dtype="f32"),
        # the same in FP64 with rows that end on no 16-byte boundary and an odd batch
        dict(name="objective_f64", path="objective", n=1001, batch=37, dtype="f64"),
        # Q larger than the L2 cache: 268 MB, 128 points
        dict(name="objective_large", path="objective", n=8192, batch=128, dtype="f32"),
        # the eigen-solver of one penalty step at the middle size of the plain sweep
        dict(name="penalty_step", path="penalty", n=1000, density=0.1),
        # one small instance from host memory to the end: the call a first user makes
        dict(name="solve_small", path="solve", sizes="50", density=0.1, kind="int", host=True),
        # one instance of the plain sweep to the end, default options
        dict(name="solve_one", path="solve", sizes="500", density=0.1, kind="int"),
        # the sweep's largest size, its first 40 subproblems
        dict(name="solve_one_large", path="solve", sizes="2500", density=0.1, kind="int", max_outer=40),
        # the plain sweep's sizes as one batch of independent FP32 lanes, 50 subproblems each
        dict(name="sweep", path="solve", sizes="250x3 500x3 1000x3 2500x3", density=0.1, kind="int", max_outer=50),
        # dense instances of uneven size, integer and Max-Cut in turn, the penalty moving
        # every 20 inner iterations
        dict(name="dense_batch", path="solve", sizes="200 333 512 777 1001 1500", density=0.5, kind="mixed",
             max_outer=50, max_inner=20),
        # the batched-restart instance: 256 starts on the tensor cores
        dict(name="restarts", path="solve", sizes="2500", density=0.1, kind="int", restarts=256, precision="bf16x2",
             tc_cluster=3, max_outer=12, max_inner=50),
        # the ragged batch: instances of 100 to 3000 variables with 8 starts each
        dict(name="ragged", path="solve", sizes="100 116 134 156 181 209 243 282 327 379 440 510 591 686 796 923 1071 "
             "1242 1440 1671 1938 2248 2607 3000", density=0.0, kind="mixed", restarts=8, precision="bf16x2",
             tc_cluster=1, max_outer=4, max_inner=200),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    what = rng.choice(["objective", "objective", "objective", "penalty", "one", "one", "sweep", "dense", "restarts",
                       "ragged"])
    if what == "objective":
        n = _log_int(rng, 50, 8192)
        most = max(1, min(256, 8192 * 8192 * 100 // (n * n)))
        return dict(path="objective", n=n, batch=_log_int(rng, 1, most), dtype=rng.choice(["f32", "f64"]))
    if what == "penalty":
        return dict(path="penalty", n=_log_int(rng, 50, 1500), density=round(rng.uniform(0.05, 0.2), 3))
    if what == "one":
        n = _log_int(rng, 50, 2500)
        c = dict(path="solve", sizes=str(n), density=0.1, kind="int", host=rng.random() < 0.3)
        if n > 300 or rng.random() < 0.5:
            c["max_outer"] = rng.randint(10, 40)
        if rng.random() < 0.2:
            c.update(method="ppa", max_outer=rng.randint(5, 15), max_inner=500)
        return c
    if what == "sweep":
        sizes = " ".join(str(_log_int(rng, 200, 2500)) for _ in range(rng.randint(4, 12)))
        return dict(path="solve", sizes=sizes, density=round(rng.uniform(0.05, 0.2), 3), kind="int",
                    max_outer=rng.randint(10, 40))
    if what == "dense":
        sizes = " ".join(str(_log_int(rng, 150, 1500)) for _ in range(rng.randint(4, 8)))
        return dict(path="solve", sizes=sizes, density=round(rng.uniform(0.4, 1.0), 3), kind="mixed",
                    max_outer=rng.randint(10, 40), max_inner=rng.choice([20, 50]))
    if what == "restarts":
        return dict(path="solve", sizes=str(_log_int(rng, 500, 2500)), density=0.1, kind="int",
                    restarts=rng.choice([32, 64, 100, 128, 256]), precision=rng.choice(["bf16x2", "bf16x2", "bf16"]),
                    tc_cluster=rng.choice([1, 2, 3]), max_outer=rng.randint(4, 12), max_inner=50)
    sizes = " ".join(str(_log_int(rng, 100, 2500)) for _ in range(rng.randint(8, 20)))
    return dict(path="solve", sizes=sizes, density=0.0, kind="mixed", restarts=rng.choice([4, 8, 16]),
                precision="bf16x2", tc_cluster=1, max_outer=rng.randint(2, 4), max_inner=200)


# ---- inputs --------------------------------------------------------------------------------

def _sizes(case):
    """The instance sizes: "250x3 500" stands for 250 250 250 500."""
    out = []
    for part in case["sizes"].split():
        n, _, k = part.partition("x")
        out += [int(n)] * int(k or 1)
    return out


def _kind(case, i):
    return ("cut" if i % 2 else "int") if case["kind"] == "mixed" else case["kind"]


def _density(case, i):
    """The case's density; 0 stands for the ragged batch's spread over [0.05, 1]."""
    return case["density"] or 0.05 + 0.95 * ((7 * i) % 24) / 24.0


def _instance(n, density, kind, g):
    """Q symmetric FP64: kept entries uniform integers in [-100, 100] with b = 0, or +-1 edge
    weights W with b = -W e (Max-Cut, f = -cut)."""
    keep = torch.rand(n, n, generator=g, device=DEVICE) < density
    if kind == "int":
        val = torch.randint(-100, 101, (n, n), generator=g, device=DEVICE)
    else:
        val = 2 * torch.randint(0, 2, (n, n), generator=g, device=DEVICE) - 1
    upper = torch.triu((keep * val).double(), 0 if kind == "int" else 1)
    Q = (upper + torch.triu(upper, 1).T).contiguous()
    b = torch.zeros(n, dtype=torch.float64, device=DEVICE) if kind == "int" else -Q.sum(1)
    return Q, b


def _perturbed(Q, g):
    """Q plus a symmetric N(0, 1e-3 max |Q|) perturbation of its stored entries."""
    noise = torch.randn(Q.shape, generator=g, device=DEVICE, dtype=torch.float64) * (1e-3 * Q.abs().max())
    keep = (Q != 0) | torch.eye(Q.shape[0], dtype=torch.bool, device=DEVICE)
    noise = torch.triu(noise * keep)
    return Q + noise + torch.triu(noise, 1).T


def _objective_inputs(case, seed):
    """Dense data as the solver's own products see it (integers plus the perturbation), box
    points, a penalty in [0, 100] and the gradient of a loss over h."""
    g = torch.Generator(device=DEVICE).manual_seed(seed)
    n, dt = case["n"], torch.float64 if case["dtype"] == "f64" else torch.float32
    Q, _ = _instance(n, 1.0, "int", g)
    Q = _perturbed(Q, g).to(dt).contiguous()
    b = torch.randint(-50, 51, (n,), generator=g, device=DEVICE).to(dt)
    p = 100 * torch.rand(n, generator=g, device=DEVICE, dtype=dt)
    x = torch.rand(case["batch"], n, generator=g, device=DEVICE, dtype=dt)
    w = 0.5 + torch.rand(case["batch"], generator=g, device=DEVICE, dtype=dt)
    return Q, b, p, x, w


def _penalty_inputs(case, seed):
    """Q', b' of Sec. 3.5, x^0 of Eq. (gamma) by Jacobi sweeps and a first penalty p = c z."""
    g = torch.Generator(device=DEVICE).manual_seed(seed)
    Q, b = _instance(case["n"], case["density"], "int", g)
    Q = _perturbed(Q, g)
    gamma = 2 * Q.abs().sum(1) + b.abs() + 1
    Qp = (Q + torch.diag(gamma)).contiguous()
    bp = b - gamma
    d = Qp.diagonal()
    x = torch.full_like(bp, 0.5)
    for _ in range(40):
        x = x - (2 * (Qp * x).sum(1) + bp) / (2 * d)
    z = x - x * x
    p = 0.5 * (d / z).min() * z
    return Qp, bp, p, x


def prepare(case, seed):
    if case["path"] == "objective":
        Q, b, p, x, w = _objective_inputs(case, seed)
        return dict(path="objective", Q=Q, b=b.requires_grad_(), p=p.requires_grad_(), x=x.requires_grad_(), w=w)
    if case["path"] == "penalty":
        Qp, bp, p, x = _penalty_inputs(case, seed)
        return dict(path="penalty", args=(Qp, bp, p, x))
    g = torch.Generator(device=DEVICE).manual_seed(seed)
    pairs = [_instance(n, _density(case, i), _kind(case, i), g) for i, n in enumerate(_sizes(case))]
    if case.get("host"):
        pairs = [(Q.cpu().numpy(), b.cpu().numpy()) for Q, b in pairs]
    kw = {k: case[k] for k in ("max_outer", "max_inner", "restarts", "tc_cluster") if k in case}
    if "precision" in case:
        kw["precision"] = {"bf16x2": ub.BF16X2_TC, "bf16": ub.BF16_TC}[case["precision"]]
    if case.get("method") == "ppa":
        kw["method"] = ub.PPA
    kw["seed"] = seed   # keys the library's own draws: the perturbation and the extra starts
    return dict(path="solve", Qs=[Q for Q, _ in pairs], bs=[b for _, b in pairs], kw=kw)


# ---- one pass ------------------------------------------------------------------------------

def run(state):
    if state["path"] == "objective":
        x, Q, b, p = state["x"], state["Q"], state["b"], state["p"]
        h = ub.PenalizedObjective.apply(x, Q, b, p)
        gx, gb, gp = torch.autograd.grad(h, (x, b, p), state["w"])
        return dict(h=h.detach(), gx=gx, gb=gb, gp=gp)
    if state["path"] == "penalty":
        r = ub.penalty_probe(*state["args"])
        return dict(lam=r["lambda"], alpha=r["alpha"], n_active=r["n_active"], iters=r["iters"])
    xs, obj, _ = ub.solve_batched(state["Qs"], state["bs"], **state["kw"])
    return dict(x=xs, objective=obj)


def work(case):
    if case["path"] == "objective":
        n, B, es = case["n"], case["batch"], 8 if case["dtype"] == "f64" else 4
        # Q, x, b, p and w in; h, gx, gb and gp out
        return dict(bytes=es * (n * n + 2 * B * n + 4 * n + 2 * B), flops=2.0 * B * n * n + 10.0 * B * n)
    if case["path"] == "penalty":
        n = case["n"]
        # about 30 eigen-solver products over the stored entries
        return dict(bytes=8.0 * (n * n + 3 * n), flops=30 * 2.0 * case["density"] * n * n)
    nbytes, flops = 0.0, 0.0
    for i, n in enumerate(_sizes(case)):
        nbytes += 8.0 * n * n + 9.0 * n
        if case.get("max_outer", 1000) >= 1000:
            steps = 120.0 * n   # a whole solve at the default caps takes about this many products
        else:
            # per subproblem: its inner iterations, about 40 products of the eigen-solver, one evaluation
            steps = case["max_outer"] * (min(case.get("max_inner", 10000), 20 + 200 * case["max_outer"] / 40) + 41)
        flops += 2.0 * _density(case, i) * n * n * steps * case.get("restarts", 1)
    return dict(bytes=nbytes, flops=flops)


def exact(case, seed):
    """What ``run`` returns, from 64-bit arithmetic.  A solve's point and objective depend on
    the whole trajectory, so they have no such value here."""
    if case["path"] == "objective":
        Q, b, p, x, w = (t.double() for t in _objective_inputs(case, seed))
        qx = x @ Q
        h = (x * qx).sum(1) + x @ b + (x - x * x) @ p
        gx = w[:, None] * (2 * qx - 2 * p * x + b + p)
        return dict(h=h, gx=gx, gb=w @ x, gp=w @ (x - x * x))
    if case["path"] == "penalty":
        Qp, _, p, x = (t.cpu().numpy() for t in _penalty_inputs(case, seed))
        z = x - x * x
        act = z > 1e-12
        s = 1 / np.sqrt(z[act])
        lam = float(np.linalg.eigvalsh(s[:, None] * (Qp - np.diag(p))[np.ix_(act, act)] * s)[0])
        return dict(lam=lam, alpha=0.9 * lam, n_active=int(act.sum()), iters=None)
    return None
