"""The check of Q in pairs of 64 x 64 tiles: a single wrong entry is found wherever it lies (tile edges,
corners, both triangles, the diagonal, b), and the stored entries are counted exactly."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _instance(n, seed=1):
    rng = np.random.default_rng(seed)
    Q = np.triu(rng.integers(-100, 101, (n, n)) * (rng.random((n, n)) < 0.3)).astype(float)
    return Q + np.triu(Q, 1).T


@pytest.mark.parametrize("n", [1, 2, 63, 64, 65, 129, 200])
def test_entries_counted_and_single_faults_found(n):
    import paper_2408_04875_gb300 as ub
    Q = _instance(n)
    _, f, st = ub.solve(torch.from_numpy(Q).cuda(), None, max_outer=1, max_inner=2)
    nnz = int((Q != 0).sum() - (np.diag(Q) != 0).sum())
    assert st["alg_bytes"] == st["ticks"] * (6 * nnz + 32 * n)
    places = sorted({min(k, n - 1) for k in (0, 1, 31, 62, 63, 64, 65, 127, 128, n - 2, n - 1) if k >= 0})
    for i in places:
        for j in (places[0], places[len(places) // 2], places[-1]):
            for value in (np.nan, np.inf):
                bad = Q.copy()
                bad[i, j] = value
                with pytest.raises(Exception, match="NaN/Inf"):
                    ub.solve(torch.from_numpy(bad).cuda(), None, max_outer=1, max_inner=2)
            if i != j:
                bad = Q.copy()
                bad[i, j] += 1e-3
                with pytest.raises(Exception, match="not symmetric"):
                    ub.solve(torch.from_numpy(bad).cuda(), None, max_outer=1, max_inner=2)
        b = np.zeros(n)
        b[i] = np.nan
        with pytest.raises(Exception, match="NaN/Inf"):
            ub.solve(torch.from_numpy(Q).cuda(), torch.from_numpy(b).cuda(), max_outer=1, max_inner=2)


def test_batch_maps_every_pair_to_its_instance():
    import paper_2408_04875_gb300 as ub
    sizes = [1, 64, 65, 300, 2, 129]
    for k in range(len(sizes)):
        Qs = [_instance(n, 3 + n) for n in sizes]
        if sizes[k] > 1:
            Qs[k][sizes[k] - 1, 0] += 1e-3
        else:
            Qs[k][0, 0] = np.nan
        with pytest.raises(Exception, match=f"instance {k}: "):
            ub.solve_batched([torch.from_numpy(q).cuda() for q in Qs], None, None, max_outer=1, max_inner=2)
