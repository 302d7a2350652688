"""Block solves where rows of very different lengths meet few or many columns:
rows of one thread, of a warp (17 to 1024 arcs, up to 16 quads of columns) and of a
block."""
import numpy as np
import pytest
import torch
from scipy import sparse

import paper_2510_20604_gb300 as rwc
import synth

pytestmark = pytest.mark.gpu


def _hubs(weighted):
    """A ring with chords and hubs whose degrees lie around the rows' bounds."""
    n, rng = 5000, np.random.default_rng(6)
    i = np.arange(n)
    u, v = [i, i], [(i + 1) % n, (i + 37) % n]
    for hub, deg in enumerate((12, 13, 14, 28, 60, 124, 125, 126, 1019, 1020, 1021, 3000)):
        u.append(np.full(deg, hub * 400))
        v.append((hub * 400 + 100 + rng.permutation(n - 200)[:deg]) % n)
    u, v = np.concatenate(u), np.concatenate(v)
    return synth.from_edges(n, u, v, rng.lognormal(0.0, 0.5, len(u)) if weighted else None)


@pytest.mark.parametrize("weighted", [False, True])
@pytest.mark.parametrize("k", [2, 4, 5, 11, 20, 33, 64, 65, 129, 300])
def test_solve_with_hub_rows(weighted, k):
    g = _hubs(weighted)
    w = np.ones(g.nnz) if g.w is None else g.w.astype(np.float64)
    b = np.random.default_rng(k).standard_normal((k, g.n))
    b -= b.mean(1, keepdims=True)
    x = torch.empty(k, g.n, dtype=torch.float64, device="cuda")
    G = rwc.Graph.from_synth(g)
    rwc.rwc_solve(G.handle, k, torch.as_tensor(b, device="cuda"), x, 1e-10)
    again = torch.empty_like(x)
    rwc.rwc_solve(G.handle, k, torch.as_tensor(b, device="cuda"), again, 1e-10)
    assert torch.equal(x, again)
    x = x.cpu().numpy()
    A = sparse.csr_matrix((w, g.col, g.row_ptr), shape=(g.n, g.n))
    r = b - (np.asarray(A.sum(1)).ravel() * x - (A @ x.T).T)
    # the solver's criterion, and rounding in the evaluation of r
    assert (np.linalg.norm(r, axis=1) <= 2e-10 * np.linalg.norm(b, axis=1)).all()


@pytest.mark.parametrize("n", [1024, 1025, 1026, 1300])
@pytest.mark.parametrize("k", [1, 3, 70])
def test_solve_where_every_row_is_heavy(n, k):
    # L = n I - J: x = b / n for mean-free b
    b = np.random.default_rng(n).standard_normal((k, n))
    b -= b.mean(1, keepdims=True)
    x = torch.empty(k, n, dtype=torch.float64, device="cuda")
    rwc.rwc_solve(rwc.Graph.from_synth(synth.complete(n)).handle, k, torch.as_tensor(b, device="cuda"), x, 1e-10)
    err = np.linalg.norm(n * x.cpu().numpy() - b, axis=1)
    assert (err <= 2e-10 * np.linalg.norm(b, axis=1)).all()
