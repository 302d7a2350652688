"""Pivot-sized solves on graphs of bounded degree with more rows than the
register kernel holds (152 x 1024 x 7), where the rows are read inline."""
import numpy as np
import pytest
import torch
from scipy import sparse

import paper_2510_20604_gb300 as rwc
import synth

pytestmark = pytest.mark.gpu


def _king(rows, cols):
    i = np.arange(rows * cols).reshape(rows, cols)
    pairs = [(i[:, :-1], i[:, 1:]), (i[:-1], i[1:]), (i[:-1, :-1], i[1:, 1:]), (i[:-1, 1:], i[1:, :-1])]
    return synth.from_edges(rows * cols, np.concatenate([a.ravel() for a, _ in pairs]),
                            np.concatenate([b.ravel() for _, b in pairs]))


# the last size held in registers, the first beyond it, degree 8, and above 8
# million rows, where the direction is an array of its own
@pytest.mark.parametrize("make,tol", [(lambda: synth.grid2d(1024, 1064), 1e-6), (lambda: synth.grid2d(1025, 1064), 1e-6),
                                      (lambda: _king(1044, 1045), 1e-6), (lambda: synth.grid2d(2833, 2825), 1e-3)])
def test_solve_beyond_the_register_kernel(make, tol):
    g = make()
    # a sum of a few waves: no long-range part that takes thousands of iterations
    b = np.cos(np.arange(g.n) * 0.7) + np.random.default_rng(3).standard_normal(g.n)
    b -= np.cumsum(b)[-1] / g.n
    b[1:] -= b[:-1].copy() * 0.9
    b -= b.mean()
    x = torch.empty(1, g.n, dtype=torch.float64, device="cuda")
    rwc.rwc_solve(rwc.Graph.from_synth(g).handle, 1, torch.as_tensor(b[None], device="cuda"), x, tol)
    x = x.cpu().numpy()[0]
    A = sparse.csr_matrix((np.ones(g.nnz), g.col, g.row_ptr), shape=(g.n, g.n))
    r = b - (np.diff(g.row_ptr) * x - A @ x)
    assert np.linalg.norm(r - r.mean()) <= 1.01 * tol * np.linalg.norm(b)
    assert abs(x.mean()) <= 1e-12 * np.abs(x).max()
