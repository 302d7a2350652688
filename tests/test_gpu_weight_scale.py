"""Laplacian solves and gradients on graphs whose weights are all scaled by a
power of two far from 1: L^+ and the gradient scale by its inverse."""
import numpy as np
import pytest
import torch
from scipy import sparse

import paper_2510_20604_gb300 as rwc
import synth

pytestmark = pytest.mark.gpu

GRAPHS = {"small": lambda: synth.ba(700, 3, seed=4, sigma=0.5),         # rows in registers
          "general": lambda: synth.rgg(30000, 10.0, seed=4, sigma=0.5),
          "hub": lambda: synth.from_edges(3000, [0] * 2999 + list(range(1, 2999)), list(range(1, 3000)) + list(range(2, 3000)),
                                          np.random.default_rng(1).lognormal(0.0, 0.5, 5997))}


def _scaled(g, e):
    return synth.graphs.Graph(g.n, g.row_ptr, g.col, np.ldexp(g.w, e).astype(np.float32))


@pytest.mark.parametrize("e", [-110, -80, 80, 110])
@pytest.mark.parametrize("k", [1, 3])
@pytest.mark.parametrize("kind", list(GRAPHS))
def test_solve_with_scaled_weights(kind, k, e):
    g = GRAPHS[kind]()
    b = np.random.default_rng(7).standard_normal((k, g.n))
    b -= b.mean(1, keepdims=True)
    bt = torch.as_tensor(b, device="cuda")
    x = torch.empty_like(bt)
    base, iters = (rwc.rwc_solve(rwc.Graph.from_synth(h).handle, k, bt, x, 1e-10) for h in (g, _scaled(g, e)))
    # the same arithmetic up to powers of two: no idle iterations
    assert iters <= 1.25 * base, (iters, base)
    x = np.ldexp(x.cpu().numpy(), e)
    A = sparse.csr_matrix((g.w.astype(np.float64), g.col, g.row_ptr), shape=(g.n, g.n))
    r = b - (np.asarray(A.sum(1)).ravel() * x - (A @ x.T).T)
    # the solver's own criterion, and rounding in the evaluation of r
    assert (np.linalg.norm(r, axis=1) <= 2e-10 * np.linalg.norm(b, axis=1)).all()


@pytest.mark.parametrize("e", [-80, 80])
def test_gradient_with_scaled_weights(e):
    g = GRAPHS["small"]()
    c = torch.as_tensor(synth.uniform_vector(g.n, 5), device="cuda")
    ref, got = (rwc.Graph.from_synth(h).grad(c, k=8, sketch_seed=2).double().cpu().numpy() for h in (g, _scaled(g, e)))
    # both solves end at a relative residual of 1e-8 on a system of condition below 1e3
    assert np.abs(np.ldexp(got, e) - ref).max() <= 1e-5 * np.abs(ref).max()
