"""Block solves whose columns converge after different numbers of iterations: the
ones that are done stand still."""
import numpy as np
import pytest
import torch

import paper_2510_20604_gb300 as rwc
import synth

pytestmark = pytest.mark.gpu


# D^-1 L has one (complete) or two (star) non-zero eigenvalues: an inner solve ends at
# its first look at the residual, after 8 iterations, and two or three reach 1e-8; a
# fourth is allowed for.
@pytest.mark.parametrize("make,n,k", [(synth.complete, 300, 33), (synth.complete, 1500, 64), (synth.star, 300, 7),
                                      (synth.star, 300, 16), (synth.star, 300, 64), (synth.star, 3000, 16), (synth.star, 300, 70)])
def test_converged_columns_stand_still(make, n, k):
    g = make(n)
    b = np.random.default_rng(k).standard_normal((k, n))
    b -= b.mean(1, keepdims=True)
    x = torch.empty(k, n, dtype=torch.float64, device="cuda")
    it = rwc.rwc_solve(rwc.Graph.from_synth(g).handle, k, torch.as_tensor(b, device="cuda"), x, 1e-8)
    assert it <= 32
    x = x.cpu().numpy()
    if make is synth.complete:
        r = b - n * x                        # L = n I - J
    else:                                    # hub 0
        r = b - x + x[:, :1]
        r[:, 0] = b[:, 0] - (n - 1) * x[:, 0] + x[:, 1:].sum(1)
    # the solver's criterion, and rounding in the evaluation of r
    assert (np.linalg.norm(r, axis=1) <= 2e-8 * np.linalg.norm(b, axis=1)).all()


@pytest.mark.parametrize("weighted", [False, True])
def test_columns_of_very_different_length(weighted):
    """A zero column, one along an eigenvector (done at once) and random ones."""
    n = 400
    i = np.arange(n)
    w = np.random.default_rng(2).lognormal(0.0, 0.3, n) if weighted else None
    g = synth.from_edges(n, i, (i + 1) % n, w)
    b = np.random.default_rng(1).standard_normal((6, n))
    b[0], b[1] = 0.0, np.cos(2 * np.pi * i * 100 / n)
    b[2] *= 1e-100
    b[3] *= 1e100
    b -= b.mean(1, keepdims=True)
    x = torch.empty(6, n, dtype=torch.float64, device="cuda")
    rwc.rwc_solve(rwc.Graph.from_synth(g).handle, 6, torch.as_tensor(b, device="cuda"), x, 1e-8)
    x = x.cpu().numpy()
    A = np.zeros((n, n))
    A[np.repeat(i, np.diff(g.row_ptr)), g.col] = 1.0 if g.w is None else g.w
    for c in range(6):
        s = np.abs(b[c]).max() or 1.0
        r = b[c] / s - (np.diag(A.sum(1)) - A) @ (x[c] / s)
        assert np.linalg.norm(r) <= 2e-8 * np.linalg.norm(b[c] / s)
    assert not x[0].any()
