"""The adjoint's kernels at the edges of their tiles.  Eigenvalue terms on the pattern against the
sums written out in numpy: symmetric patterns (mirrored entries), patterns whose mirror entries are
missing or whose rows are not sorted, even and odd numbers of eigenpairs, row counts around the
row bundles of a warp."""
import numpy as np
import pytest
import scipy.linalg as sla
import torch

import slrf_inputs as si
from gpu_common import slrf_mod  # noqa: F401
from oracle import slrf_oracle as orc

pytestmark = pytest.mark.gpu


def _pattern(n, form, rng):
    """CSR pattern with a full diagonal: symmetric, without most mirrors, or unsorted."""
    D = rng.random((n, n)) < 0.3
    D = (D | D.T) if form == "symmetric" else D
    np.fill_diagonal(D, True)
    rows = [np.nonzero(D[i])[0] for i in range(n)]
    if form == "unsorted":
        rows = [rng.permutation(r) for r in rows]
    rowptr = np.concatenate([[0], np.cumsum([len(r) for r in rows])]).astype(np.int64)
    return rowptr, np.concatenate(rows).astype(np.int32)


@pytest.mark.parametrize("form", ["symmetric", "missing", "unsorted"])
@pytest.mark.parametrize("n,k", [(1, 1), (7, 2), (8, 33), (65, 3), (130, 50), (64, 200), (9, 1600)])
def test_eigenvalue_adjoint_sums(slrf_mod, n, k, form):  # noqa: F811
    rng = np.random.default_rng(n * 1000 + k)
    rowptr, col = _pattern(n, form, rng)
    vals = np.ones(len(col))
    ctx = slrf_mod.Context(rowptr, col, vals, vals, 1.0, 1, slrf_mod.slrf_opts_default(m=1, group=1))
    lam, g, X = rng.random(k) + 0.5, rng.standard_normal(k), rng.standard_normal((n, k))
    gA, gB = (t.cpu().numpy() for t in ctx.eig_grad(torch.from_numpy(lam), torch.from_numpy(X), torch.from_numpy(g)))
    r = np.repeat(np.arange(n), np.diff(rowptr))
    terms = g * X[r] * X[col]
    # three roundings a product, k additions
    bound = (k + 3) * 2.0 ** -53
    assert np.all(np.abs(gA - terms.sum(1)) <= 2 * bound * np.abs(terms).sum(1))
    assert np.all(np.abs(gB + (lam * terms).sum(1)) <= 2 * bound * np.abs(lam * terms).sum(1))
    ctx.close()


@pytest.mark.parametrize("k", [1, 8, 9, 16, 17, 33, 65])
def test_eigenvector_adjoint_column_tiles(slrf_mod, k):  # noqa: F811
    """Eigenvector terms at block widths around the lane groups (8, 16, 32 columns) and tiles
    of the MINRES kernels, against the oracle's dense least squares; the relative residual
    1e-12 grows by the 1D bar's spread lambda_max / gap < 1e4."""
    p = si.bar1d_pencil(90)
    lam, X = sla.eigh(p.A().toarray(), p.B().toarray())
    lam, X = lam[:k], np.ascontiguousarray(X[:, :k])
    rng = np.random.default_rng(k)
    g, gX = rng.standard_normal(k), rng.standard_normal((p.n, k))
    ctx = slrf_mod.Context(p.rowptr, p.col, p.valA, p.valB, 1.0, k, slrf_mod.slrf_opts_default(tol_inner=1e-13))
    out = ctx.eig_grad(*(torch.from_numpy(t) for t in (lam, X, g, gX)))
    for got, want in zip(out, orc.eig_grad_full(p.rowptr, p.col, p.A(), p.B(), lam, X, g, gX)):
        assert np.abs(got.cpu().numpy() - want).max() <= 1e-8 * np.abs(want).max()
    ctx.close()
