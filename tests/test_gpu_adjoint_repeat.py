"""The eigenvector adjoint gives the same bits every time.  The last update of a column's solution
is left pending when its iteration stops and is added by a later launch; every block of the column
tile must add its rows' share of it.  Blocks that leave that launch before others have started must
not change what the others read, else rows miss the update in some calls and not in others (by
about the MINRES tolerance, which no comparison with a reference sees).  One and two column
tiles, tiles that stop at different steps, 108 row blocks."""
import numpy as np
import pytest
import scipy.linalg as sla
import torch

import slrf_inputs as si
from gpu_common import slrf_mod  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("k", [5, 40, 70])
def test_eigenvector_adjoint_is_repeatable(slrf_mod, k):  # noqa: F811
    nodes = (12, 12, 12)
    p = si.q1_scalar(nodes, coef=np.exp(np.random.default_rng(4).normal(0, 0.3, 11**3)), shift=1e-3)
    lam, X = sla.eigh(p.A().toarray(), p.B().toarray(), subset_by_index=[0, k - 1])
    rng = np.random.default_rng(k)
    args = [torch.from_numpy(np.ascontiguousarray(t))
            for t in (lam, X, rng.standard_normal(k), rng.standard_normal((p.n, k)))]
    ctx = slrf_mod.Context(p.rowptr, p.col, p.valA, p.valB, 1.0, k, slrf_mod.slrf_opts_default())
    first = [t.clone() for t in ctx.eig_grad(*args)]
    for _ in range(12):
        for a, b in zip(first, ctx.eig_grad(*args)):
            assert torch.equal(a, b)
    ctx.close()
