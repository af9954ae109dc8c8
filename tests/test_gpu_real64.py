"""FP64 products A X and B X through the node-triple records (slrf_apply on elasticity boxes) at the
edges of their column lanes: one column, around one, two, three and four sets of 32, and a second
pass beyond 128; with and without the row scaling of the preconditioner, from FP64 and from
mixed-precision contexts, and a box of fewer node groups than a block has warps.  Against the sparse
products in FP64, elementwise |Y - A X| <= c u (|A| |X|): a row of 81 products, the scales (ten at
most) and the final rounding stay below c = 100 roundings of u = 2^-53 each."""
import numpy as np
import pytest
import torch

import slrf_inputs as si
from gpu_common import slrf_mod  # noqa: F401

pytestmark = pytest.mark.gpu

BOUND = 100 * 2.0**-53


@pytest.mark.parametrize("nodes", [(6, 5, 4), (2, 2, 2)])
@pytest.mark.parametrize("precision,precond", [(0, 0), (0, 1), (1, 0), (1, 1)])
@pytest.mark.parametrize("k", [1, 31, 32, 33, 64, 65, 96, 97, 128, 129, 161])
def test_fp64_products_column_widths(slrf_mod, nodes, precision, precond, k):  # noqa: F811
    ne = int(np.prod([s - 1 for s in nodes]))
    p = si.q1_elasticity(nodes, E=np.exp(np.random.default_rng(1).normal(0, 0.5, ne)))
    k = min(k, p.n)
    opts = slrf_mod.slrf_opts_default(it_max=4, precision=precision, precond=precond, group=3)
    ctx = slrf_mod.Context(p.rowptr, p.col, p.valA, p.valB, 1.0, k, opts)
    X = np.random.default_rng(7 + k).standard_normal((p.n, k))
    Y = [t.cpu().numpy() for t in ctx.apply(torch.from_numpy(X), fp32=False)]
    ctx.close()
    for got, M in zip(Y, (p.A(), p.B())):
        assert np.all(np.abs(got - M @ X) <= BOUND * (abs(M) @ np.abs(X)))
