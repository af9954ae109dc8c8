"""The FP32 SpMM on bricks (row groups with their gathered rows staged in shared memory) against
the plain CSR kernel: the same filter apply, from the same block, with slrf_opts.group = 0 (bricks
where the pattern has them) and group = 1.  Meshes whose sides leave ragged bricks and single rows
at the end of a line, planes, a line, 3-dof boxes, one column tile and many, one to 32 poles, a
numbering without locality (no bricks), refinement steps and a batch."""
import numpy as np
import pytest
import torch

import slrf_inputs as si
from gpu_common import slrf_mod  # noqa: F401

pytestmark = pytest.mark.gpu


def _scalar(nodes, seed=0):
    ne = int(np.prod([s - 1 for s in nodes]))
    return si.q1_scalar(nodes, coef=np.exp(np.random.default_rng(seed).normal(0, 0.3, ne)), shift=1e-3)


def _shuffled(p):
    import scipy.sparse as sp

    q = np.random.default_rng(5).permutation(p.n)
    A, B = p.A()[q][:, q].tocsr(), p.B()[q][:, q].tocsr()
    A.sort_indices()
    B.sort_indices()
    return type(p)(p.n, A.indptr.astype(np.int64), A.indices.astype(np.int32), A.data, B.data)


PENCILS = {
    "box": lambda: _scalar((9, 8, 7)),
    "odd box": lambda: _scalar((13, 5, 3)),
    "thin box": lambda: _scalar((2, 2, 40)),
    "plane": lambda: _scalar((17, 22)),
    "line": lambda: si.bar1d_pencil(203),
    "one row": lambda: si.bar1d_pencil(1),
    "shuffled": lambda: _shuffled(_scalar((9, 8, 7))),
    "elastic": lambda: si.q1_elasticity((6, 5, 4), E=np.exp(np.random.default_rng(1).normal(0, 0.5, 60))),
    "elastic line": lambda: si.q1_elasticity((2, 2, 9)),
}


@pytest.mark.parametrize("m,k,refine", [(8, 5, 1), (8, 33, 1), (1, 40, 1), (2, 3, 1), (32, 7, 1), (8, 9, 2)])
@pytest.mark.parametrize("name", list(PENCILS))
def test_bricks_equal_plain_rows(slrf_mod, name, m, k, refine):  # noqa: F811
    p = PENCILS[name]()
    k = min(k, p.n)
    X = torch.from_numpy(si.start_block(p.n, k, 3))
    d = p.A().diagonal() / p.B().diagonal()
    gamma = float(d.mean())  # poles next to the diagonal: three updates stay well conditioned
    out = []
    for group in (0, 1):
        opts = slrf_mod.slrf_opts_default(m=m, it_max=3, precision=1, group=group, refine_max=refine)
        ctx = slrf_mod.Context(p.rowptr, p.col, p.valA, p.valB, gamma, k, opts)
        out.append(ctx.filter_apply(X).cpu().numpy())
        ctx.close()
    # FP32 sums of up to 81 terms, about 81 x 2^-24 each, through three updates
    assert np.abs(out[0] - out[1]).max() <= 1e-4 * np.abs(out[1]).max()


def test_batch_on_bricks(slrf_mod):  # noqa: F811
    """A mixed batch of boxes, a plane and a 3-dof box (all on bricks) finds what single solves find."""
    probs = [_scalar((9, 8, 7)), _scalar((17, 22)), PENCILS["elastic"]()]
    import scipy.linalg as sla

    lams = [sla.eigh(p.A().toarray(), p.B().toarray(), eigvals_only=True) for p in probs]
    gammas = [float(0.5 * (lam[7] + lam[8])) for lam in lams]
    batch = slrf_mod.Batch([(p.rowptr, p.col, p.valA, p.valB) for p in probs], gammas, [14] * 3,
                           slrf_mod.slrf_opts_default(it_max=60, precision=1))
    rc, res, _ = batch.solve([si.start_block(p.n, 14, 7) for p in probs])
    assert rc == 0
    for lam, (status, nf, ev, X, rs) in zip(lams, res):
        assert status == 0 and nf == 8
        assert np.all(np.abs(ev.cpu().numpy() - lam[:8]) <= 1e-8 * lam[:8])
    batch.close()
