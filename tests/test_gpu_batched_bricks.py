"""Mixed-precision batches whose problems are on bricks, all of them or some: every problem finds
the pairs of a dense eigensolver (eigenvalues to 1e-8, the tolerance of mixed solves), with and without
refinement steps and the CUDA graph, and each problem keeps its own format."""
import numpy as np
import pytest
import scipy.linalg as sla

import slrf_inputs as si
from gpu_common import slrf_mod  # noqa: F401
from test_gpu_bricks import PENCILS, _scalar, _shuffled

pytestmark = pytest.mark.gpu

PROBLEMS = {"box": lambda: _scalar((9, 8, 7)), "plane": lambda: _scalar((17, 22)),
            "odd box": lambda: _scalar((13, 5, 3)), "elastic": PENCILS["elastic"],
            "shuffled": lambda: _shuffled(_scalar((8, 7, 6)))}
ON_BRICKS = {"box", "plane", "odd box"}


def _batch(slrf, names, **opts):
    probs = [PROBLEMS[s]() for s in names]
    lams = [sla.eigh(p.A().toarray(), p.B().toarray(), eigvals_only=True) for p in probs]
    gammas = [float(0.5 * (lam[7] + lam[8])) for lam in lams]
    b = slrf.Batch([(p.rowptr, p.col, p.valA, p.valB) for p in probs], gammas, [14] * len(probs),
                   slrf.slrf_opts_default(it_max=60, precision=1, **opts))
    return b, probs, lams


@pytest.mark.parametrize("opts", [{}, {"refine_max": 2}, {"use_graph": 0}], ids=["graph", "refined", "launches"])
@pytest.mark.parametrize("names", [["box", "plane", "odd box"], ["elastic", "box", "shuffled", "plane"],
                                   ["box", "elastic"], ["shuffled", "elastic"]], ids="-".join)
def test_batches_of_both_formats(slrf_mod, names, opts):  # noqa: F811
    b, probs, lams = _batch(slrf_mod, names, **opts)
    for i, s in enumerate(names):
        assert (b.bricks(i)[0] > 0) == (s in ON_BRICKS), s
    rc, res, _ = b.solve([si.start_block(p.n, 14, 7) for p in probs])
    assert rc == 0
    for lam, (status, nf, ev, X, rs) in zip(lams, res):
        assert status == 0 and nf == 8
        assert np.all(np.abs(ev.cpu().numpy() - lam[:8]) <= 1e-8 * lam[:8])
    b.close()


def test_a_batch_honours_plain_rows(slrf_mod):  # noqa: F811
    """slrf_opts.group = 1 asks for plain CSR in a batch as in a single context."""
    b, _, _ = _batch(slrf_mod, ["box", "plane"], group=1)
    assert b.bricks(0) == b.bricks(1) == (0, 0)
    b.close()
