"""Where the mixed-precision COCG SpMM goes through bricks and where it does not (slrf_bricks), and
the forms of it that need the choice to be known: the Jacobi preconditioner and the autotuner."""
import numpy as np
import pytest
import torch

import slrf_inputs as si
from gpu_common import slrf_mod  # noqa: F401
from test_gpu_bricks import PENCILS, _scalar

pytestmark = pytest.mark.gpu


def _ctx(slrf, p, k, **opts):
    d = p.A().diagonal() / p.B().diagonal()
    return slrf.Context(p.rowptr, p.col, p.valA, p.valB, float(d.mean()), k, slrf.slrf_opts_default(it_max=3, **opts))


@pytest.mark.parametrize("name,used", [("box", True), ("odd box", True), ("thin box", True), ("plane", True),
                                       ("line", True), ("one row", False), ("shuffled", False), ("elastic", False),
                                       ("elastic line", True)])
def test_patterns_on_bricks(slrf_mod, name, used):  # noqa: F811
    """Boxes, planes and lines of any size; not a numbering without locality, and not a pencil that the
    cost model gives B-diagonal groups of three rows (12 rows of one plane share all their columns
    in the elastic line, so there four rows cost less than three)."""
    p = PENCILS[name]()
    k = min(5, p.n)
    ctx = _ctx(slrf_mod, p, k, precision=1)
    count, staged = ctx.bricks()
    assert (count > 0) == used
    if used:  # 32 rows a brick at most, 192 staged ones
        assert count * 32 >= p.n and 2 <= staged <= 192
        assert ctx.format() == (2, 0, 2)
    ctx.close()
    for opts in ({"precision": 0}, {"precision": 1, "group": 1}, {"precision": 1, "group": 2}):
        ctx = _ctx(slrf_mod, p, k, **opts)
        assert ctx.bricks() == (0, 0)
        ctx.close()


@pytest.mark.parametrize("opts", [{"precond": 1}, {"autotune": 1}, {"precond": 1, "refine_max": 2}])
@pytest.mark.parametrize("nodes,k", [((9, 8, 7), 33), ((17, 22), 5)])
def test_preconditioned_and_tuned_bricks_equal_plain_rows(slrf_mod, nodes, k, opts):  # noqa: F811
    p = _scalar(nodes)
    X = torch.from_numpy(si.start_block(p.n, k, 3))
    out = []
    for group in (0, 1):
        ctx = _ctx(slrf_mod, p, k, precision=1, group=group, **opts)
        if "precond" in opts:
            assert (ctx.bricks()[0] > 0) == (group == 0)
        out.append(ctx.filter_apply(X).cpu().numpy())
        ctx.close()
    # FP32 sums of up to 27 terms, about 27 x 2^-24 each, through three updates
    assert np.abs(out[0] - out[1]).max() <= 1e-4 * np.abs(out[1]).max()
