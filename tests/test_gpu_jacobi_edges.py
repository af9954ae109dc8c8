"""The projected eigensolver at the ends of the number range: a projection that is not finite ends
after a sweep instead of running all of them, and subnormal entries give no NaN."""
import time

import numpy as np
import pytest
import torch

import slrf_inputs as si
from gpu_common import slrf_mod  # noqa: F401

pytestmark = pytest.mark.gpu


def test_not_finite_projection_ends_at_once(slrf_mod):  # noqa: F811
    """A block with NaNs is refused (its Gram matrix has no Cholesky factor) in no more time than a
    good block takes; the eigensolver runs in both calls, eight sweeps or so for the good one."""
    p = si.q1_scalar((12, 12, 12), shift=1e-3)
    k = 480
    ctx = slrf_mod.Context(p.rowptr, p.col, p.valA, p.valB, 1.0, k, slrf_mod.slrf_opts_default())
    good = torch.from_numpy(si.start_block(p.n, k, 3)).cuda()
    bad = torch.full_like(good, float("nan"))
    times = []
    for U in (good, good, bad):
        torch.cuda.synchronize()
        t = time.perf_counter()
        if U is bad:
            with pytest.raises(RuntimeError):
                ctx.rayleigh_ritz(U.clone())
        else:
            ctx.rayleigh_ritz(U.clone())
        torch.cuda.synchronize()
        times.append(time.perf_counter() - t)
    ctx.close()
    assert times[2] <= times[1]


@pytest.mark.parametrize("scale", [1e-310, 1e-305, 1e-200, 1e200, 1e300])
def test_projection_at_the_ends_of_the_range(slrf_mod, scale):  # noqa: F811
    """A = scale K with K = [[3, 1], [1, 3]] blocks, B = 1, U = unit vectors: the projection is A itself,
    its eigenvalues 2 and 4 times scale.  Below 2.3e-308 the entries are subnormal and are left as
    they are."""
    n, k = 8, 4
    rowptr = np.arange(0, 2 * n + 1, 2)
    col = np.repeat(np.arange(n).reshape(-1, 2), 2, 0).ravel()
    K = np.tile([3.0, 1.0, 1.0, 3.0], n // 2)
    one = np.tile([1.0, 0.0, 0.0, 1.0], n // 2)
    ctx = slrf_mod.Context(rowptr, col, scale * K, one, 1.0, k, slrf_mod.slrf_opts_default(dense=0, m=1))
    V, theta = (t.cpu().numpy() for t in ctx.rayleigh_ritz(torch.eye(n, k, dtype=torch.float64))[1:3])
    ctx.close()
    assert np.all(np.isfinite(V)) and np.all(np.isfinite(theta))
    assert np.abs(V.T @ V - np.eye(k)).max() <= 1e-14
    if scale >= 2.3e-308:
        assert np.abs(theta / scale - [2, 2, 4, 4]).max() <= 1e-14
