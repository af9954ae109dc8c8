"""A batch of blocks wide enough for the many-CTA Cholesky (96 columns and more).  The problems'
outer updates run side by side on their own streams, so CTAs of one factorisation start at any time
of it, also after its first CTA has finished; the factor must not depend on that.  Every problem is
bitwise equal to its own single FP64 solve (plain CSR), and a second pass of the batch to the
first."""
import numpy as np
import pytest
import torch

import pins
import slrf_inputs as si
from gpu_common import slrf_mod  # noqa: F401

pytestmark = pytest.mark.gpu


def test_wide_blocks_in_a_batch_equal_single_solves(slrf_mod):  # noqa: F811
    probs = []
    for i, nodes in enumerate([(13, 12, 11), (12, 12, 12), (14, 11, 10), (11, 13, 12), (12, 13, 13), (10, 14, 12)]):
        lam = pins.q1_neumann_eigs(nodes, 1e-3)
        gamma, cnt = pins.gap_gamma(lam, 66)
        L = 97 + 7 * i  # the last panel of 32 columns has 1 to 32 of them
        probs.append((si.q1_scalar(nodes, shift=1e-3), gamma, cnt, L))
    opts = dict(it_max=30, precision=0, group=1)
    V0 = [si.start_block(p.n, L, 40 + i) for i, (p, _, _, L) in enumerate(probs)]
    batch = slrf_mod.Batch([(p.rowptr, p.col, p.valA, p.valB) for p, *_ in probs], [g for _, g, _, _ in probs],
                           [L for *_, L in probs], slrf_mod.slrf_opts_default(**opts))
    passes = []
    for _ in range(2):
        rc, res, _ = batch.solve(V0)
        assert rc == 0
        passes.append([(nf, ev.clone(), X.clone()) for _, nf, ev, X, _ in res])
    batch.close()
    for i, (p, gamma, cnt, L) in enumerate(probs):
        ctx = slrf_mod.Context(p.rowptr, p.col, p.valA, p.valB, gamma, L, slrf_mod.slrf_opts_default(**opts))
        _, nf1, ev1, X1, _, _ = ctx.solve(torch.from_numpy(V0[i]))
        ctx.close()
        for nf, ev, X in (passes[0][i], passes[1][i]):
            assert nf == nf1 == cnt, i
            assert torch.equal(ev1, ev) and torch.equal(X1, X), i
