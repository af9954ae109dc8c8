"""Setup when device memory is short: the SpMM formats that the library chooses by itself must not
take the memory that the rest of the working set needs."""
import numpy as np
import pytest
import torch

from gpu_common import slrf_mod  # noqa: F401

pytestmark = pytest.mark.gpu


def _free():
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    return torch.cuda.mem_get_info()[0]


def test_chosen_formats_leave_room_for_the_working_set(slrf_mod):  # noqa: F811
    """A line of 2M rows (15 GB of working set, 0.27 GB of bricks and pair records): with 0.1 GB
    more free memory than plain rows need, group = 0 sets up and gives what plain rows give."""
    n, k = 2_000_000, 1
    ptr = np.minimum(np.maximum(3 * np.arange(n + 1) - 1, 0), 3 * n - 2).astype(np.int64)
    col = (np.arange(n)[:, None] + np.arange(-1, 2)).ravel()
    A = np.tile([-1.0, 2.5, -1.0], n)
    B = np.tile([0.0, 1.0, 0.0], n)
    ok = (col >= 0) & (col < n)
    args = [torch.from_numpy(t[ok] if t is not ptr else t).cuda() for t in (ptr, col.astype(np.int32), A, B)]
    X = torch.randn(n, k, dtype=torch.float64, generator=torch.Generator().manual_seed(1)).cuda()

    def apply(group):
        ctx = slrf_mod.Context(*args, 0.5, k, slrf_mod.slrf_opts_default(m=1, it_max=3, precision=1, group=group))
        left, U = torch.cuda.mem_get_info()[0], ctx.filter_apply(X).clone()
        ctx.close()
        return left, U

    apply(1)  # loads what the process keeps
    before = _free()
    left, want = apply(1)
    room = before - left + 100 * 2**20
    hog = torch.empty(_free() - room, dtype=torch.uint8, device="cuda")
    try:
        _, got = apply(0)
    finally:
        del hog
        torch.cuda.empty_cache()
    assert torch.equal(got, want)
