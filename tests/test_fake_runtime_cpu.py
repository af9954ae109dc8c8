"""The host side of the library on a runtime without a GPU (fake_cuda_runtime.c): what the entry
points set up for each device and what they do when device memory runs short."""
import ctypes as ct
import os
import subprocess
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

PRELUDE = """
import ctypes as ct, sys
import numpy as np
sys.path.insert(0, {root!r})
from paper_2510_17334_gb300 import slrf
fake, lib = ct.CDLL({fake!r}), slrf.lib()
fake.fake_used.restype = ct.c_size_t
fake.fake_set_limit.argtypes = [ct.c_size_t]

def pencil(n):
    ptr, col = np.arange(n + 1, dtype=np.int64), np.arange(n, dtype=np.int32)
    val = np.ones(n)
    keep = (ptr, col, val)
    p = slrf.CsrPair(n, n, *(ct.c_void_p(a.ctypes.data) for a in (ptr, col, val, val)))
    return p, keep

def setup(p, k, **opts):
    h, o = ct.c_void_p(), slrf.slrf_opts_default(**opts)
    rc = lib.slrf_setup(ct.byref(h), ct.byref(p), 1.0, k, ct.byref(o), None)
    return rc, h

def block(*shape):
    a = np.zeros(shape)
    return a, ct.c_void_p(a.ctypes.data)
"""


@pytest.fixture(scope="module")
def run(tmp_path_factory):
    """run(code): code after PRELUDE in a process with the fake runtime preloaded."""
    from paper_2510_17334_gb300 import build

    build.build()
    so = str(tmp_path_factory.mktemp("fake") / "libfakecuda.so")
    subprocess.run(["gcc", "-O1", "-shared", "-fPIC", "-o", so, os.path.join(ROOT, "tests", "fake_cuda_runtime.c")],
                   check=True)

    def go(code):
        r = subprocess.run([sys.executable, "-c", PRELUDE.format(root=ROOT, fake=so) + code], capture_output=True,
                           text=True, timeout=300, env={**os.environ, "LD_PRELOAD": so})
        assert r.returncode == 0, r.stdout + r.stderr
        return r.stdout

    return go


def test_every_device_gets_its_kernel_attributes(run):
    """The same calls on a second device of the process: FP64 groups of four rows, a split-bf16
    product and a Cholesky factor in shared memory all need more than 48 KB of it."""
    run("""
n, k = 512, 80
p, keep = pencil(n)
for dev in (0, 1, 3):
    fake.fake_set_device(dev)
    rc, h = setup(p, k, precision=0)
    assert rc == 0, (dev, rc)
    (U, u), (V, v), (t, th), (r, rs) = block(n, k), block(n, k), block(k), block(k)
    assert lib.slrf_filter_apply(h, u, k, None, v) == 0, dev
    assert lib.slrf_rayleigh_ritz(h, u, k, None, None, 0, 1, v, th, rs) == 0, dev
    lib.slrf_destroy(h)
    assert lib.slrf_tsgram(n, u, k, k, u, k, k, v, k, 1, None) == 0, dev
    assert fake.fake_refused() == 0 and fake.fake_launches() > 20, dev
""")


def test_row_scaled_copy_only_with_the_preconditioner(run):
    """The FP64 copy of a block with scaled rows (n x L doubles) is memory of preconditioned contexts
    alone; beside it they hold four arrays of a row or an entry each."""
    run("""
n, k = 4096, 96
p, keep = pencil(n)
used = []
for precond in (0, 1):
    before = fake.fake_used()
    rc, h = setup(p, k, precision=0, precond=precond)
    assert rc == 0
    used.append(fake.fake_used() - before)
    lib.slrf_destroy(h)
assert used[1] - used[0] >= 8 * n * k, used
""")
