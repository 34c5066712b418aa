"""Results too large for the pinned buffer (64 MB): read through plain host memory, with
the same values; and HSG_ENOMEM, not an exception through the C entry point, where the
host has none left."""
import ctypes
import os
import subprocess
import sys

import numpy as np
import pytest

from paper_1204_6192_gb300 import hsg, inputs

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module", autouse=True)
def _build():
    import __graft_entry__
    __graft_entry__.build()


def large(n):
    """n samples of L = 4 with 128 temperatures: 64 kB of q and q(k) each."""
    one = [inputs.small_sample(4, n_temps=128, disorder_seed=k) for k in range(4)]
    return hsg.Context([one[k % 4] for k in range(n)], 2, 3, variant=hsg.VARIANT_TWO_PASS)


def test_results_beyond_the_pinned_buffer():
    """77 MB of results at once, and the same arrays one at a time (11 MB of q: pinned)."""
    ctx = large(1200)
    ctx.step(1)
    m = ctx.measure()
    for name in ("q", "qk"):
        out, obs = np.full_like(m[name], np.nan), hsg.Obs()
        setattr(obs, name, out.ctypes.data_as(ctypes.POINTER(ctypes.c_double)))
        assert hsg.lib().hsg_measure(ctx.handle, ctypes.byref(obs)) == 0
        np.testing.assert_array_equal(out, m[name])
    e = ctx.measure(q=False)
    for name in ("E", "perm"):
        np.testing.assert_array_equal(e[name], m[name])
    np.testing.assert_array_equal(ctx.get_perm(), m["perm"])
    ctx.close()


CODE = r"""
import resource, sys
sys.path.insert(0, ROOT)
sys.path.insert(0, ROOT + "/tests")
import test_gpu_large_results as t
from paper_1204_6192_gb300 import hsg
few = t.large(4)
few.step(1)
few.measure()
ctx = t.large(1200)
ctx.step(1)
ctx.measure()
import ctypes, numpy as np
qk = np.zeros((1200, 128, 3, 3, 3, 2))
obs = hsg.Obs()
obs.qk = qk.ctypes.data_as(ctypes.POINTER(ctypes.c_double))
used = int(open("/proc/self/statm").read().split()[0]) * resource.getpagesize()
resource.setrlimit(resource.RLIMIT_AS, (used + (8 << 20), resource.RLIM_INFINITY))
st = hsg.lib().hsg_measure(ctx.handle, ctypes.byref(obs))
resource.setrlimit(resource.RLIMIT_AS, (resource.RLIM_INFINITY, resource.RLIM_INFINITY))
print("status", st, hsg.lib().hsg_last_error(ctx.handle).decode())
ctx.close()
"""


def test_no_host_memory_for_the_results():
    r = subprocess.run([sys.executable, "-c", f"ROOT = {ROOT!r}\n" + CODE], capture_output=True, text=True,
                       timeout=300, cwd=ROOT)
    assert r.returncode == 0 and "status 2" in r.stdout, r.stdout[-1000:] + r.stderr[-2000:]
