"""The bounds-checked build (-DHSG_CHECK) on the resident sweeps, which small lattices run
by default: half-sites within the block's threads and shared memory, neighbours within
the lattice, the pair of systems within the sample.  In a child process (the binding
loads one build per process) it must report no error and give the same spins and
energies, bit for bit, as the normal build."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

# lattices of a context, precision, j_fp16, options
CASES = [((L,), prec, j16, {}) for L in (4, 6, 8, 10, 12) for prec, j16 in (("fp32", False), ("fp16", True), ("oct16", False))]
CASES += [((12, 4, 10), "bf16", True, {}), ((6, 8), "yx4", False, {}), ((4, 12), "angle16", False, {"n_hb": 2, "n_or": 0})]

CODE = r"""
import hashlib, sys
sys.path.insert(0, ROOT)
from paper_1204_6192_gb300 import hsg, inputs
if LIB:
    hsg.use_library(LIB)
for Ls, prec, j16, kw in CASES:
    samples = [inputs.small_sample(L, n_temps=5, h_r=0.1, disorder_seed=L) for L in Ls]
    ctx = hsg.Context(samples, 3, 7, precision=prec, j_fp16=j16, variant=hsg.VARIANT_TWO_PASS, **kw)
    assert ctx.info().sweep_kernel == 5
    ctx.step(2)
    ctx.set_active([k != 1 for k in range(len(Ls))])
    ctx.step(1)
    m = ctx.last_energies()
    print(hashlib.sha256(b"".join(x.tobytes() for x in ctx.get_spins()) + m.tobytes()).hexdigest(), flush=True)
    ctx.sync()
    ctx.close()
print("ok")
"""


def digests(lib):
    code = f"ROOT = {ROOT!r}\nLIB = {lib!r}\nCASES = {CASES!r}\n" + CODE
    r = subprocess.run([sys.executable, "-c", code], capture_output=True, text=True, timeout=900, cwd=ROOT)
    assert r.returncode == 0 and r.stdout.strip().endswith("ok"), r.stdout[-2000:] + r.stderr[-2000:]
    return r.stdout.split()[:-1]


def test_resident_sweeps_in_the_checked_build():
    import __graft_entry__
    __graft_entry__.build()
    from paper_1204_6192_gb300 import build
    got = digests(build.build(check=True))
    assert len(got) == len(CASES)
    for case, a, b in zip(CASES, got, digests(None)):
        assert a == b, case
