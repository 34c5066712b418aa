"""Staged and wave sweeps at every row length that has its own code (L = 32 to 256 here,
alone and mixed in one context): the same bits as half-sweeps that load into registers."""
import numpy as np
import pytest

from paper_1204_6192_gb300 import hsg, inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _build():
    import __graft_entry__
    __graft_entry__.build()


@pytest.mark.parametrize("Ls,n_temps,precision,j16", [
    ((32,), 5, "fp32", False), ((32, 32), 9, "bf16", True), ((64,), 5, "fp16", False), ((128,), 3, "bf16", False),
    ((32, 128), 3, "bf16", True), ((64, 32, 128, 64), 5, "fp32", False), ((64, 32, 128, 64), 5, "fp16", True),
    ((256,), 1, "fp16", True), ((32, 256), 1, "fp32", False)])
def test_staged_and_wave_equal_half_sweeps(Ls, n_temps, precision, j16):
    """With one and several chunk groups a thread (one stage and two), a frozen sample."""
    distinct = {L: inputs.small_sample(L, n_temps=n_temps, disorder_seed=L) for L in Ls}
    samples = [distinct[L] for L in Ls]
    for chunks in ((0,) if max(Ls) > 128 else (1, 3)):
        out = []
        for kernel in (hsg.SWEEP_HALF, hsg.SWEEP_STAGED, hsg.SWEEP_WAVE):
            ctx = hsg.Context(samples, 2, 5, precision=precision, j_fp16=j16, variant=hsg.VARIANT_TWO_PASS,
                              sweep_kernel=kernel, chunks_per_thread=chunks)
            assert ctx.info().sweep_kernel == kernel
            ctx.sweep_or(1)
            ctx.set_active([k != 1 for k in range(len(Ls))])
            ctx.step(1)
            out.append([ctx.last_energies(), ctx.get_perm()] + [s.copy().view(np.uint32) for s in ctx.get_spins()])
            ctx.close()
        for o in out[1:]:
            for a, b in zip(o, out[0]):
                np.testing.assert_array_equal(a, b)
