"""Energies of contexts whose threads walk many chunk groups: the energy kernel's
per-warp sums take 256 bytes of shared memory a chunk group, beyond the 48 kB a launch
has without asking from 193 groups a thread on."""
import numpy as np
import pytest

import oracle
from paper_1204_6192_gb300 import hsg, inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _build():
    import __graft_entry__
    __graft_entry__.build()


def sample():
    raw = inputs.small_sample(4, n_temps=256, h_r=0.1, disorder_seed=21, t_min=0.2, t_max=3.0)
    return inputs.Sample(L=4, J=inputs.round_fp16(raw.J), H=inputs.round_fp16(raw.H), temps=raw.temps)


def run(precision, chunks):
    """Spins and energies of the initial state, a measurement after set_spins, a PT pass,
    and a step without over-relaxation (whose energies come from the same kernel)."""
    ctx = hsg.Context([sample()], 4, 3, precision=precision, chunks_per_thread=chunks, n_hb=1, n_or=0)
    assert ctx.info().chunks_per_thread == chunks
    out = [ctx.get_spins()[0].copy(), ctx.energies()[0]]
    ctx.set_spins([out[0][::-1].copy()])
    out.append(ctx.measure()["E"])
    ctx.pt_exchange()
    out += [ctx.last_energies(), ctx.get_perm()]
    ctx.step(1)
    out += [ctx.last_energies(), ctx.get_perm(), ctx.get_spins()[0].copy()]
    ctx.close()
    return out


@pytest.mark.parametrize("precision", ["fp32", "fp16", "oct16"])
def test_energies_with_many_chunk_groups_per_thread(precision):
    """256 temperatures of four replicas at L = 4 (256 chunk groups): the same numbers
    with 16, 192 (48 kB), 193 and 256 groups a thread, and the oracle's energies."""
    ref = run(precision, 16)
    for chunks in (192, 193, 256):
        for k, (a, b) in enumerate(zip(run(precision, chunks), ref)):
            np.testing.assert_array_equal(a, b, err_msg=f"{chunks} {k}")
    smp = sample()
    o = oracle.OracleSample(4, smp.J, smp.H, smp.temps, 4, 0, 0, 3, 0)
    o.s = ref[0].astype(np.float64)
    # ten binary32 roundings on the way to a site's term, five in its warp's sum
    bound = 15 * 2.0 ** -24 * (np.abs(smp.J).sum() + np.linalg.norm(smp.H, axis=1).sum())
    assert np.abs(ref[1] - o.energies()).max() <= bound
