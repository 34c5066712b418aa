"""Steps whose passes run on two branches of the graph, against one branch: the branches
share the decoded spins' and the energy partials' buffers, meet in the step's tail, and
fork again in the next replay."""
import numpy as np
import pytest

from paper_1204_6192_gb300 import hsg, inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _build():
    import __graft_entry__
    __graft_entry__.build()


def run(samples, branches, **kw):
    ctx = hsg.Context(samples, 2, 3, step_branches=branches, **kw)
    n = len(samples)
    out = []

    def state():
        m = ctx.measure()
        out.extend([np.concatenate([s.ravel() for s in ctx.get_spins()]), ctx.last_energies(), ctx.get_perm(),
                    m["E"], m["q"], m["qk"], ctx.pt_stats()[0], np.stack(ctx.counters())])

    ctx.step(5)
    state()
    ctx.set_active([n == 1 or k != n // 2 for k in range(n)])
    ctx.step(3)
    state()
    ctx.set_active(None)
    ctx.sweep_or(1)
    ctx.step(2)
    keep = np.concatenate([s.ravel() for s in ctx.get_spins()])
    ctx.step(1)
    ctx.set_spins(keep)
    ctx.step(2)
    state()
    info = ctx.info()
    ctx.close()
    return out, info


@pytest.mark.parametrize("parts", [2, 3, 4, 5])
@pytest.mark.parametrize("precision,Ls,kernel,chunks", [
    ("fp16", (32, 32, 32), hsg.SWEEP_HALF, 1), ("fp32", (16, 20, 24, 14), hsg.SWEEP_HALF, 2),
    ("oct16", (16, 20, 24, 14), hsg.SWEEP_HALF, 1), ("fp16", (32, 32, 32), hsg.SWEEP_STAGED, 2),
    ("bf16", (64,), hsg.SWEEP_STAGED, 1), ("yx4", (24,), hsg.SWEEP_HALF, 1)])
def test_two_branches_equal_one(precision, Ls, kernel, chunks, parts):
    """Several passes (odd and even numbers of them), a frozen sample, replays, and spins
    read, measured and set between them: the same bits as the passes one after the other."""
    samples = [inputs.small_sample(L, n_temps=12, disorder_seed=L + k) for k, L in enumerate(Ls)]
    kw = {"variant": hsg.VARIANT_TWO_PASS, "precision": precision, "j_fp16": precision == "fp16",
          "chunks_per_thread": chunks, "sweep_kernel": kernel}
    ctx = hsg.Context(samples, 2, 3, **kw)
    footprint = (ctx.info().spin_bytes + ctx.info().rec_bytes) // parts
    ctx.close()
    ref, one = run(samples, 1, pass_bytes=footprint, **kw)
    out, two = run(samples, 2, pass_bytes=footprint, **kw)
    assert one.step_branches == 1 and two.step_branches == 2
    assert one.n_passes == two.n_passes >= 2
    for k, (a, b) in enumerate(zip(out, ref)):
        np.testing.assert_array_equal(a, b, err_msg=str(k))


def test_asked_for_of_the_tuner_and_without_passes():
    """Two branches asked for without a pass footprint: two halves of the systems; the
    automatic schedule then times two-branch steps only, and none with one asked for."""
    samples = [inputs.small_sample(24, n_temps=12, disorder_seed=1)]
    ref, info = run(samples, 1, variant=hsg.VARIANT_TWO_PASS)
    assert (info.step_branches, info.n_passes) == (1, 1)
    for variant, branches in ((hsg.VARIANT_TWO_PASS, 2), (hsg.VARIANT_AUTO, 2), (hsg.VARIANT_AUTO, 1)):
        out, info = run(samples, branches, variant=variant)
        assert info.step_branches == branches
        for k, (a, b) in enumerate(zip(out, ref)):
            np.testing.assert_array_equal(a, b, err_msg=str((variant, k)))


def test_schedules_without_branches():
    """The wave and fused sweeps, the persistent schedule and a single chunk group run on
    one branch; other values are refused."""
    smp = inputs.small_sample(16, n_temps=8, disorder_seed=1)
    for kw in ({"variant": hsg.VARIANT_TWO_PASS, "sweep_kernel": hsg.SWEEP_WAVE}, {"variant": hsg.VARIANT_PERSISTENT},
               {"variant": hsg.VARIANT_TWO_PASS, "sweep_kernel": hsg.SWEEP_FUSED}, {"sweep_kernel": hsg.SWEEP_WAVE}):
        _, info = run([smp], 2, **kw)
        assert info.step_branches == 1, kw
    one = inputs.small_sample(16, n_temps=2, disorder_seed=1)
    ctx = hsg.Context([one], 2, 3, variant=hsg.VARIANT_TWO_PASS, step_branches=2, chunks_per_thread=2)
    assert ctx.info().step_branches == 1
    ctx.close()
    for bad in (-1, 3):
        with pytest.raises(hsg.HsgError, match="step_branches"):
            hsg.Context([smp], 2, 1, step_branches=bad)


@pytest.mark.parametrize("L,n_samples,kernel", [(8, 64, 5), (10, 8, 5), (12, 28, 5), (12, 32, 1), (10, 64, 1)])
def test_explicit_two_pass_takes_the_resident_sweeps_where_they_win(L, n_samples, kernel):
    """No timing stands behind an explicit schedule: resident up to L = 8, above only with
    few systems (32 a sample here), where launches and latency count."""
    samples = [inputs.small_sample(L, n_temps=16, disorder_seed=k) for k in range(2)] * (n_samples // 2)
    ctx = hsg.Context(samples, 2, 3, precision="fp16", variant=hsg.VARIANT_TWO_PASS)
    assert ctx.info().sweep_kernel == kernel
    ctx.close()
