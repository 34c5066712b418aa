"""The paths a step and its tail can take, against each other and the oracle: the
resident sweeps (small lattices), the parallel-tempering pass with its decisions
taken in parallel, the packed formats' decoded neighbours carried from one
half-sweep to the next, the staged half-sweeps, and the heat bath's choice of
hemisphere at small beta |h|."""
import numpy as np
import pytest

import oracle
from paper_1204_6192_gb300 import hsg, inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _build():
    import __graft_entry__
    __graft_entry__.build()


def state(ctx):
    return {"spins": np.concatenate([s.ravel() for s in ctx.get_spins()]), "E": ctx.last_energies(),
            "perm": ctx.get_perm(), "accepted": ctx.pt_stats()[0], "moved": ctx.pt_diagnostics()[0],
            "tunnel": ctx.pt_diagnostics()[1], "counters": np.stack(ctx.counters())}


def same(a, b):
    for k in a:
        np.testing.assert_array_equal(a[k], b[k], err_msg=k)


@pytest.mark.parametrize("Ls,precision,j16,kw", [
    ((4,), "fp32", False, {}), ((6,), "fp16", True, {}), ((8,), "fp32", True, {}), ((10,), "fp16", False, {}),
    ((12,), "fp32", False, {}), ((12, 4, 8, 6), "bf16", True, {}), ((8, 10), "oct16", False, {}),
    ((12,), "angle16", True, {}), ((6, 8), "yx4", False, {}), ((8,), "fp32", False, {"n_hb": 2, "n_or": 0}),
    ((8,), "fp16", True, {"n_hb": 0, "n_or": 1}), ((10,), "fp32", False, {"fast_math": True})])
def test_resident_step_equals_half_sweeps(Ls, precision, j16, kw):
    """Three replicas of five temperatures (15 systems, one padded), a frozen sample
    in a batch: the same bits as one launch per half-sweep, energies to the order of
    their FP64 sums."""
    samples = [inputs.small_sample(L, n_temps=5, disorder_seed=L) for L in Ls]
    out = []
    for kernel in (hsg.SWEEP_HALF, hsg.SWEEP_AUTO):
        ctx = hsg.Context(samples, 3, 7, precision=precision, j_fp16=j16, variant=hsg.VARIANT_TWO_PASS,
                          sweep_kernel=kernel, **kw)
        assert ctx.info().sweep_kernel == (1 if kernel == hsg.SWEEP_HALF else 5)
        ctx.step(2)
        if len(Ls) > 1:
            ctx.set_active([k != 1 for k in range(len(Ls))])
            ctx.step(1)
            ctx.set_active(None)
        ctx.step(1)
        out.append(state(ctx))
        ctx.close()
    np.testing.assert_allclose(out[1].pop("E"), out[0].pop("E"), rtol=1e-14)
    same(out[0], out[1])


def test_resident_limit():
    """L = 12 is the largest lattice the resident sweeps take."""
    for L, kernel in ((12, 5), (14, 1)):
        ctx = hsg.Context([inputs.small_sample(L, n_temps=2)], 1, 1, variant=hsg.VARIANT_TWO_PASS)
        assert ctx.info().sweep_kernel == kernel
        ctx.close()


@pytest.mark.parametrize("R_T,R_O", [(1, 3), (2, 300), (3, 100), (5, 7), (8, 64), (9, 33), (17, 20), (31, 3), (32, 3), (33, 2), (64, 2), (97, 5), (256, 4)])
def test_pt_decisions_match_oracle(R_T, R_O):
    """Passes on given energies, where the decision words of the chains need one or
    several words a pair and one or several batches: permutations and diagnostics
    equal the oracle's sequential binary64 walk; a frozen sample keeps its own."""
    temps = inputs.geometric_temperatures(0.2, 0.2 + 0.05 * R_T, R_T)
    samples = [inputs.Sample(L=4, J=np.zeros((64, 3)), H=None, temps=temps) for _ in range(2)]
    ctx = hsg.Context(samples, R_O, 9)
    orc = oracle.OracleSim(samples, R_O, 9)
    rng = np.random.default_rng(R_T)
    for call in range(6):
        active = [1, call != 3]
        ctx.set_active(active)
        orc.set_active(active)
        E = [rng.normal(0, 4, R_T * R_O) for _ in samples]
        ctx.pt_exchange_energies(np.stack(E))
        orc.pt_exchange(E)
        for s, o in enumerate(orc.samples):
            np.testing.assert_array_equal(ctx.get_perm()[s], o.perm)
    moved, tunnel, _ = ctx.pt_diagnostics()
    for s, o in enumerate(orc.samples):
        np.testing.assert_array_equal(moved[s], o.moved)
        np.testing.assert_array_equal(tunnel[s], o.tunnel)
    ctx.close()


@pytest.mark.parametrize("precision", ["angle16", "oct16", "yx4"])
def test_decoded_neighbours_are_carried(precision):
    """Steps and sweeps that read the neighbours decoded by the half-sweep before
    them equal those of the persistent schedule, which decodes every neighbour
    itself: in several passes, with a frozen sample, and after the spins were set."""
    samples = [inputs.small_sample(L, n_temps=6, disorder_seed=L) for L in (14, 16, 20)]
    out = []
    for kw in ({"variant": hsg.VARIANT_PERSISTENT}, {"variant": hsg.VARIANT_TWO_PASS, "sweep_kernel": hsg.SWEEP_HALF},
               {"variant": hsg.VARIANT_TWO_PASS, "chunks_per_thread": 1, "pass_bytes": 300000}):
        ctx = hsg.Context(samples, 2, 3, precision=precision, **kw)
        ctx.step(2)
        ctx.set_active([1, 0, 1])
        ctx.step(1)
        ctx.set_active(None)
        keep = np.concatenate([s.ravel() for s in ctx.get_spins()])
        ctx.step(1)
        ctx.set_spins(keep)
        ctx.step(2)
        out.append(state(ctx))
        ctx.close()
    for o in out:
        o.pop("E")
    same(out[0], out[1])
    same(out[0], out[2])
    a = hsg.Context(samples, 2, 3, precision=precision)
    b = hsg.Context(samples, 2, 3, precision=precision)
    a.sweep_hb(2)
    a.sweep_or(3)
    for _ in range(2):
        b.sweep_hb(1)      # (decodes anew in each call)
    for _ in range(3):
        b.sweep_or(1)
    same({"s": np.concatenate([s.ravel() for s in a.get_spins()])},
         {"s": np.concatenate([s.ravel() for s in b.get_spins()])})


@pytest.mark.parametrize("T", [8.0, 100.0, 1e5, 1e9])
def test_heat_bath_hemispheres_at_small_a(T):
    """One heat-bath sweep where beta |h| is below 0.35 (from about it down to 1e-9):
    both hemispheres take half of the draws.  Each component within the one-sweep
    bound of 1e-5 of the oracle."""
    smp = inputs.small_sample(16, n_temps=1, h_r=0.1, disorder_seed=4, t_min=T)
    smp = inputs.Sample(L=16, J=smp.J.astype(np.float32).astype(np.float64),
                        H=smp.H.astype(np.float32).astype(np.float64), temps=smp.temps)
    ctx = hsg.Context([smp], 8, 5)
    orc = oracle.OracleSim([smp], 8, 5)
    orc.samples[0].s = ctx.get_spins()[0].astype(np.float64)
    ctx.sweep_hb(1)
    orc.sweep_hb(1)
    assert np.abs(ctx.get_spins()[0] - orc.spins()[0]).max() < 1e-5
    ctx.close()


@pytest.mark.parametrize("Ls,n_temps,precision,j16", [
    ((128,), 5, "fp32", False), ((128,), 5, "fp32", True), ((128,), 5, "fp16", False), ((128,), 9, "bf16", True),
    ((64, 64), 3, "bf16", False), ((32, 64), 3, "fp32", False), ((32, 64), 3, "fp16", True), ((32,), 9, "fp16", False)])
def test_staged_half_sweeps(Ls, n_temps, precision, j16):
    """Staged over-relaxation half-sweeps (L / 2 of 64 and 32 in constants, any other
    and mixed lattices at run time), odd and even numbers of chunk groups per block:
    the same bits as half-sweeps that load into registers, energies included."""
    samples = [inputs.small_sample(L, n_temps=n_temps, disorder_seed=L + k) for k, L in enumerate(Ls)]
    out = []
    for kernel in (hsg.SWEEP_HALF, hsg.SWEEP_STAGED):
        ctx = hsg.Context(samples, 1, 5, precision=precision, j_fp16=j16, variant=hsg.VARIANT_TWO_PASS,
                          sweep_kernel=kernel)
        assert ctx.info().sweep_kernel == kernel
        ctx.step(1)
        out.append(state(ctx))
        ctx.close()
    same(out[0], out[1])


@pytest.mark.parametrize("scale", [0.0, 1e-22, 1e-20, 4e-20, 1e-19, 1.0, 1e18, 3e18, 1e19, 1e20])
def test_staged_move_at_extreme_fields(scale):
    """Fields whose squares are zero, subnormal, at the edges of the normal numbers and
    infinite: the staged move, which takes a shorter way for normal squares, gives the
    spins of the plain half-sweep."""
    base = inputs.small_sample(32, n_temps=2, disorder_seed=7)
    smp = inputs.Sample(L=32, J=np.asarray(base.J) * scale, H=None, temps=base.temps)
    out = []
    for kernel in (hsg.SWEEP_HALF, hsg.SWEEP_STAGED):
        ctx = hsg.Context([smp], 2, 5, variant=hsg.VARIANT_TWO_PASS, sweep_kernel=kernel)
        ctx.sweep_or(2)
        out.append(np.concatenate([s.ravel() for s in ctx.get_spins()]))
        ctx.close()
    np.testing.assert_array_equal(out[0], out[1])
