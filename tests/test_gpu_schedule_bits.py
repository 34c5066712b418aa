"""Every step schedule and over-relaxation kernel gives the same bits: the energies'
FP64 sums are taken in one order, and a move leaves the same spins down to the sign of
a zero component."""
import numpy as np
import pytest

from paper_1204_6192_gb300 import hsg, inputs

pytestmark = pytest.mark.gpu

HALF = {"variant": hsg.VARIANT_TWO_PASS, "sweep_kernel": hsg.SWEEP_HALF}
PERSISTENT = {"variant": hsg.VARIANT_PERSISTENT}


@pytest.fixture(scope="module", autouse=True)
def _build():
    import __graft_entry__
    __graft_entry__.build()


def energies(samples, replicas, kw, steps, **opt):
    """The energies after each of the steps, by sample and system."""
    ctx = hsg.Context(samples, replicas, 5, **{**opt, **kw})
    out = []
    for _ in range(steps):
        ctx.step(1)
        out.append(ctx.last_energies().copy())
    ctx.close()
    return np.stack(out)


def scattered(L, n_temps):
    """Random fields of 1e-8 to 1e8 from plane to plane: the blocks' and warps' sums then
    span more bits than binary64 holds, so every order of adding them rounds differently."""
    rng = np.random.default_rng(L)
    s = inputs.small_sample(L, n_temps=n_temps, disorder_seed=L)
    size = np.repeat(10.0 ** rng.uniform(-8, 8, L), L * L)[:, None]
    return inputs.Sample(L=L, J=s.J, H=rng.standard_normal((L ** 3, 3)) * size, temps=s.temps)


@pytest.mark.parametrize("Ls,precision", [((20,), "fp32"), ((32,), "fp32"), ((48,), "fp16"), ((64,), "fp32"), ((16, 64), "oct16")])
def test_energies_do_not_depend_on_the_schedule(Ls, precision):
    """One sum of splits at L = 20, 4 at L = 32, 13 at L = 48, 32 at L = 64: two-pass with
    any chunks per thread and passes, and the persistent schedule, to the last bit."""
    samples = [scattered(L, 12) for L in Ls]
    ways = [HALF, {**HALF, "chunks_per_thread": 1}, {**HALF, "chunks_per_thread": 5, "pass_bytes": 4 << 20},
            PERSISTENT, {**PERSISTENT, "chunks_per_thread": 2}]
    if precision != "oct16" and set(Ls) <= {32, 64}:
        ways += [{"variant": hsg.VARIANT_TWO_PASS, "sweep_kernel": hsg.SWEEP_STAGED},
                 {"variant": hsg.VARIANT_TWO_PASS, "sweep_kernel": hsg.SWEEP_WAVE}]
    E = [energies(samples, 2, kw, 2, precision=precision) for kw in ways]
    for kw, e in zip(ways[1:], E[1:]):
        np.testing.assert_array_equal(e, E[0], err_msg=str(kw))


@pytest.mark.parametrize("Ls,precision", [((12,), "fp32"), ((10,), "fp16"), ((8, 12, 4), "fp32"), ((12, 6), "yx4")])
def test_resident_energies_are_summed_in_the_same_order(Ls, precision):
    """The resident sweeps' energies against half-sweeps' and the persistent schedule's,
    to the last bit."""
    samples = [scattered(L, 7) for L in Ls]
    resident = {"variant": hsg.VARIANT_TWO_PASS}
    E = [energies(samples, 3, kw, 3, precision=precision) for kw in (HALF, resident, PERSISTENT)]
    np.testing.assert_array_equal(E[1], E[0])
    np.testing.assert_array_equal(E[2], E[0])


# unit vectors with zero components of both signs
UNITS = np.array([[1, 0, 0], [0, 1, 0], [0, 0, 1], [0.6, 0.8, 0], [0, -0.6, 0.8], [-0.8, 0, 0.6]])
UNITS = np.concatenate([UNITS, -UNITS, UNITS * np.where(UNITS == 0, -1, 1)])


def structured(L, kind, seed):
    """Couplings and fields among a few values, so that local fields vanish, lie along the
    axes, or stand at right angles to the spins up to tiny components."""
    rng = np.random.default_rng(seed)
    values = {"axes": [1.0, -1.0, 0.0, 0.5], "tiny": [1.0, -1.0, 0.0, 1e-20, -1e-30, 1e-38, -3e-39],
              "wide": [1.0, 1e-18, -1e17, 3e-25, 0.0, -2e-12]}[kind]
    J = rng.choice(values, (L ** 3, 3))
    H = UNITS[rng.integers(len(UNITS), size=L ** 3)] * rng.choice(values, (L ** 3, 1))
    spins = UNITS[rng.integers(len(UNITS), size=(6, L ** 3))]
    if kind == "axes":          # half of the systems ordered
        spins[::2] = UNITS[rng.integers(len(UNITS), size=3)][:, None]
    return inputs.Sample(L=L, J=J, H=H if seed % 2 else None, temps=np.array([0.5, 1.0, 2.0])), spins.astype(np.float32)


@pytest.mark.parametrize("seed", [0, 1])
@pytest.mark.parametrize("kind", ["axes", "tiny", "wide"])
@pytest.mark.parametrize("L,precision", [(8, "fp32"), (8, "fp16"), (32, "fp32"), (32, "fp16"),
                                         (32, "fp16j"), (32, "bf16"), (64, "fp32"), (64, "fp16")])
def test_moves_leave_the_same_bits(L, precision, kind, seed):
    """Spins and fields with zero components, zero, subnormal and far apart fields:
    over-relaxation by every kernel, and steps by every schedule, the sign of zeros
    included."""
    smp, spins = structured(L, kind, seed)
    ways = [HALF, PERSISTENT, {"variant": hsg.VARIANT_TWO_PASS, "sweep_kernel": hsg.SWEEP_FUSED},
            {"variant": hsg.VARIANT_TWO_PASS, "sweep_kernel": hsg.SWEEP_WAVE}]
    ways.append({"variant": hsg.VARIANT_TWO_PASS, "sweep_kernel": hsg.SWEEP_STAGED if L >= 32 else hsg.SWEEP_AUTO})
    out = []
    for kw in ways:
        ctx = hsg.Context([smp], 2, 5, precision=precision[:4], j_fp16=precision == "fp16j", n_hb=0, n_or=3, **kw)
        ctx.set_spins([spins])
        ctx.sweep_or(2)
        a = ctx.get_spins()[0].copy()
        ctx.step(1)
        out.append((a, ctx.get_spins()[0].copy()))
        ctx.close()
    for kw, o in zip(ways[1:], out[1:]):
        for x, ref in zip(o, out[0]):
            np.testing.assert_array_equal(x.view(np.uint32), ref.view(np.uint32), err_msg=str(kw))
