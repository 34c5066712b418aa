"""The packed formats' two buffers of decoded spins: the second one only saves time, so a
context works without it, and gives it back to an allocation that has to succeed."""
import numpy as np
import pytest

from paper_1204_6192_gb300 import hsg, inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _build():
    import __graft_entry__
    __graft_entry__.build()


def context(precision, **kw):
    samples = [inputs.small_sample(L, n_temps=6, disorder_seed=L) for L in (14, 20)]
    kw = {"variant": hsg.VARIANT_TWO_PASS, "sweep_kernel": hsg.SWEEP_HALF, **kw}
    return hsg.Context(samples, 2, 3, precision=precision, **kw)


def last_of_create(precision):
    """The number of the last allocation of hsg_create: the optional one."""
    for n in range(1, 200):
        try:
            ctx = context(precision, inject_alloc_fault=n)
        except hsg.HsgError as e:
            assert e.status == 2
            continue
        parities = ctx.info().decoded_parities
        ctx.close()
        return n, parities
    raise AssertionError("no context")


def run(ctx, between=lambda c: None):
    ctx.sweep_hb(1)
    ctx.sweep_or(3)
    ctx.step(2)
    between(ctx)
    ctx.set_active([0, 1])
    ctx.step(1)
    ctx.set_active(None)
    ctx.step(2)
    ctx.sweep_or(2)
    out = np.concatenate([s.ravel() for s in ctx.get_spins()]), ctx.last_energies(), ctx.get_perm()
    parities = ctx.info().decoded_parities
    ctx.close()
    return out, parities


@pytest.mark.parametrize("precision", ["angle16", "oct16", "yx4"])
def test_one_buffer_and_two_give_the_same_bits(precision):
    ref, parities = run(context(precision))
    assert parities == 2
    n, parities = last_of_create(precision)
    assert parities == 1
    out, parities = run(context(precision, inject_alloc_fault=n))
    assert parities == 1
    for a, b in zip(out, ref):
        np.testing.assert_array_equal(a, b)


@pytest.mark.parametrize("when", ["before the first step", "between steps", "by the tuner"])
def test_second_buffer_gives_way_to_a_later_allocation(when):
    """The first allocation after hsg_create fails once: that of get_spins (before a step
    was captured, or after), or of the tuner's copy of the spins."""
    kw = {"variant": hsg.VARIANT_AUTO, "sweep_kernel": hsg.SWEEP_AUTO} if when == "by the tuner" else {}
    ref, parities = run(context("oct16", **kw))
    assert parities == 2
    n, _ = last_of_create("oct16")
    ctx = context("oct16", inject_alloc_fault=n + 1, **kw)
    assert ctx.info().decoded_parities == 2
    if when == "before the first step":
        ctx.get_spins()
        assert ctx.info().decoded_parities == 1
    out, parities = run(ctx, (lambda c: c.get_spins()) if when == "between steps" else lambda c: None)
    assert parities == 1
    for a, b in zip(out, ref):
        np.testing.assert_array_equal(a, b)


def test_second_buffer_stays_for_a_graph_of_the_callers():
    """Sweeps that the caller captured on its stream refer to both buffers: replays give
    the sweeps' spins, and an allocation that fails afterwards is an error."""
    import ctypes

    import torch
    rt = ctypes.CDLL("libcudart.so.13")
    for name, args in (("BeginCapture", [ctypes.c_void_p, ctypes.c_int]),
                       ("EndCapture", [ctypes.c_void_p, ctypes.POINTER(ctypes.c_void_p)])):
        getattr(rt, "cudaStream" + name).argtypes = args
    rt.cudaGraphInstantiate.argtypes = [ctypes.POINTER(ctypes.c_void_p), ctypes.c_void_p, ctypes.c_ulonglong]
    rt.cudaGraphLaunch.argtypes = [ctypes.c_void_p, ctypes.c_void_p]
    n, _ = last_of_create("oct16")
    stream = torch.cuda.Stream()
    ctx = context("oct16", stream=stream.cuda_stream, inject_alloc_fault=n + 3)
    plain = context("oct16")
    ctx.get_spins()
    assert rt.cudaStreamBeginCapture(stream.cuda_stream, 1) == 0
    ctx.sweep_or(2)
    graph, exe = ctypes.c_void_p(), ctypes.c_void_p()
    assert rt.cudaStreamEndCapture(stream.cuda_stream, ctypes.byref(graph)) == 0
    assert rt.cudaGraphInstantiate(ctypes.byref(exe), graph, 0) == 0
    for _ in range(2):
        assert rt.cudaGraphLaunch(exe, stream.cuda_stream) == 0
    plain.sweep_or(4)
    for a, b in zip(ctx.get_spins(), plain.get_spins()):
        np.testing.assert_array_equal(a, b)
    with pytest.raises(hsg.HsgError) as err:
        ctx.measure()
    assert err.value.status == 2
    torch.cuda.synchronize()
    ctx.close()
    plain.close()
