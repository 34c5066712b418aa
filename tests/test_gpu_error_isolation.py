"""A CUDA error that one call returns is reported there and nowhere else: contexts
created afterwards in the same thread work."""
import ctypes

import numpy as np
import pytest

from paper_1204_6192_gb300 import hsg, inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _build():
    import __graft_entry__
    __graft_entry__.build()


@pytest.mark.parametrize("call", ["energies", "measure", "get_perm", "sync"])
def test_error_of_a_refused_call_does_not_reach_the_next_context(call):
    """A call that synchronises is refused while the caller captures its stream."""
    import torch
    rt = ctypes.CDLL("libcudart.so.13")
    rt.cudaStreamBeginCapture.argtypes = [ctypes.c_void_p, ctypes.c_int]
    rt.cudaStreamEndCapture.argtypes = [ctypes.c_void_p, ctypes.POINTER(ctypes.c_void_p)]
    smp = inputs.small_sample(8, n_temps=4, disorder_seed=1)
    stream = torch.cuda.Stream()
    ctx = hsg.Context([smp], 2, 1, stream=stream.cuda_stream)
    torch.cuda.synchronize()
    assert rt.cudaStreamBeginCapture(stream.cuda_stream, 1) == 0    # (this thread's calls)
    with pytest.raises(hsg.HsgError) as err:
        getattr(ctx, call)()
    graph = ctypes.c_void_p()
    rt.cudaStreamEndCapture(stream.cuda_stream, ctypes.byref(graph))
    rt.cudaGetLastError()       # the capture's failure, in this runtime (torch's)
    assert err.value.status in (2, 3)      # (the allocation or the wait that is refused)
    ctx.close()
    out = []
    for _ in range(2):
        ctx = hsg.Context([smp], 2, 1)
        ctx.step(2)
        out.append(np.concatenate([s.ravel() for s in ctx.get_spins()]))
        ctx.sync()
        ctx.close()
    np.testing.assert_array_equal(out[0], out[1])
