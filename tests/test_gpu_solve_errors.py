"""A solve that ends in an error: nothing is left running on its stream, and the workspace
solves again.  The reduction hook of a sharded workspace queues 50 ms of work behind the
slab's scoring and then reports a failure."""
import numpy as np
import pytest

from paper_2403_03571_gb300 import synth
from _gpu import host, instance_tensors, require_gpu, torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("fail_at", [1, 4])  # at the first evaluation, inside a line search
def test_the_stream_is_idle_after_an_error(fail_at):
    require_gpu()
    from paper_2403_03571_gb300 import capi, shard
    inst = synth.make_instance(3, 200, 24, 71)
    x, A, w0, v = instance_tensors(inst)
    o = capi.solve_opts(eps=0.05)
    calls = []

    def hook(ctx, mom_ptr, words, seeds, stream_ptr):
        calls.append(1)
        if len(calls) != fail_at:
            return 0
        with torch.cuda.stream(shard._stream_of(stream_ptr)):
            torch.cuda._sleep(100_000_000)
        return 1

    st = torch.cuda.Stream()
    st.wait_stream(torch.cuda.current_stream())
    ws = capi.Workspace(3, inst.n, inst.grid.num_pixels)
    ws.set_pruning(True)
    w = torch.zeros(inst.n, dtype=torch.float64, device="cuda")
    torch.cuda.synchronize()
    fn = capi.REDUCE_FN(hook)
    ws.set_shard(0, 2, fn)
    with pytest.raises(capi.ApdError) as e:
        capi.apd_solve_weights(inst.grid, x, A, w0, v, w, ws, o, stream=st)
    assert st.query()
    assert e.value.code == capi.APD_ERR_CUDA and len(calls) == fail_at
    ws.set_shard(0, 1)
    fresh = capi.Workspace(3, inst.n, inst.grid.num_pixels)
    fresh.set_pruning(True)
    want = torch.zeros_like(w)
    _, i0 = capi.apd_solve_weights(inst.grid, x, A, w0, v, want, fresh, o)
    _, i1 = capi.apd_solve_weights(inst.grid, x, A, w0, v, w, ws, o, stream=st)
    assert i0.evaluations == i1.evaluations
    assert np.array_equal(host(w), host(want))
