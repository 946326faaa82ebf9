"""Stored primitives and a caller's own graphs.  A graph that the caller captured
writes the context's stored primitives, or its state, whenever it is replayed:
no later call may take what was stored before for the primitives of its state.
Steps after a replay equal, bitwise, those of a context without graphs."""
import pytest

from paper_2606_18927_gb300 import dg, inputs as I
from gpu_helpers import torch_cuda

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("captured", ["other state's time derivative", "set_state"])
@pytest.mark.parametrize("by_graph", [False, True], ids=["rk_steps", "rk_steps_graph"])
@pytest.mark.parametrize("N,precision", [(3, dg.FP64), (2, dg.FP64), (3, dg.FP32_MIXED)])
def test_steps_after_a_replay(N, precision, by_graph, captured):
    torch = torch_cuda()
    wl = I.workload("tgv_sine_n7_48", N=N, elems=(3, 2, 3))
    x, w = dg.lgl_nodes(N)
    X = I.node_coordinates(wl.spec, x)
    d0 = torch.from_numpy(I.initial_state(wl, X)).cuda()
    d1 = torch.from_numpy(I.perturb(d0.cpu().numpy(), rel=1e-2, seed=3)).cuda()
    stream = torch.cuda.Stream()
    torch.cuda.synchronize()

    def make():
        op = dg.Operator(N, X, I.connectivity(wl.spec), wl.phys, precision=precision, surf_flux=wl.surf_flux)
        op.set_stream(stream)
        return op

    def steps(op, count):
        (op.rk_steps_graph if by_graph else op.rk_steps)(0.0, dt, count)

    def state(op):
        out = torch.empty_like(d0)
        op.get_state(out)
        torch.cuda.synchronize()
        return out

    a = make()
    dt = a.time_step(0.5, d0)
    a.set_state(d0)
    steps(a, 1)
    if captured == "set_state":
        a.set_state(d1)
    steps(a, 2)

    b = make()
    b.set_state(d0)
    steps(b, 1)
    kept = state(b)
    graph = torch.cuda.CUDAGraph()
    out = torch.empty_like(d0)
    with torch.cuda.graph(graph, stream=stream):
        if captured == "set_state":
            b.set_state(d1)
        else:
            b.time_derivative(out, d1)
    b.set_state(kept)
    b.rk_steps(0.0, 0.0, 1)  # (dt = 0: the state stays, its primitives are stored)
    assert torch.equal(state(b), kept)
    with torch.cuda.stream(stream):
        graph.replay()
    steps(b, 1)
    with torch.cuda.stream(stream):
        if captured != "set_state":
            graph.replay()
    steps(b, 1)
    assert torch.equal(state(b), state(a))
    if captured != "set_state":
        ref = torch.empty_like(d0)
        a.time_derivative(ref, d1)
        torch.cuda.synchronize()
        assert torch.equal(out, ref)
    for op in (a, b):
        op.check_status()
        op.close()
