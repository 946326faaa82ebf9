"""A stage stores the primitives of the state it writes.  At every degree (even,
odd with the double-float lifting's pairs, and with FP64 lifting) steps must
equal, bitwise, stages whose primitives are formed afresh: after dg_set_state of
the same values, and in a caller's own graph, captured when the stored
primitives were valid and replayed after another state."""
import pytest

from paper_2606_18927_gb300 import dg, inputs as I
from gpu_helpers import torch_cuda

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,double_float,vol", [(1, True, 0), (2, True, 0), (3, True, 0), (4, True, 2), (7, True, 0),
                                                (7, False, 0), (5, True, 2), (8, True, 0)])
def test_steps_equal_fresh_primitives(N, double_float, vol):
    torch = torch_cuda()
    wl = I.workload("tgv_sine_n7_48", N=N, elems=(3, 2, 3))
    x, w = dg.lgl_nodes(N)
    X = I.node_coordinates(wl.spec, x)
    nbr = I.connectivity(wl.spec)
    d0 = torch.from_numpy(I.initial_state(wl, X)).cuda()
    d1 = torch.from_numpy(I.perturb(d0.cpu().numpy(), rel=1e-2, seed=3)).cuda()
    stream = torch.cuda.Stream()
    torch.cuda.synchronize()

    def make():
        op = dg.Operator(N, X, nbr, wl.phys, vol_flux=vol, surf_flux=wl.surf_flux)
        op.set_stream(stream)
        if N % 2 and not double_float:
            op.set_lifting_arithmetic(0)
        return op

    def state(op):
        out = torch.empty_like(d0)
        op.get_state(out)
        torch.cuda.synchronize()
        return out

    a = make()
    dt = a.time_step(0.5, d0)
    a.set_state(d0)
    a.rk_steps(0.0, dt, 2)
    ref = state(a)

    b = make()  # a fresh state before the second step
    b.set_state(d0)
    b.rk_steps(0.0, dt, 1)
    mid = state(b)
    b.set_state(mid)
    b.rk_steps(dt, dt, 1)
    assert torch.equal(state(b), ref)

    c = make()
    c.set_state(d1)
    c.rk_steps(0.0, dt, 1)
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=stream):
        c.rk_steps(0.0, dt, 1)
    c.set_state(d0)
    with torch.cuda.stream(stream):
        graph.replay()
        graph.replay()
    assert torch.equal(state(c), ref)
    c.set_state(d0)
    c.rk_steps_graph(0.0, dt, 2)
    assert torch.equal(state(c), ref)
    for op in (a, b, c):
        op.check_status()
        op.close()
