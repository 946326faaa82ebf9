"""Device memory of a context: a mesh that filled the device before the fixed-point
kernels still does.  Bytes of the state, metrics, lifting and scratch arrays per node
and per face node, without fixed-point copies of the metrics (N = 7 keeps some, where
it kept the pairs' metric sums, 252 bytes a node, before; meshes below 2^20 nodes do) and
without an array of its own for the adjoint's volume part."""
import pytest

from paper_2606_18927_gb300 import dg, inputs as I
from gpu_helpers import torch_cuda

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,side", [(4, 21), (5, 17), (7, 13)])
def test_bytes_of_a_context(N, side):
    torch = torch_cuda()
    spec, phys = I.BoxSpec(N, side, side, side), I.phys_params(Ma=0.3, Re=1600.0)
    X, nbr = I.node_coordinates(spec, dg.lgl_nodes(N)[0]), I.connectivity(spec)
    nodes, faces = spec.dofs, 6 * spec.K * (N + 1) ** 2  # (elements' face nodes)
    per_node = 4 * 40 + 72 + 8 + 32 + 56 + 72 + 48       # states, Ja, 1/J, R_v, primitives, Ja/J, (Ja Ja^T)/J
    per_node += (192 + 32) if N % 2 else 0               # the double-float lifting's pairs
    per_node += 252 if N == 7 else 0
    budget = per_node * nodes + (32 + 20 + 16) * faces   # viscous flux; surface flux and geometry per face
    torch.cuda.synchronize()
    U = torch.ones((5, spec.K, (N + 1) ** 3), dtype=torch.float64, device="cuda")
    U[4] = 10.0
    lam, gU = torch.ones_like(U), torch.ones_like(U)
    torch.cuda.empty_cache()
    free = torch.cuda.mem_get_info()[0]
    op = dg.Operator(N, X, nbr, phys, surf_flux=2)
    used = free - torch.cuda.mem_get_info()[0]
    op.vjp(lam, gU, U)
    torch.cuda.synchronize()
    with_vjp = free - torch.cuda.mem_get_info()[0]
    slack = 32 * 2 ** 21  # every array is a whole number of 2 MiB pages
    print(N, nodes, used / nodes, budget / nodes, with_vjp / nodes, slack / nodes)
    assert used <= budget + slack
    assert with_vjp <= budget + slack + (40 + 32 + 32) * faces
    op.close()
