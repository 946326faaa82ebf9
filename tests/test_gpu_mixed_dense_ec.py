"""The entropy-conserving FP32-mixed kernel on either side of the mesh size at which it
takes the dense register budget (14 elements per SM at N = 3, 3 at N = 5, 20 at N = 6, 5 at N = 7): one
period of a flow against many, as for the other kernels, bound 2e-5."""
import pytest

import numpy as np

from paper_2606_18927_gb300 import dg, inputs as I
from gpu_helpers import torch_cuda

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,per_sm", [(3, 14), (5, 3), (6, 20), (7, 5)])
def test_both_budgets(N, per_sm):
    torch = torch_cuda()
    phys = I.phys_params(Ma=0.1, Re=1600.0)
    xi = dg.lgl_nodes(N)[0]
    last = per_sm * 152 // 16  # elements in x of the largest mesh of the other budget (4 x 4 across)
    out = []
    for ex in (2, last // 2 * 2, last // 2 * 2 + 2):
        spec = I.BoxSpec(N, ex, 4, 4, lengths=(np.pi * ex, 2 * np.pi, 2 * np.pi))
        X = I.node_coordinates(spec, xi)
        g = dg.Operator(N, X, I.connectivity(spec), phys, vol_flux=dg.VOL_EC_CHANDRASHEKAR, surf_flux=2,
                        precision=dg.FP32_MIXED)
        U = torch.from_numpy(I.taylor_green(X, phys)).cuda()
        Ut = torch.empty_like(U)
        g.time_derivative(Ut, U)
        g.check_status()
        out.append(Ut.cpu().numpy().reshape(5, 16, ex // 2, 2, -1))
        g.close()
    for many in out[1:]:
        for v in range(5):
            ref = np.broadcast_to(out[0][v], many[v].shape)
            e = np.linalg.norm(many[v] - ref) / np.linalg.norm(ref)
            assert e <= 2e-5, (N, v, e)
