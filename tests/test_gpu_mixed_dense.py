"""The FP32-mixed kernels' two register budgets (dense_mesh): a flow that repeats
along x on a mesh of many periods takes the dense kernels, one period the others.
Both are within the form's 1e-5 (relative L2) of the exact operator, so within
2e-5 of each other in every period, at each degree and for both fluxes."""
import numpy as np
import pytest

from paper_2606_18927_gb300 import dg, inputs as I
from gpu_helpers import torch_cuda

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N", range(1, 9))
@pytest.mark.parametrize("vol", [dg.VOL_KEP_PIROZZOLI, dg.VOL_EC_CHANDRASHEKAR])
def test_periods_agree(N, vol):
    torch = torch_cuda()
    ey = ez = 6 if N < 4 else 4
    # more elements per SM than five and than twice the CTAs of 819 threads
    periods = 152 * max(5, 2 * 819 // (N + 1) ** 3) // (3 * ey * ez) + 2
    phys = I.phys_params(Ma=0.1, Re=1600.0)
    x, w = dg.lgl_nodes(N)
    out = []
    for m in (1, periods):
        spec = I.BoxSpec(N, 3 * m, ey, ez, lengths=(2 * np.pi * m, 2 * np.pi, 2 * np.pi))
        X = I.node_coordinates(spec, x)
        g = dg.Operator(N, X, I.connectivity(spec), phys, vol_flux=vol, surf_flux=2, precision=dg.FP32_MIXED)
        U = torch.from_numpy(I.taylor_green(X, phys)).cuda()
        Ut = torch.empty_like(U)
        g.time_derivative(Ut, U)
        torch.cuda.synchronize()
        g.check_status()
        out.append(Ut.cpu().numpy().reshape(5, ez, ey, m, 3, -1))
    one, many = out[0], out[1]
    for v in range(5):
        ref = np.broadcast_to(one[v], many[v].shape)
        e = np.linalg.norm(many[v] - ref) / np.linalg.norm(ref)
        print(N, vol, v, "%.1e" % e)
        assert e <= 2e-5
