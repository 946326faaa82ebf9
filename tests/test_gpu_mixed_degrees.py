"""The FP32-mixed volume sums by line threads (volume_line.cuh): every degree
against the oracle (the form's bound, 1e-5 relative L2), and results written over
their input (the sums' storage must not be the state that the source term still
reads), bitwise the same as into an array of their own."""
import numpy as np
import pytest

from paper_2606_18927_gb300 import dg, inputs as I
from gpu_helpers import torch_cuda

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N", range(1, 9))
def test_every_degree_and_in_place(ora, N):
    torch = torch_cuda()
    spec = I.BoxSpec(N, 3, 2, 3, geometry="sine", amplitude=0.05)
    phys = I.phys_params(Ma=0.1, Re=1600.0, force=(0.3, -0.2, 0.1))
    x, w, D = ora.lgl(N)
    X = I.node_coordinates(spec, x)
    nbr = I.connectivity(spec)
    U = I.perturb(I.taylor_green(X, phys))
    o = ora.Oracle(N, X, nbr, phys, vol_flux=0, surf_flux=2, viscous=1, extended=True)
    g = dg.Operator(N, X, nbr, phys, surf_flux=2, precision=dg.FP32_MIXED)
    Ud = torch.from_numpy(U).cuda()
    Ut = torch.empty_like(Ud)
    g.time_derivative(Ut, Ud)
    both = Ud.clone()
    g.time_derivative(both, both)
    torch.cuda.synchronize()
    assert torch.equal(both, Ut)
    a, ref = Ut.cpu().numpy().reshape(5, -1), o.time_derivative(U).reshape(5, -1)
    e = [float(np.linalg.norm(a[v] - ref[v]) / np.linalg.norm(ref[v])) for v in range(5)]
    print(N, ["%.1e" % q for q in e])
    assert max(e) <= 1e-5, e
