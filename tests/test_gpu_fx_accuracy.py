"""The fixed-point volume term against the FP64 passes it stands in for: the error of
every row (2-norm over the nodes inside the elements and over several states, against
the extended oracle) is at most a tenth above FP64's, up to the density contrast at
which an element is summed in FP64.  The FP64 passes run on the same mesh in units of
2^-100 of its size: its metrics, 2^200 times as large, are out of the fixed-point
range, and Ut scales by 2^-100, exactly."""
import numpy as np
import pytest

from paper_2606_18927_gb300 import dg, inputs as I
from gpu_helpers import gpu_ut, torch_cuda
from test_gpu_stretched import inner

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N", [3, 4, 7])
@pytest.mark.parametrize("vol,contrast", [(0, 0.1), (0, 1.2), (0, 1.7), (0, 1.95), (1, 1.2), (1, 1.7), (2, 0.02)])
def test_rows_are_as_good_as_fp64(ora, vol, contrast, N):
    torch = torch_cuda()
    phys = I.phys_params(Ma=0.3, Re=1600.0, inviscid=True)
    spec = I.BoxSpec(N, 2, 2, 2, geometry="sine", amplitude=0.1)
    X = I.node_coordinates(spec, ora.lgl(N)[0])
    nbr = I.connectivity(spec)
    a = dg.Operator(N, X, nbr, phys, vol_flux=vol, surf_flux=2, viscous=0)
    b = dg.Operator(N, X * 2.0 ** 100, nbr, phys, vol_flux=vol, surf_flux=2, viscous=0)
    o = ora.Oracle(N, X, nbr, phys, vol_flux=vol, surf_flux=2, viscous=0, extended=True)
    x, y, z = X
    # the density falls from one end of every element to the other (a step between elements in x)
    s = (x / np.pi) % 1.0
    e = np.zeros((2, 5))
    for seed in range(6):
        rho = np.exp(contrast * (s - 0.5)) * (1.0 + 0.01 * np.cos(y + z + seed))
        u = np.sin(x + seed) * np.cos(y) + 0.3
        v = 0.4 - np.cos(x) * np.sin(y + seed)
        w = 0.5 * np.cos(z - x)
        p = phys["p0"] + 0.2 * np.cos(2 * x) * np.sin(y)
        U = I.perturb(I.conservative(rho, u, v, w, p, phys["gamma"]), rel=1e-4, seed=seed)
        ref = o.time_derivative(U)[:, :, inner(N)]
        for k, (g, f) in enumerate(((a, 1.0), (b, 2.0 ** 100))):
            e[k] += ((gpu_ut(torch, g, U)[:, :, inner(N)] * f - ref) ** 2).sum(axis=(1, 2))
    r = np.sqrt(e[0] / e[1])
    print(vol, N, contrast, ["%.3f" % q for q in r])
    assert r.max() <= 1.1, r
