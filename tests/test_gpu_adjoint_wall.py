"""The wall model in reverse mode (wall_stress_vjp): both laws at adiabatic and
isothermal walls, cooled and heated, with constant and Sutherland viscosity, at
degrees with fewer and with more planes than the kernel's warps and with wall
nodes that do not fill the last block, against the extended oracle's forward
derivative (dot products, the bounds of the adjoint's other tests)."""
import numpy as np
import pytest

from paper_2606_18927_gb300 import dg, inputs as I
from gpu_helpers import case, torch_cuda

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N", [2, 5, 8])
@pytest.mark.parametrize("law", [0, 1])
@pytest.mark.parametrize("wall,suth", [(0.0, False), (0.0, True), (0.9, False), (1.2, True)])
def test_state_and_parameters(ora, N, law, wall, suth):
    torch = torch_cuda()
    wl = I.workload("channel_n5", N=N, elems=(3, 4, 1) if N > 2 else (3, 4, 3))
    phys = dict(wl.phys)
    if wall:
        phys["T_wall"] = wall * phys["p0"] / phys["R"]
    if suth:
        phys.update(T_ref=phys["p0"] / phys["R"], suth_S=0.4 * phys["p0"] / phys["R"])
    o, g, X, U = case(ora, wl.spec, phys, surf_flux=2, law=law, ic="channel")
    lam = I.random_direction(U.shape, seed=21)
    Ud, ld = torch.from_numpy(U).cuda(), torch.from_numpy(np.ascontiguousarray(lam)).cuda()
    out = torch.empty_like(Ud)
    gth = torch.zeros(2, dtype=torch.float64, device="cuda")
    g.vjp(ld, out, Ud, gth)
    torch.cuda.synchronize()
    g.check_status()
    d = I.random_direction(U.shape, seed=22) * np.abs(U)
    _, Jd = o.jvp(U, d)
    a, b, sc = float((lam * Jd).sum()), float((out.cpu().numpy() * d).sum()), float(np.abs(lam * Jd).sum())
    print(N, law, wall, suth, "state %.1e" % (abs(a - b) / sc))
    assert abs(a - b) <= 1e-11 * sc
    for k, (dk, dB) in enumerate(((1.0, 0.0), (0.0, 1.0))):
        _, Jt = o.jvp(U, None, dk, dB)
        ref, sc = float((lam * Jt).sum()), float(np.abs(lam * Jt).sum())
        print("  parameter", k, "%.1e" % (abs(ref - float(gth[k])) / sc))
        assert abs(ref - float(gth[k])) <= 1e-10 * sc
