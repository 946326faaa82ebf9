"""dg_set_wall_solve_limit caps the evaluations of the law per wall node: a cold
FP64 solve that needs one more than the cap is reported, one that needs the cap is
not.  A uniform flow, in which every wall node has the same solve; its count from
the documented steps (bracket growth from the laminar estimate, then Newton)."""
import math

import numpy as np
import pytest

from paper_2606_18927_gb300 import dg, inputs as I
from gpu_helpers import torch_cuda

pytestmark = pytest.mark.gpu


def steps_needed(phys, u):
    """Bracket growth and Newton steps together, for Reichardt's law."""
    g, T, Pr = phys["gamma"], phys["p0"], phys["Pr"]
    cp = g / (g - 1.0)
    r = Pr ** (1.0 / 3.0)
    Tw = T + r * u * u / (2.0 * cp)
    a = math.sqrt(r / (2.0 * cp * Tw))
    lnRe = math.log(phys["hwm"] * (math.asin(a * u) / a) / (phys["mu"] * Tw / T))
    k, C = phys["kappa"], phys["B"] - math.log(phys["kappa"]) / phys["kappa"]

    def F(t):
        w = math.exp(t)
        e1, e2 = math.exp(-w / 11.0), math.exp(-0.33 * w)
        L = math.log1p(k * w) / k + C * (1.0 - e1 - (w / 11.0) * e2)
        dL = 1.0 / (1.0 + k * w) + C * (e1 / 11.0 - e2 / 11.0 + 0.33 * (w / 11.0) * e2)
        return t + math.log(L) - lnRe, 1.0 + w * dL / L

    t0 = 0.5 * lnRe
    lo, hi, it, st = t0, t0, 0, 1.0
    while not F(lo)[0] < 0.0:
        lo -= st; st *= 2.0; it += 1
    st = 1.0
    while not F(hi)[0] > 0.0:
        hi += st; st *= 2.0; it += 1
    t = t0 if lo < t0 < hi else 0.5 * (lo + hi)
    while True:
        f, d = F(t)
        it += 1
        if f == 0.0:
            return it
        lo, hi = (t, hi) if f < 0.0 else (lo, t)
        nt = t - f / d
        newton = lo <= nt <= hi
        nt = nt if newton else 0.5 * (lo + hi)
        step, t = abs(nt - t), nt
        if (newton and step <= 1e-12 * max(1.0, abs(t))) or hi - lo <= 2e-15 * max(1.0, abs(t)):
            return it


@pytest.mark.parametrize("Re", [500.0, 20000.0, 1e6])
def test_the_cap_counts_the_evaluations(Re):
    torch = torch_cuda()
    wl = I.workload("channel_n5", N=3, elems=(2, 4, 2))
    phys = dict(wl.phys, mu=1.0 / Re)
    X = I.node_coordinates(wl.spec, dg.lgl_nodes(3)[0])
    U = torch.from_numpy(I.free_stream(X, phys, velocity=(1.0, 0.0, 0.0))).cuda()
    need = steps_needed(phys, 1.0)
    out = torch.empty_like(U)
    got = []
    for cap in range(1, need + 4):
        op = dg.Operator(3, X, I.connectivity(wl.spec), phys, surf_flux=2, law=1)  # (no earlier solution)
        op.set_wall_solve_limit(cap)
        op.time_derivative(out, U)
        torch.cuda.synchronize()
        try:
            op.check_status()
            got.append(True)
        except dg.DGError:
            got.append(False)
        op.close()
    print(Re, need, got)
    assert got == [cap >= need for cap in range(1, need + 4)]
