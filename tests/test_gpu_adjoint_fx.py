"""The KEP flux's transposed volume integral in fixed point (adjoint_fx.cuh):
every degree against the oracle's forward-mode derivative (the dot-product
identity, bound 1e-13: FP64 sums of some 1e4 terms of either sign), cotangents
of one equation alone or on one node, whose parts lie in units far apart, and
cotangents so large that the elements are summed in FP64, against the scaled
result (the adjoint is linear: equal to FP64 rounding of two summation orders,
1e-13 of the largest value)."""
import numpy as np
import pytest

from paper_2606_18927_gb300 import dg, inputs as I
from gpu_helpers import tgv_with_offset, torch_cuda

pytestmark = pytest.mark.gpu


def operator(ora, N):
    spec = I.BoxSpec(N, 3, 2, 2, geometry="sine", amplitude=0.1)
    phys = I.phys_params(Ma=0.3, Re=1600.0)
    x, w, D = ora.lgl(N)
    X = I.node_coordinates(spec, x)
    nbr = I.connectivity(spec)
    U = I.perturb(tgv_with_offset(X, phys))
    return (dg.Operator(N, X, nbr, phys, surf_flux=2),
            ora.Oracle(N, X, nbr, phys, vol_flux=0, surf_flux=2, viscous=1, extended=True), U)


def vjp(torch, g, U, lam):
    out = torch.empty(U.shape, dtype=torch.float64, device="cuda")
    g.vjp(torch.from_numpy(np.ascontiguousarray(lam)).cuda(), out, torch.from_numpy(U).cuda())
    return out.cpu().numpy()


def cotangent(kind, shape):
    lam = I.random_direction(shape, 41)
    if kind == "mass":
        lam[1:] = 0.0
    elif kind == "momentum":
        lam[[0, 4]] = 0.0
    elif kind == "energy":
        lam[:4] = 0.0
    elif kind == "node":
        one = np.zeros_like(lam)
        one[:, 1, 5] = lam[:, 1, 5]
        lam = one
    elif kind == "apart":
        lam[0] *= 1e-9
        lam[4] *= 1e7
    return lam


@pytest.mark.parametrize("N,kind", [(N, "all") for N in range(1, 9)]
                         + [(7, k) for k in ("mass", "momentum", "energy", "node", "apart")] + [(4, "node")])
def test_dot_product_with_the_forward_derivative(ora, N, kind):
    torch = torch_cuda()
    g, o, U = operator(ora, N)
    lam, d = cotangent(kind, U.shape), I.random_direction(U.shape, 42)
    gU = vjp(torch, g, U, lam)
    _, dUt = o.jvp(U, d)
    lhs, rhs = float((lam * dUt).sum()), float((gU * d).sum())
    scale = float(np.abs(lam * dUt).sum())
    print(N, kind, lhs, rhs, abs(lhs - rhs) / scale)
    assert abs(lhs - rhs) <= 1e-13 * scale


@pytest.mark.parametrize("N", [2, 7])
def test_out_of_range_cotangents_in_fp64(ora, N):
    torch = torch_cuda()
    g, o, U = operator(ora, N)
    lam = cotangent("all", U.shape)
    a, big = vjp(torch, g, U, lam), vjp(torch, g, U, lam * 2.0 ** 300) * 2.0 ** -300
    e = [float(np.abs(a[v] - big[v]).max() / np.abs(a[v]).max()) for v in range(5)]
    print(N, ["%.1e" % x for x in e])
    assert 0.0 < max(e) <= 1e-13, e
