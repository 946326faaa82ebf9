"""Limb sums at their bounds (volume_fx.cuh, adjoint_fx.cuh).  Numbers just below
a power of two whose low limbs are near 2^30 make the cross products of the
three-term sums u . Ja, mu . u and mu . Ja as large as they can get: 9/8 and 12/8
of what 64 bits hold, were they added up in one accumulator.  The mesh is a
lattice of parallelepipeds with Ja^xi = a (1, 1, 1), a = 1 - 2^-29 - 2^-45, the
velocity u = v = w = 1 - 2^-30 - 2^-46.

Bounds: a uniform state's Ut is that of the mesh's rounded nodes (the extended
oracle's) but for some four roundings of a flux (the energy's, 3 rho h u, is the
largest) in each of the pairs, weighted 2 |D|, and at the faces, weighted 1 / w_0.  (Low
degrees: the limbs do not depend on it, the rounding of the metrics grows with it.)
The adjoint against all of the oracle's
columns: 1e-12 of the largest value (FP64 sums of some tens of terms)."""
import numpy as np
import pytest

from paper_2606_18927_gb300 import dg, inputs as I
from gpu_helpers import gpu_ut, torch_cuda

pytestmark = pytest.mark.gpu


def lattice(N, xi):
    spec = I.BoxSpec(N, 2, 2, 2, lengths=(4.0, 4.0, 4.0))
    s = I.node_coordinates(spec, xi)
    a = 1.0 - 2.0 ** -29 - 2.0 ** -45
    axes = ((0.25, 0.25, 0.25), (1.0, -1.0, 0.0), (0.0, a, -a))
    return spec, np.ascontiguousarray(sum(np.array(v)[:, None, None] * s[d] for d, v in enumerate(axes)))


def state(X, phys):
    u = 1.0 - 2.0 ** -30 - 2.0 ** -46
    return I.free_stream(X, phys, velocity=(u, u, u))


@pytest.mark.parametrize("N", [1, 2, 3])
@pytest.mark.parametrize("vol", [0, 1, 2])
def test_free_stream_at_the_limbs_bounds(ora, vol, N):
    torch = torch_cuda()
    phys = I.phys_params(Ma=0.3, Re=1600.0)
    spec, X = lattice(N, ora.lgl(N)[0])
    g = dg.Operator(N, X, I.connectivity(spec), phys, vol_flux=vol, surf_flux=2)
    Ja, J = g.metrics()
    assert np.abs(Ja[:, :, 0] - (1.0 - 2.0 ** -29)).max() < 2.0 ** -44
    U = state(X, phys)
    ref = ora.Oracle(N, X, I.connectivity(spec), phys, vol_flux=vol, surf_flux=2, extended=True).time_derivative(U)
    e = np.abs(gpu_ut(torch, g, U) - ref).max()
    x, w, D = ora.lgl(N)
    flux = 3.0 * (U[4, 0, 0] + phys["p0"])
    bound = 4.0 * 2.0 ** -53 * flux * (2.0 * np.abs(D).sum(1).max() + 1.0 / w[0]) / J.min()
    print(vol, N, e, bound)
    assert bound < 2e-11 and e <= bound


@pytest.mark.parametrize("signs", [(1, 1, 1), (1, -1, 1)])
def test_adjoint_at_the_limbs_bounds(ora, signs):
    torch = torch_cuda()
    phys = I.phys_params(Ma=0.3, Re=1600.0)
    spec, X = lattice(1, ora.lgl(1)[0])
    nbr = I.connectivity(spec)
    g = dg.Operator(1, X, nbr, phys, surf_flux=1)
    o = ora.Oracle(1, X, nbr, phys, vol_flux=0, surf_flux=1, viscous=1, extended=True)
    U = state(X, phys)
    J = g.metrics()[1]
    p = np.arange(8)
    turn = (-1.0) ** (p % 2 + p // 2 % 2 + p // 4)  # neighbours on every line differ in sign
    lam = np.zeros(U.shape)
    for c in range(3):
        lam[1 + c] = signs[c] * turn[None, :] * (1.0 - 2.0 ** -50) * J
    out = torch.empty(U.shape, dtype=torch.float64, device="cuda")
    g.vjp(torch.from_numpy(lam).cuda(), out, torch.from_numpy(U).cuda())
    got, ref = out.cpu().numpy().ravel(), np.zeros(U.size)
    d = np.zeros(U.size)
    for c in range(U.size):
        d[c] = 1.0
        ref[c] = (lam * o.jvp(U, d.reshape(U.shape))[1]).sum()
        d[c] = 0.0
    e = np.abs(got - ref).max() / np.abs(ref).max()
    print(signs, e)
    assert e <= 1e-12
