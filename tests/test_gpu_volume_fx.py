"""The FP64 volume term in fixed point (volume_fx.cuh) against the extended
oracle: every degree (lines that fill a warp and lines that do not), a state at
the edge of the common units (no reference pressure), and elements outside
their range (a large density contrast),
which are summed in FP64, alone and beside elements in range.

Bounds.  The volume sums are exact but for the rounding of the products, below
FP64's; what remains is the rest of the operator, held to 1e-12 as everywhere.
Without a reference pressure the FP64 face fluxes carry O(p0) terms whose
cancellation against the volume term leaves p0 2^-53 (1 / w_0) (2 / h) / |Ut|:
1e-10 at N = 7 (as for the oracle's own FP64 build)."""
import numpy as np
import pytest

from paper_2606_18927_gb300 import dg, inputs as I
from gpu_helpers import gpu_ut, parity_per_var, torch_cuda

pytestmark = pytest.mark.gpu


def build(ora, spec, phys, U_of, **opts):
    x, w, D = ora.lgl(spec.N)
    X = I.node_coordinates(spec, x)
    nbr = I.connectivity(spec)
    o = ora.Oracle(spec.N, X, nbr, phys, vol_flux=opts.get("vol_flux", 0), surf_flux=2, viscous=1, extended=True)
    g = dg.Operator(spec.N, X, nbr, phys, surf_flux=2, **opts)
    return o, g, U_of(X, phys)


def flow(speed=1.0, contrast=0.0):
    def U_of(X, phys):
        x, y, z = X
        rho = np.exp(contrast * np.sin(x)) * (1.0 + 0.02 * np.cos(y + z))
        u = speed * (np.sin(x) * np.cos(y) + 0.3)
        v = speed * (0.4 - np.cos(x) * np.sin(y))
        w = speed * 0.5 * np.cos(z - x)
        p = phys["p0"] + speed ** 2 * 0.2 * np.cos(2 * x) * np.sin(y)
        return I.perturb(I.conservative(rho, u, v, w, p, phys["gamma"]), rel=1e-4)
    return U_of


CASES = [(N, "flow", {}, {}, 1e-12) for N in range(1, 9)] + [
    (5, "no reference pressure", {}, dict(p_ref=0.0), 1e-10),
    (7, "no reference pressure", {}, dict(p_ref=0.0), 1e-10),
    (7, "density contrast in FP64", dict(contrast=2.5), {}, 2e-12),
    (4, "density contrast in FP64", dict(contrast=2.5), {}, 2e-12),
]
# entropy-conserving flux: in range while density and internal energy vary by
# less than an eighth over an element
EC_CASES = [(N, "flow", {}, {}, 1e-12) for N in (1, 2, 4, 5, 7, 8)] + [
    (7, "density steps", dict(contrast=0.02), {}, 1e-12),
    (5, "no reference pressure", {}, dict(p_ref=0.0), 1e-10),
    (7, "density contrast in FP64", dict(contrast=1.0), {}, 2e-12),
]

KG_CASES = [(N, "flow", {}, {}, 1e-12) for N in (1, 4, 7)] + [(5, "density contrast in FP64", dict(contrast=2.5), {}, 2e-12)]


@pytest.mark.parametrize("vol,N,label,state,phys_over,bound",
                         [(0,) + c for c in CASES] + [(2,) + c for c in EC_CASES] + [(1,) + c for c in KG_CASES],
                         ids=["kep n%d %s" % c[:2] for c in CASES] + ["ec n%d %s" % c[:2] for c in EC_CASES]
                         + ["kg n%d %s" % c[:2] for c in KG_CASES])
def test_fixed_point_volume_term(ora, vol, N, label, state, phys_over, bound):
    torch = torch_cuda()
    phys = dict(I.phys_params(Ma=0.3, Re=1600.0), **phys_over)
    o, g, U = build(ora, I.BoxSpec(N, 3, 2, 2, geometry="sine", amplitude=0.1), phys, flow(**state), vol_flux=vol)
    e = parity_per_var(gpu_ut(torch, g, U), o.time_derivative(U))
    print(N, label, ["%.1e" % x for x in e])
    assert max(e) <= bound, e


@pytest.mark.parametrize("vol", [0, 2])
def test_elements_in_and_out_of_range_side_by_side(ora, vol):
    torch = torch_cuda()
    phys = I.phys_params(Ma=0.3, Re=1600.0)
    o, g, U = build(ora, I.BoxSpec(5, 4, 2, 2), phys, flow(), vol_flux=vol)
    U = U.reshape(5, -1, 216)
    U[0, 3] *= np.exp(2.3 * np.linspace(-1.0, 1.0, 216))  # element 3: a contrast of 100
    U = np.ascontiguousarray(U)
    ref = o.time_derivative(U)
    e = parity_per_var(gpu_ut(torch, g, U), ref)
    print(["%.1e" % x for x in e])
    assert max(e) <= 2e-12, e


def test_non_finite_values_stay_on_their_lines(ora):
    """A NaN reaches the nodes of its own lines only, as in FP64."""
    torch = torch_cuda()
    phys = I.phys_params(Ma=0.3, Re=1600.0, inviscid=True)
    o, g, U = build(ora, I.BoxSpec(3, 3, 3, 3), phys, flow())
    op = dg.Operator(3, I.node_coordinates(I.BoxSpec(3, 3, 3, 3), ora.lgl(3)[0]), I.connectivity(I.BoxSpec(3, 3, 3, 3)),
                     phys, surf_flux=2, viscous=0)
    U = U.reshape(5, 27, 4, 4, 4)
    U[4, 13, 1, 2, 1] = np.nan
    Ut = torch.empty(U.size, dtype=torch.float64, device="cuda")
    op.time_derivative(Ut, torch.from_numpy(np.ascontiguousarray(U)).cuda().reshape(-1))
    bad = ~np.isfinite(Ut.cpu().numpy().reshape(5, 27, 4, 4, 4))
    want = np.zeros((4, 4, 4), dtype=bool)
    want[:, 2, 1] = want[1, :, 1] = want[1, 2, :] = True
    assert np.array_equal(bad[4, 13], want)
    assert not bad[0].any() and not bad[:, :13].any() and not bad[:, 14:].any()
