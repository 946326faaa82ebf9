"""Cotangents far below one: the adjoint is linear down to FP64's own range, for all
equations together and for one alone beside zeros.  Scaled by a power of two the
result is that of the unscaled cotangent to FP64 rounding of two summation orders
(1e-13 of the largest value; 2^-150 stays in fixed point, 2^-230 and 2^-300 do not)."""
import numpy as np
import pytest

from paper_2606_18927_gb300 import dg, inputs as I
from gpu_helpers import torch_cuda
from test_gpu_adjoint_fx import cotangent, operator, vjp
from test_gpu_stretched import inner, stretched_case

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N", [2, 7])
@pytest.mark.parametrize("kind", ["all", "mass", "momentum", "energy", "energy small", "mass small"])
@pytest.mark.parametrize("power", [-150, -230, -300])
def test_small_cotangents(ora, N, kind, power):
    torch = torch_cuda()
    g, o, U = operator(ora, N)
    lam = cotangent(kind.split()[0] if "small" not in kind else "all", U.shape)
    if "small" in kind:  # one equation's cotangent small, the others' not: by linearity the sum of the parts
        one = np.zeros_like(lam)
        v = 4 if kind.startswith("energy") else 0
        one[v] = lam[v]
        rest = lam - one
        a = vjp(torch, g, U, rest) + vjp(torch, g, U, one) * 2.0 ** power
        b = vjp(torch, g, U, rest + one * 2.0 ** power)
    else:
        a, b = vjp(torch, g, U, lam), vjp(torch, g, U, lam * 2.0 ** power) * 2.0 ** -power
    e = [float(np.abs(a[v] - b[v]).max() / max(np.abs(a[v]).max(), 1e-300)) for v in range(5)]
    print(N, kind, power, ["%.1e" % x for x in e])
    assert max(e) <= 1e-13, e


def columns(ora, o, U, lam, cols):
    """(J^T lam)_c of the extended oracle, and the sum of the magnitudes it adds up."""
    g, scale, d = np.zeros(len(cols)), np.zeros(len(cols)), np.zeros(U.size)
    for k, c in enumerate(cols):
        d[c] = 1.0
        t = lam * o.jvp(U, d.reshape(U.shape))[1]
        d[c] = 0.0
        g[k], scale[k] = t.sum(), np.abs(t).sum()
    return g, scale


@pytest.mark.parametrize("N", [3, 5])
@pytest.mark.parametrize("contrast", [0.8, 1.9, 3.0, 6.0])
def test_density_contrast(ora, N, contrast):
    """A density that differs by e^contrast over an element: the gradients at its light nodes,
    divided by their own density, against the oracle's columns.  Bound: 4e-15 (some 36 roundings)
    of the magnitudes that a column adds up."""
    torch = torch_cuda()
    spec = I.BoxSpec(N, 2, 1, 1)
    phys = I.phys_params(Ma=0.3, Re=1600.0)
    X = I.node_coordinates(spec, ora.lgl(N)[0])
    x, y, z = X
    rho = np.exp(0.5 * contrast * np.cos(x))
    u = np.sin(x) * np.cos(y) + 0.3
    v = 0.4 - np.cos(x) * np.sin(y)
    w = 0.5 * np.cos(z - x)
    U = I.perturb(I.conservative(rho, u, v, w, phys["p0"] + 0.2 * np.cos(2 * x) * np.sin(y), phys["gamma"]), rel=1e-3)
    g = dg.Operator(N, X, I.connectivity(spec), phys, surf_flux=2)
    o = ora.Oracle(N, X, I.connectivity(spec), phys, vol_flux=0, surf_flux=2, viscous=1, extended=True)
    lam = I.random_direction(U.shape, 43)
    got = vjp(torch, g, U, lam).ravel()
    light = np.argsort(U[0].ravel())[: U[0].size // 6]
    cols = np.concatenate([v * U[0].size + light[v::5][:12] for v in range(5)])
    ref, scale = columns(ora, o, U, lam, cols)
    e = np.abs(got[cols] - ref) / scale
    print(N, contrast, e.max(), np.sqrt((e * e).mean()))
    assert e.max() <= 4e-15


def two_elements(ora, N, ratio, along):
    """Two of the twelve elements of the stretched box, joined in x, between outflow boundaries."""
    phys = I.phys_params(Ma=0.3, Re=1600.0, inviscid=True)
    spec, X, U = stretched_case(N, ratio, phys, ora.lgl(N)[0], along)
    X, U = (np.ascontiguousarray(a.reshape(-1, 12, (N + 1) ** 3)[:, :2]) for a in (X, U))
    nbr = np.full((2, 6), -3, dtype=np.int32)
    nbr[0, 1], nbr[1, 0] = 1, 0
    return dict(phys, p_out=phys["p0"]), X, U, nbr


@pytest.mark.parametrize("N", [2, 3, 5, 7])
@pytest.mark.parametrize("ratio,along", [((1, 3, 1), True), ((1, 30, 1), True), ((1, 3, 1), False), ((1, 30, 1), False),
                                         ((1, 300, 30), False), ((300, 1, 300), False)])
def test_stretched_elements(ora, N, ratio, along):
    """Elements with sides far apart, with velocities along the sides or alike; sampled columns
    of the oracle, bound as above.  (Velocities 300 apart beside one pressure: FP64's recovery
    of p from the energy exceeds that bound, so they are in the next test.)"""
    torch = torch_cuda()
    phys, X, U, nbr = two_elements(ora, N, ratio, along)
    g = dg.Operator(N, X, nbr, phys, surf_flux=1, viscous=0)
    o = ora.Oracle(N, X, nbr, phys, vol_flux=0, surf_flux=1, viscous=0, extended=True)
    lam = I.random_direction(U.shape, 44)
    got = vjp(torch, g, U, lam).ravel()
    cols = np.concatenate([v * U[0].size + np.arange(3 + v, U[0].size, max(1, U[0].size // 10)) for v in range(5)])
    ref, scale = columns(ora, o, U, lam, cols)
    e = np.abs(got[cols] - ref) / scale
    print(N, ratio, along, e.max(), np.sqrt((e * e).mean()))
    assert e.max() <= 4e-15


@pytest.mark.parametrize("N", [2, 3, 5, 7])
def test_mass_cotangent_keeps_its_bits(ora, N):
    """Stretched by powers of two with the velocities along, the gradients of the mass row at the
    nodes inside the elements (volume terms alone) scale by powers of two: the same bits at every
    ratio, as in FP64."""
    torch = torch_cuda()
    rows = []
    for ratio in ((1, 8, 1), (1, 256, 8), (64, 1, 1024), (16, 16, 1)):
        phys, X, U, nbr = two_elements(ora, N, ratio, True)
        g = dg.Operator(N, X, nbr, phys, surf_flux=1, viscous=0)
        lam = np.zeros(U.shape)
        lam[0] = I.random_direction(U[0].shape, 45)
        r = vjp(torch, g, U, lam)[:4, :, inner(N)]
        rows.append(r / np.array((1.0,) + ratio)[:, None, None])
    for r in rows[1:]:
        print(N, np.abs(r - rows[0]).max() / np.abs(rows[0]).max())
        assert np.array_equal(r, rows[0])
