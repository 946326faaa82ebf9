"""Elements with sides far apart, as boundary-layer meshes have them: the volume
term in fixed point keeps FP64's accuracy whatever the ratio of the sides.

Stretching a box by a power of two along an axis, with the velocity along it,
scales the contravariant velocities u . Ja^d, the Jacobian and so the mass row of
the volume term by powers of two and leaves its density alone: the units follow, and
the nodes inside the elements (no face fluxes) get the same bits at every ratio.

The rows against the extended oracle, with a bound on the rounding of FP64: 8
roundings, of half an ulp each, of the terms of a pair flux, in the square mean over
independent terms (m_c Ja_c, m_c Ja_c u_k, p Ja_k as p' is recovered to an ulp of p,
m_c Ja_c h, with the nodes' own values)."""
import numpy as np
import pytest

from paper_2606_18927_gb300 import dg, inputs as I
from gpu_helpers import gpu_ut, torch_cuda

pytestmark = pytest.mark.gpu


def stretched_case(N, ratio, phys, xi, along=True):
    """Box with sides 2 pi (1, 1 / ratio[1], 1 / ratio[2]) and a flow whose velocities follow the sides."""
    L = [2 * np.pi / r for r in ratio]
    spec = I.BoxSpec(N, 3, 2, 2, lengths=tuple(L))
    X = I.node_coordinates(I.BoxSpec(N, 3, 2, 2), xi)
    x, y, z = X
    s = [1.0 / r if along else 1.0 for r in ratio]
    rho = 1.0 + 0.03 * np.cos(x + y) + 0.01 * np.sin(z)
    u = s[0] * (np.sin(x) * np.cos(y) + 0.3)
    v = s[1] * (0.4 - np.cos(x) * np.sin(y))
    w = s[2] * 0.5 * np.cos(z - x)
    p = phys["p0"] + 0.02 * np.cos(2 * x) * np.sin(y)
    m = [rho * c * (1.0 + e) for c, e in zip((u, v, w), I.uniform(3 * x.size, -1e-4, 1e-4).reshape(3, *x.shape))]
    E = p / (phys["gamma"] - 1.0) + 0.5 * sum(c * c for c in m) / rho
    U = np.ascontiguousarray(np.stack([rho] + m + [E]))
    return spec, np.ascontiguousarray(X / np.array(ratio)[:, None, None]), U


def inner(N):
    n = N + 1
    i = np.arange(n ** 3)
    ijk = np.stack([i % n, i // n % n, i // n // n])
    return ((ijk > 0) & (ijk < N)).all(0)


@pytest.mark.parametrize("N", [2, 3, 4, 7])
@pytest.mark.parametrize("vol", [0, 1, 2])
def test_mass_row_keeps_its_bits(ora, vol, N):
    torch = torch_cuda()
    phys = I.phys_params(Ma=0.3, Re=1600.0, inviscid=True)
    xi = ora.lgl(N)[0]
    rows = []
    for ratio in ((1, 8, 1), (1, 256, 8), (64, 1, 1024), (16, 16, 1)):
        spec, X, U = stretched_case(N, ratio, phys, xi)
        g = dg.Operator(N, X, I.connectivity(spec), phys, vol_flux=vol, surf_flux=2, viscous=0)
        rows.append(gpu_ut(torch, g, U)[0][:, inner(N)])
        g.close()
    for r in rows[1:]:
        print(vol, N, np.abs(r - rows[0]).max() / np.abs(rows[0]).max())
        # (the states differ in the energy alone: its recovery does not touch rho and u)
        assert np.array_equal(r, rows[0])


@pytest.mark.parametrize("along", [True, False])
@pytest.mark.parametrize("ratio", [(1, 3, 1), (1, 30, 1), (1, 300, 30), (300, 1, 300)])
@pytest.mark.parametrize("vol,N", [(0, 3), (0, 4), (0, 7), (1, 4), (2, 3), (2, 7)])
def test_rows_against_the_extended_oracle(ora, vol, N, ratio, along):
    torch = torch_cuda()
    phys = I.phys_params(Ma=0.3, Re=1600.0, inviscid=True)
    x, w, D = ora.lgl(N)
    n = N + 1
    spec, X, U = stretched_case(N, ratio, phys, x, along)
    nbr = I.connectivity(spec)
    g = dg.Operator(N, X, nbr, phys, vol_flux=vol, surf_flux=2, viscous=0)
    a = gpu_ut(torch, g, U)
    ref = ora.Oracle(N, X, nbr, phys, vol_flux=vol, surf_flux=2, viscous=0, extended=True).time_derivative(U)
    Ja, J = g.metrics()
    r, m, E = U[0], U[1:4], U[4]
    p = (phys["gamma"] - 1.0) * (E - 0.5 * (m * m).sum(0) / r)
    terms = np.zeros((5,) + r.shape)  # squares of the node's flux terms, summed over the directions
    for d in range(3):
        for c in range(3):
            q = (m[c] * Ja[:, :, d, c]) ** 2  # products m_c Ja^d_c
            terms[0] += q
            terms[4] += q * ((E + p) / r) ** 2
            for k in range(3):
                terms[1 + k] += q * (m[k] / r) ** 2
        for k in range(3):
            terms[1 + k] += (p * Ja[:, :, d, k]) ** 2
    D2 = (4.0 * D * D).sum(1).max()
    sel = np.tile(inner(N), (spec.K, 1))
    for v in range(5):
        bound = np.sqrt(8.0 * D2) * 2.0 ** -54 * np.sqrt(terms[v].mean(axis=1, keepdims=True).max()) / J.min()
        e = np.sqrt(((a[v] - ref[v])[sel] ** 2).mean())
        print(vol, N, ratio, v, "%.2e %.2e" % (e, bound))
        assert e <= bound


@pytest.mark.parametrize("N,grade", [(4, 0.88), (7, 0.88), (7, 0.98)])
def test_elements_thin_at_one_end(ora, N, grade):
    """y graded 16 : 1 (99 : 1) along the elements, a flow across it: the lines at the thin
    end have their own, small, fluxes.  The bound above, line by line."""
    torch = torch_cuda()
    phys = I.phys_params(Ma=0.3, Re=1600.0, inviscid=True)
    x, w, D = ora.lgl(N)
    n = N + 1
    spec, X, U = stretched_case(N, (1, 1, 1), phys, x)
    X[1] += grade * np.sin(X[1])
    X = np.ascontiguousarray(X)
    U[2] *= 1e-3
    nbr = I.connectivity(spec)
    g = dg.Operator(N, X, nbr, phys, surf_flux=2, viscous=0)
    a = gpu_ut(torch, g, U)
    ref = ora.Oracle(N, X, nbr, phys, vol_flux=0, surf_flux=2, viscous=0, extended=True).time_derivative(U)
    Ja, J = g.metrics()
    D2 = (4.0 * D * D).sum(1).max()
    total = np.zeros(U[0].shape)
    for d in range(3):
        q = sum((U[1 + c] * Ja[:, :, d, c]) ** 2 for c in range(3)).reshape(-1, n, n, n)
        total += np.broadcast_to(q.mean(axis=3 - d, keepdims=True), q.shape).reshape(total.shape)
    bound = np.sqrt(8.0 * D2 * total) * 2.0 ** -54 / J
    sel = np.tile(inner(N), (spec.K, 1))
    e = np.sqrt((((a[0] - ref[0]) / bound)[sel] ** 2).mean())
    print(N, grade, e)
    assert e <= 1.0
