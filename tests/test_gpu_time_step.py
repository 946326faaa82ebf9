"""dg_time_step: the maximum over the nodes equals the FP64 formula on every
node, whatever the FP32 bounds that choose the nodes to evaluate: one node far
above the rest, all nodes alike, a node without a sound speed beside fast ones,
units in which FP32 under- or overflows; FP64 and FP32-mixed contexts.  The
bound is FP64 rounding of some twenty operations, 1e-14."""
import numpy as np
import pytest

from paper_2606_18927_gb300 import dg, inputs as I
from gpu_helpers import torch_cuda

pytestmark = pytest.mark.gpu


def formula(U, Ja, iJ, gamma):
    r, m, E = U[0].ravel(), U[1:4].reshape(3, -1), U[4].ravel()
    with np.errstate(all="ignore"):
        u = m / r
        c = np.sqrt(gamma * (gamma - 1.0) * (E - 0.5 * r * (u * u).sum(0)) / r)
        lam = sum(np.abs((Ja[:, d].T * u).sum(0)) + c * np.sqrt((Ja[:, d] ** 2).sum(1)) for d in range(3))
        return np.nanmax(lam * iJ)


@pytest.mark.parametrize("precision", [dg.FP64, dg.FP32_MIXED])
@pytest.mark.parametrize("case", ["flow", "one fast node", "uniform", "no sound speed", "tiny", "huge"])
def test_time_step_is_the_formula_s(case, precision):
    torch = torch_cuda()
    spec, phys = I.BoxSpec(3, 5, 4, 3, geometry="sine", amplitude=0.1), I.phys_params(Ma=0.3, Re=1600.0)
    x, w = dg.lgl_nodes(3)
    X = I.node_coordinates(spec, x)
    U = I.free_stream(X, phys) if case == "uniform" else I.perturb(I.taylor_green(X, phys))
    if case in ("one fast node", "no sound speed"):
        U[1, 7, 11] += 30.0
        U[4, 7, 11] += 450.5
    if case == "no sound speed":  # the largest finite value is another node's
        U[4, 7, 11] = -1.0
        U[1, 9, 2] += 3.0
        U[4, 9, 2] += 9.0
    if case == "tiny":
        U *= 1e-60
    if case == "huge":
        U *= 1e60
    op = dg.Operator(3, X, I.connectivity(spec), phys, precision=precision)
    Ja, J = op.metrics()
    iJ = 1.0 / J.ravel()
    Ja = Ja.reshape(-1, 3, 3)
    if precision == dg.FP32_MIXED:
        Ja, iJ = Ja.astype(np.float32).astype(np.float64), iJ.astype(np.float32).astype(np.float64)
    want = 0.9 * 2.0 / 7.0 / formula(U, Ja, iJ, phys["gamma"])
    got = op.time_step(0.9, torch.from_numpy(np.ascontiguousarray(U)).cuda())
    print(case, got, want)
    assert abs(got - want) <= 1e-14 * want
