"""dg_time_step where its FP32 bounds reach the end of FP32's range: meshes in
units far from their size (the squares of the metrics under- or overflow), states
in such units, and a ratio of specific heats near one, whose gamma - 1 has few
bits in FP32.  The largest value is a node at rest with a large sound speed beside
a slow one with a large velocity.  Bound: FP64 rounding of some twenty operations,
1e-14."""
import numpy as np
import pytest

from paper_2606_18927_gb300 import dg, inputs as I
from gpu_helpers import torch_cuda
from test_gpu_time_step import formula

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", [dg.FP64, dg.FP32_MIXED])
@pytest.mark.parametrize("length,speed,density,gamma",
                         [(s, 1.0, 1.0, 1.4) for s in (1e-7, 1e-10, 1e-11, 1e-12, 1e9, 1e11)]
                         + [(1.0, 1e-17, 1.0, 1.4), (1.0, 1e-9, 1e-25, 1.4), (1e-8, 1e-12, 1e-20, 1.4),
                            (1.0, 1e15, 1e-10, 1.4), (1.0, 1.0, 1.0, 1.0003)])
def test_time_step_is_the_formula_s(length, speed, density, gamma, precision):
    torch = torch_cuda()
    phys = I.phys_params(Ma=0.3, Re=1600.0, gamma=gamma)
    spec = I.BoxSpec(3, 3, 2, 2, lengths=(length, 1.1 * length, 0.9 * length))
    x, w = dg.lgl_nodes(3)
    X = I.node_coordinates(spec, x)
    one = np.ones_like(X[0])
    r, u, v, w_, p = (a * one for a in (1.0, 0.0, 0.0, 0.0, 1.0))
    u[7, 11] = 3.0        # flow: lam = (3 + c) a_x + c (a_y + a_z), c = 0.01
    p[7, 11] = 1e-4 / gamma
    c = 1.0 + (1e-5 if gamma < 1.1 else 0.05)  # sound, in units of the speed at which the two are equal
    s = np.array((3, 2, 2)) / np.array(spec.lengths)
    p[4, 5] = ((3.0 * s[0] + 0.01 * s.sum()) / s.sum() * c) ** 2 / gamma
    p[p == 1.0] = 1e-2
    U = I.conservative(density * r, speed * u, speed * v, speed * w_, density * speed ** 2 * p, gamma)
    op = dg.Operator(3, X, I.connectivity(spec), phys, precision=precision)
    Ja, J = op.metrics()
    iJ = 1.0 / J.ravel()
    Ja = Ja.reshape(-1, 3, 3)
    if precision == dg.FP32_MIXED:
        with np.errstate(all="ignore"):
            Ja, iJ = Ja.astype(np.float32).astype(np.float64), iJ.astype(np.float32).astype(np.float64)
    lam = formula(U, Ja, iJ, gamma)
    if not np.isfinite(lam) or lam == 0.0:
        pytest.skip("outside the range of the FP32 metrics")
    want = 0.9 * 2.0 / 7.0 / lam
    got = op.time_step(0.9, torch.from_numpy(np.ascontiguousarray(U)).cuda())
    print(length, speed, density, gamma, got, want)
    assert abs(got - want) <= 1e-14 * want
