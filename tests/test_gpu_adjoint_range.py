"""Cotangents far below one: the adjoint is linear down to FP64's own range, for all
equations together and for one alone beside zeros.  Scaled by a power of two the
result is that of the unscaled cotangent to FP64 rounding of two summation orders
(1e-13 of the largest value; 2^-150 stays in fixed point, 2^-230 and 2^-300 do not)."""
import numpy as np
import pytest

from gpu_helpers import torch_cuda
from test_gpu_adjoint_fx import cotangent, operator, vjp

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
