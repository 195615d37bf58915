"""Reverse steps of grids with more levels than the adjoint gather's shared
memory or a launch grid's z dimension holds: the gradient against a central
difference of the step itself."""
import numpy as np
import pytest

from paper_2103_10114_gb300 import agcm, inputs

pytestmark = pytest.mark.gpu
FIELDS = agcm.FIELDS


@pytest.mark.parametrize("grid", [(12, 4, 17500, 1), (72, 3, 66000, 35)], ids=lambda g: "%dx%dx%d-%d" % g)
def test_gradient_of_many_levels(cuda_ok, grid):
    """FP64, without the identity's part (the step's Jacobian less 1, some 1e-2
    of it here): a central difference of step h is off by (h / |x|)^2 and by
    eps |x| / h, with h = 1e-3 and |x| >= 20 under 1e-8 and 1e-9 of that part;
    1e-6 of the sum of magnitudes."""
    import torch

    agcm.build()
    I, J, K, M = grid
    g = agcm.Grid(I, J, K, leap_u=np.full(J, M, np.int32), leap_v=np.full(J - 1, M, np.int32))
    x, v = inputs.random_state(I, J, K, seed=1), inputs.random_direction(I, J, K, seed=2)
    dev = lambda a: {f: torch.as_tensor(a[f], dtype=torch.float64, device="cuda") for f in FIELDS}
    x, v, lam = dev(x), dev(v), dev(inputs.random_direction(I, J, K, seed=3))
    s = agcm.State(g, agcm.AGCM_FP64)
    dt, h = 10.0, 1e-3

    def step(sign):
        s.load({f: x[f] + sign * h * v[f] for f in FIELDS})
        s.step(1, dt)
        return s.store()

    a, b = step(1), step(-1)
    d = {f: (a[f] - b[f]) / (2 * h) - v[f] for f in FIELDS}
    lhs = sum((lam[f] * d[f]).sum().item() for f in FIELDS)
    mag = sum((lam[f] * d[f]).abs().sum().item() for f in FIELDS)
    s.load(x)
    grad = s.step_adjoint(lam, dt)
    rhs = sum(((grad[f] - lam[f]) * v[f]).sum().item() for f in FIELDS)
    assert np.isfinite(lhs) and abs(lhs - rhs) <= 1e-6 * mag
    s.close()
