"""The adjoint's column pass at the level counts where its forms change: both
arrays in shared memory up to 57 levels in FP32, one above, the form without
staging from 184 levels (on grids of more blocks than SMs) and from 397 in FP32,
from 199 in FP64; the dot test against the oracle's tangent-linear step."""
import numpy as np
import pytest

import oracle
from paper_2103_10114_gb300 import agcm, inputs

pytestmark = pytest.mark.gpu
FIELDS = agcm.FIELDS

GRIDS = [
    (124, 14, 57),
    (123, 14, 58),
    (130, 80, 183),
    (129, 80, 184),
    (36, 8, 198),
    (37, 8, 199),
    (36, 6, 396),
    (36, 6, 397),
]


@pytest.mark.parametrize("grid", GRIDS, ids=lambda g: "%dx%dx%d" % g)
def test_adjoint_dot_product(cuda_ok, grid):
    """<lam, J v> = <J^T lam, v>: FP64 to 1e-12, FP32 to 1e-5 of the sum of
    magnitudes (the tolerances of the adjoint tests)."""
    agcm.build()
    I, J, K = grid
    st = inputs.random_state(I, J, K, seed=I)
    x = {f: st[f] for f in FIELDS}
    g = agcm.Grid(I, J, K, phis=st["phis"])
    o = oracle.Oracle(I, J, K, phis=st["phis"])
    dt = 0.1 * g.dt(100.0)
    v, lam = inputs.random_direction(I, J, K, seed=1), inputs.random_direction(I, J, K, seed=2)
    _, jv = o.step_jvp(x, v, dt, 1)
    lhs = sum(float(np.sum(lam[f] * jv[f])) for f in FIELDS)
    mag = sum(float(np.sum(np.abs(lam[f] * jv[f]))) for f in FIELDS)
    for prec, tol in ((agcm.AGCM_FP64, 1e-12), (agcm.AGCM_FP32, 1e-5)):
        s = agcm.State(g, prec)
        s.load(x)
        got = [{f: t.double().cpu().numpy() for f, t in s.step_adjoint(lam, dt).items()} for _ in range(2)]
        rhs = sum(float(np.sum(got[0][f] * v[f])) for f in FIELDS)
        assert abs(lhs - rhs) <= tol * mag, (prec, lhs, rhs, mag)
        assert all(np.array_equal(got[0][f], got[1][f]) for f in FIELDS), prec
        s.close()
