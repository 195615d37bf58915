"""The row-segment form of the adjoint's column pass at its edges: segments of
one column to several hundred, rows that are not 16-byte aligned, levels around
its group of eight, divergence pairs past its halo, and more levels than its
shared memory holds (above about 200), where the form without staging runs;
the dot test against the oracle's tangent-linear step."""
import numpy as np
import pytest

import oracle
from paper_2103_10114_gb300 import agcm, inputs

pytestmark = pytest.mark.gpu
FIELDS = agcm.FIELDS

GRIDS = [
    (120, 14, 7, "ones"),
    (124, 14, 8, "eq7"),
    (123, 21, 9, "random"),
    (250, 18, 16, "random"),
    (8, 8, 17, "ones"),
    (360, 180, 3, "eq7"),  # strides above 64 next to the poles
    (36, 12, 110, "eq7"),
    (36, 12, 210, "eq7"),  # without staging
]


@pytest.mark.parametrize("grid", GRIDS, ids=lambda g: "%dx%dx%d-%s" % g)
def test_adjoint_dot_product(cuda_ok, grid):
    """<lam, J v> = <J^T lam, v>: FP64 to 1e-12, FP32 to 1e-5 of the sum of
    magnitudes (the tolerances of the adjoint tests)."""
    agcm.build()
    I, J, K, kind = grid
    mu = mv = None
    if kind == "ones":
        mu, mv = np.ones(J, np.int32), np.ones(J - 1, np.int32)
    elif kind == "random":
        rng = np.random.default_rng(11)
        mu = (2 * rng.integers(0, min(40, I // 4), J) + 1).astype(np.int32)
        mv = (2 * rng.integers(0, min(40, I // 4), J - 1) + 1).astype(np.int32)
    st = inputs.random_state(I, J, K, seed=I)
    x = {f: st[f] for f in FIELDS}
    g = agcm.Grid(I, J, K, leap_u=mu, leap_v=mv, phis=st["phis"])
    o = oracle.Oracle(I, J, K, leap_u=mu, leap_v=mv, phis=st["phis"])
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
