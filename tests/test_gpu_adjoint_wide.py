"""The adjoint gather's rows of halo 33 to 48 in blocks of 192 threads, and the
unstaged form's chunks of several levels: full and ragged segments, rows that are
not 16-byte aligned, beside rows of the other forms and alone; the dot test
against the oracle's tangent-linear step."""
import numpy as np
import pytest

import oracle
from paper_2103_10114_gb300 import agcm, inputs

pytestmark = pytest.mark.gpu
FIELDS = agcm.FIELDS

# blocks of 192 threads where they are 1.5 an SM, 228 on 152 SMs
GRIDS = [
    (288, 80, 5, (33, 47)),   # three segments of 96 columns a row
    (289, 90, 1, (33, 47)),   # unaligned
    (130, 140, 6, (1, 47)),   # every form
    (200, 100, 7, (49, 99)),  # unstaged rows alone, two levels a chunk
    (230, 180, 9, (35, 75)),
]


@pytest.mark.parametrize("grid", GRIDS, ids=lambda g: "%dx%dx%d-%s" % g)
def test_adjoint_dot_product(cuda_ok, grid):
    """<lam, J v> = <J^T lam, v>: FP64 to 1e-12, FP32 to 1e-5 of the sum of
    magnitudes (the tolerances of the adjoint tests)."""
    agcm.build()
    I, J, K, (lo, hi) = grid
    rng = np.random.default_rng(9)
    mu = (2 * rng.integers(lo // 2, hi // 2 + 1, J) + 1).astype(np.int32)
    mv = (2 * rng.integers(lo // 2, hi // 2 + 1, J - 1) + 1).astype(np.int32)
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
