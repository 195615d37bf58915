"""Two short remainders of rows in one block of the row-segment stage kernel:
one column, a full half block, an odd count of remainders, unaligned rows, one
level and more levels than the ring holds, against the FP64 oracle."""
import numpy as np
import pytest

import oracle
from paper_2103_10114_gb300 import agcm, inputs

pytestmark = pytest.mark.gpu
FIELDS = agcm.FIELDS

# segments hold 120 columns of halo 4, half a block 56; blocks are shared where
# that saves a wave of three blocks (FP64: two) on each of 152 SMs
GRIDS = [
    (405, 203, 3, "eq7"),   # FP32: remainder 45, unaligned, strides of every class
    (176, 600, 5, "ones"),  # FP32: remainder 56, aligned
    (121, 602, 1, "ones"),  # FP32: remainder 1
    (250, 350, 6, "ones"),  # FP32: remainder 10, nlon % 4 == 2
    (176, 404, 4, "ones"),  # FP64
    (121, 621, 2, "ones"),  # FP64
    (250, 232, 3, "ones"),  # FP64
]


@pytest.mark.parametrize("grid", GRIDS, ids=lambda g: "%dx%dx%d-%s" % g)
def test_shared_blocks_match_oracle(cuda_ok, grid):
    """Tendency and two steps in both precisions, two runs bit for bit; the
    parity tests' tolerances."""
    agcm.build()
    I, J, K, kind = grid
    mu = mv = None
    if kind == "ones":
        mu, mv = np.ones(J, np.int32), np.ones(J - 1, np.int32)
    st = inputs.random_state(I, J, K, seed=I)
    g = agcm.Grid(I, J, K, leap_u=mu, leap_v=mv, phis=st["phis"])
    o = oracle.Oracle(I, J, K, leap_u=mu, leap_v=mv, phis=st["phis"])
    dt = (0.1 if kind == "eq7" else 0.01) * g.dt(100.0)  # strides of 1: short cells next to the poles
    want_t, want_x = o.tendency(st), o.step(st, dt, 2)
    err = lambda got, want: max(np.abs(got[f] - want[f]).max() / np.abs(want[f]).max() for f in FIELDS)
    for prec, tol_t, tol_x in ((agcm.AGCM_FP64, 1e-11, 1e-12), (agcm.AGCM_FP32, 1e-4, 1e-5)):
        runs = []
        for _ in range(2):
            s = agcm.State(g, prec)
            s.load(st)
            t = {f: v.double().cpu().numpy() for f, v in s.tendency().items()}
            s.step(2, dt)
            x = {f: v.double().cpu().numpy() for f, v in s.store().items()}
            s.close()
            assert err(t, want_t) <= tol_t and err(x, want_x) <= tol_x, prec
            runs.append((t, x))
        assert all(np.array_equal(runs[0][q][f], runs[1][q][f]) for q in (0, 1) for f in FIELDS), prec
