"""Grids with many rows of strides above 31, which the row-segment kernel leaves
to the column body: some (blocks of 32 columns), more (blocks of 128), most of
them (the column kernel), against the FP64 oracle."""
import numpy as np
import pytest

import oracle
from paper_2103_10114_gb300 import agcm, inputs

pytestmark = pytest.mark.gpu
FIELDS = agcm.FIELDS


@pytest.mark.parametrize("grid", [(256, 60, 5, 0.1), (720, 60, 3, 0.3), (150, 64, 4, 0.5), (130, 64, 17, 1.0)],
                         ids=lambda g: "%dx%dx%d-%.1f" % g)
def test_wide_rows_match_oracle(cuda_ok, grid):
    """A share of the rows, half at each pole: tendency and two steps, by the
    grid's own rule and with the row kernel asked for, in both precisions; the
    parity tests' tolerances."""
    agcm.build()
    I, J, K, share = grid
    mu, mv = (np.array(v) for v in agcm.Grid(I, J, K).leap())
    rows = np.minimum(np.arange(J), J - 1 - np.arange(J)) < share * J / 2
    mu[rows] = np.maximum(mu[rows], 2 * np.random.default_rng(I).integers(17, 30, rows.sum()) + 1)
    st = inputs.random_state(I, J, K, seed=I)
    g = agcm.Grid(I, J, K, leap_u=mu, leap_v=mv, phis=st["phis"])
    o = oracle.Oracle(I, J, K, leap_u=mu, leap_v=mv, phis=st["phis"])
    dt = 0.1 * g.dt(100.0)
    want_t, want_x = o.tendency(st), o.step(st, dt, 2)
    err = lambda got, want: max(np.abs(got[f] - want[f]).max() / np.abs(want[f]).max() for f in FIELDS)
    for prec, tol_t, tol_x in ((agcm.AGCM_FP64, 1e-11, 1e-12), (agcm.AGCM_FP32, 1e-4, 1e-5)):
        for choice in (agcm.STAGE_AUTO, agcm.STAGE_ROW):
            s = agcm.State(g, prec)
            s.set_stage_kernel(choice)
            s.load(st)
            t = {f: v.double().cpu().numpy() for f, v in s.tendency().items()}
            s.step(2, dt)
            x = {f: v.double().cpu().numpy() for f, v in s.store().items()}
            s.close()
            assert err(t, want_t) <= tol_t and err(x, want_x) <= tol_x, (prec, choice)
