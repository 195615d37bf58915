"""Rows next to the poles in items of 16 columns whose levels eight groups of
threads share out, on grids where these fit beside the other rows: even and
uneven level shares, rows that end inside an item, against the FP64 oracle."""
import numpy as np
import pytest

import oracle
from paper_2103_10114_gb300 import agcm, inputs

pytestmark = pytest.mark.gpu
FIELDS = agcm.FIELDS

GRIDS = [(200, 100, 16, False), (198, 99, 17, True), (257, 128, 30, False)]


@pytest.mark.parametrize("grid", GRIDS, ids=lambda g: "%dx%dx%d-%d" % g)
def test_polar_rows_match_oracle(cuda_ok, grid):
    """Tendency and two steps in both precisions, two runs bit for bit; the
    parity tests' tolerances."""
    agcm.build()
    I, J, K, th = grid
    thermo = dict(profile=1, delta=0.5, delta_c=0.1, delta_p=0.05) if th else None
    st = inputs.random_state(I, J, K, seed=I)
    g = agcm.Grid(I, J, K, phis=st["phis"], thermo=thermo)
    assert g.leap()[0].max() > 31
    o = oracle.Oracle(I, J, K, phis=st["phis"], thermo=thermo)
    dt = 0.1 * g.dt(100.0)
    want_t, want_x = o.tendency(st), o.step(st, dt, 2)
    assert all(np.isfinite(want_x[f]).all() for f in FIELDS)
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
