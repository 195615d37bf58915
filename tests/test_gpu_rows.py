"""The row-segment stage kernel at the edges of its forms: pairs of rows and
single rows, rows that end a row short of a segment, rows that are not 16-byte
aligned, wraps of the periodic seam, one level, and rows left to the column
body, each against the FP64 oracle."""
import numpy as np
import pytest

import oracle
from paper_2103_10114_gb300 import agcm, inputs

pytestmark = pytest.mark.gpu
FIELDS = agcm.FIELDS

# (nlon, nlat, nlev, strides, thermo): an item is a segment of at most 128 - 2 H
# columns; 120 columns of halo 4 are one full segment
GRIDS = [
    (120, 36, 3, "ones", False),    # one segment, every row in pairs but the last
    (121, 35, 2, "ones", True),     # one column more: two segments, unaligned rows
    (124, 34, 1, "eq7", False),     # one level
    (130, 70, 7, "eq7", True),      # nlon % 4 == 2: a chunk of four columns straddles the seam
    (97, 45, 5, "eq7", False),      # odd nlon, odd nlat
    (488, 220, 4, "eq7", False),    # pairs and single rows; strides above 31 next to the poles
    (486, 244, 3, "eq7", True),     # the same, unaligned
    (960, 90, 2, "random", False),  # ragged odd strides: single rows among pairs
]


def _strides(kind, I, J):
    if kind == "ones":
        return np.ones(J, np.int32), np.ones(J - 1, np.int32)
    if kind == "random":
        rng = np.random.default_rng(5)
        mu, mv = 2 * rng.integers(0, 18, J) + 1, 2 * rng.integers(0, 18, J - 1) + 1
        mu[20:40], mv[20:40] = 3, 3
        return mu.astype(np.int32), mv.astype(np.int32)
    return None, None


def _err(got, want):
    return max(np.abs(got[f] - want[f]).max() / np.abs(want[f]).max() for f in FIELDS)


@pytest.mark.parametrize("grid", GRIDS, ids=lambda g: "%dx%dx%d-%s" % g[:4])
def test_row_segments_match_oracle(cuda_ok, grid):
    """Tendency and two steps with the row-segment kernel asked for, and two
    steps as the grid's own rule has it, in both precisions; two runs agree bit
    for bit.  Tolerances: those of the parity tests (FP64 differs from the
    oracle in the order of sums, FP32 rounds at 6e-8 an operation; the tendency
    of pi is a small difference of fluxes)."""
    agcm.build()
    I, J, K, kind, th = grid
    mu, mv = _strides(kind, I, J)
    thermo = dict(profile=1, delta=0.5, delta_c=0.1, delta_p=0.05) if th else None
    st = inputs.random_state(I, J, K, seed=I)
    g = agcm.Grid(I, J, K, leap_u=mu, leap_v=mv, phis=st["phis"], thermo=thermo)
    o = oracle.Oracle(I, J, K, leap_u=mu, leap_v=mv, phis=st["phis"], thermo=thermo)
    dt = 0.1 * g.dt(100.0)
    want_t, want_x = o.tendency(st), o.step(st, dt, 2)
    for prec, tol_t, tol_x in ((agcm.AGCM_FP64, 1e-11, 1e-12), (agcm.AGCM_FP32, 1e-4, 1e-5)):
        runs = []
        for choice in (2, 2, 0):
            s = agcm.State(g, prec)
            s.set_stage_kernel(choice)
            s.load(st)
            t = {f: v.double().cpu().numpy() for f, v in s.tendency().items()}
            s.step(2, dt)
            x = {f: v.double().cpu().numpy() for f, v in s.store().items()}
            s.close()
            assert _err(t, want_t) <= tol_t and _err(x, want_x) <= tol_x, (prec, choice)
            runs.append((t, x))
        for a, b in zip(runs[0], runs[1]):
            assert all(np.array_equal(a[f], b[f]) for f in FIELDS), prec
