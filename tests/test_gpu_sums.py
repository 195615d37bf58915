"""The FP32 states' exact sums (vertical means, diagnostics) over the range of
FP32: ordinary values, values whose products leave that range (summed in
FP64), zeros, non-finite values, rows of any alignment."""
import numpy as np
import pytest

import oracle
from paper_2103_10114_gb300 import agcm, inputs

pytestmark = pytest.mark.gpu
FIELDS = agcm.FIELDS


def _state(I, J, K, scale):
    st = inputs.random_state(I, J, K, seed=I + K)
    for f in ("U", "V", "Phi"):
        st[f] = (st[f] * scale).astype(np.float32).astype(np.float64)
    st["pi"] = st["pi"].astype(np.float32).astype(np.float64)
    return st


@pytest.mark.parametrize("scale", [1.0, 1e-10, 1e-16, 1e-24, 1e14, 1e28])
@pytest.mark.parametrize("grid", [(64, 30, 7), (37, 23, 13)], ids=lambda g: "%dx%dx%d" % g)
def test_diagnostics_over_the_range(cuda_ok, grid, scale):
    """Energies against the oracle's FP64 sums of the same values: the FP32
    path drops nothing above 2^-60 of a sum, so both differ by FP64 rounding
    (1e-13 for sums of 1e4 terms); maxima exact."""
    agcm.build()
    I, J, K = grid
    st = _state(I, J, K, scale)
    g = agcm.Grid(I, J, K, phis=st["phis"])
    s = agcm.State(g, agcm.AGCM_FP32)
    s.load(st)
    got, want = s.diagnostics(), oracle.Oracle(I, J, K, phis=st["phis"]).diagnostics(st)
    for k in ("mass", "e_kin", "e_pot", "e_ps", "energy"):
        assert abs(got[k] - want[k]) <= 1e-13 * abs(want[k]), (k, got[k], want[k])
    assert got["max_u"] == want["max_u"] and got["max_v"] == want["max_v"] and got["finite"] == 1
    s.close()


@pytest.mark.parametrize("value", [np.inf, -np.inf, np.nan])
def test_diagnostics_of_non_finite_values(cuda_ok, value):
    agcm.build()
    I, J, K = 64, 30, 4
    st = _state(I, J, K, 1.0)
    st["U"][2, 3, 5] = value
    g = agcm.Grid(I, J, K)
    s = agcm.State(g, agcm.AGCM_FP32)
    s.load(st)
    d = s.diagnostics()
    assert d["finite"] == 0
    assert np.isnan(d["e_kin"]) if np.isnan(value) else d["e_kin"] == np.inf
    assert d["max_u"] == (np.inf if np.isinf(value) else np.nanmax(np.abs(st["U"])))
    assert np.isfinite(d["e_pot"])
    s.close()


@pytest.mark.parametrize("scale", [1.0, 1e-10, 1e-24, 1e-35, 1e14, 1e30])
@pytest.mark.parametrize("levels", [1, 6, 7, 30])
def test_vertical_means_over_the_range(cuda_ok, levels, scale):
    """The tendency of pi is linear in U and V through their vertical means
    (non-uniform levels): FP32 against the oracle within the FP32 tolerance of
    a tendency at any scale."""
    agcm.build()
    I, J, K = 96, 48, levels
    st = _state(I, J, K, scale)
    sh = np.concatenate([[0.0], np.cumsum(np.linspace(1.0, 3.0, K))])
    sh = sh / sh[-1]
    g = agcm.Grid(I, J, K, sigma_half=sh)
    s = agcm.State(g, agcm.AGCM_FP32)
    s.load(st)
    got = s.tendency()["pi"].double().cpu().numpy()
    one = {**st, "U": st["U"] / scale, "V": st["V"] / scale, "Phi": 0 * st["Phi"]}
    want = oracle.Oracle(I, J, K, sigma_half=sh).tendency(one)["pi"] * scale
    big = np.abs(want).max()
    assert np.abs(got - want).max() <= 1e-5 * big + 1e-44, (np.abs(got - want).max() / big)
    s.close()
