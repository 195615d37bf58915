"""agcm_tendency_static on grids that take the row-segment kernel: its tables are
built on the device and its row items kept beside them; against agcm_tendency,
two calls and a change of grid in between."""
import ctypes

import numpy as np
import pytest

from paper_2103_10114_gb300 import agcm, inputs

pytestmark = pytest.mark.gpu
FIELDS = agcm.FIELDS

# (nlon, nlat, nlev, share of rows with strides above 31)
GRIDS = [(130, 70, 3, 0.0), (257, 128, 5, 0.0), (256, 60, 4, 0.2), (150, 64, 4, 0.6)]


@pytest.mark.parametrize("precision,tol", [(agcm.AGCM_FP64, 1e-12), (agcm.AGCM_FP32, 1e-6)])
def test_static_tendency_matches_state_path(cuda_ok, precision, tol):
    """The tolerances of the static tendency's test on small grids: tables
    formed on the device may differ by a rounding."""
    import torch

    agcm.build()

    def static(g, x):
        out = {f: torch.empty_like(x[f]) for f in FIELDS}
        agcm.check(agcm.lib().agcm_tendency_static(g.handle, precision, *[ctypes.c_void_p(x[f].data_ptr()) for f in FIELDS],
                                                   *[ctypes.c_void_p(out[f].data_ptr()) for f in FIELDS],
                                                   agcm._stream_ptr()))
        return out

    held = []
    for I, J, K, share in GRIDS:
        mu, mv = (np.array(v) for v in agcm.Grid(I, J, K).leap())
        rows = np.minimum(np.arange(J), J - 1 - np.arange(J)) < share * J / 2
        mu[rows] = np.maximum(mu[rows], 45)
        st = inputs.random_state(I, J, K, seed=I)
        g = agcm.Grid(I, J, K, leap_u=mu, leap_v=mv, phis=st["phis"])
        s = agcm.State(g, precision)
        x = {f: torch.as_tensor(st[f], dtype=s.dtype, device="cuda") for f in FIELDS}
        s.load(x)
        held.append((g, s, x, s.tendency()))
    for _ in range(2):
        for g, s, x, want in held:
            first, second = static(g, x), static(g, x)
            for f in FIELDS:
                assert (first[f] - want[f]).abs().max() <= tol * want[f].abs().max(), (g.nlon, f)
                assert torch.equal(first[f], second[f]), (g.nlon, f)
    for g, s, x, want in held:
        s.close()
