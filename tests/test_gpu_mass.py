"""Mass of an FP32 run: what crosses a row edge leaves one row and enters the
other, also where the rows' strides differ.  Over 300 steps the start of the
jet moves some 1e-3 of the mass between the latitudes; a face length that
differs by an FP32 rounding (6e-8) between the two rows of an edge shows as
some 6e-11 of the total, the rounding of pi itself (6e-8 of |pi| ~ 1e-2 over
sqrt(points)) below 2e-11 on these grids."""
import numpy as np
import pytest

from paper_2103_10114_gb300 import agcm, inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("grid", [(720, 360, 10), (405, 203, 6)], ids=lambda g: "%dx%dx%d" % g)
def test_mass_is_kept_across_stride_changes(cuda_ok, grid):
    agcm.build()
    I, J, K = grid
    st = inputs.baroclinic_jet(I, J, K, seed=3, noise=1e-3, terrain_seed=2)
    g = agcm.Grid(I, J, K, phis=st["phis"])
    s = agcm.State(g, agcm.AGCM_FP32)
    s.load(st)
    before = s.diagnostics()["mass"]
    s.step(300, g.dt(100.0))
    assert abs(s.diagnostics()["mass"] / before - 1.0) <= 4e-11
    s.close()


def test_mass_is_kept_across_the_edges_of_the_column_body(cuda_ok):
    """The same where every third row has a stride above 31 and is left to the
    column body, which takes its edges' lengths from other tables: two of three
    edges lie between the two bodies.  Seen in one tendency, free of the state's
    own rounding: with V the same everywhere the mass that leaves all rows and
    enters none, in units of an edge's flux over the square root of the number
    of edge points.  Each of an edge point's two rows rounds the product of
    length and P^v once, 2.5e-8 root mean square and independent of the other:
    3.5e-8 together, 1.4e-7 at four times that.  Lengths that differ by an FP32
    rounding between the rows add up over the 720 points of an edge: 8e-7."""
    agcm.build()
    I, J, K = 720, 360, 4
    mu, mv = (np.array(v) for v in agcm.Grid(I, J, K).leap())
    mu[1::3] = np.maximum(mu[1::3], 45)
    g = agcm.Grid(I, J, K, leap_u=mu, leap_v=mv)
    s = agcm.State(g, agcm.AGCM_FP32)
    s.set_stage_kernel(agcm.STAGE_ROW)
    s.load({"U": np.zeros((K, J, I)), "V": np.full((K, J - 1, I), 10.0), "Phi": np.zeros((K, J, I)),
            "pi": np.random.default_rng(3).normal(0.0, 0.01, (J, I))})
    t = s.tendency()["pi"].double().cpu().numpy()
    s.close()
    a, dlam, dth = 6.371e6, 2 * np.pi / I, np.pi / J
    area = a * a * np.sin((np.arange(J) + 0.5) * dth)[:, None] * dlam * dth
    flux = 10.0 * a * dlam
    assert abs((area * t).sum()) <= 1.4e-7 * flux * np.sqrt(I * (J - 1))
