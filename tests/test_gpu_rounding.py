"""FP32 tendencies against the FP64 oracle at the level of rounding: what the
row-segment kernel's tables and sums add to the rounding of the inputs."""
import numpy as np
import pytest

import oracle
from paper_2103_10114_gb300 import agcm, inputs

pytestmark = pytest.mark.gpu


def _tendency(I, J, K):
    """(FP32 tendency, FP64 tendency) of the same FP32 state."""
    agcm.build()
    st = inputs.random_state(I, J, K, seed=I + K, terrain=False)
    st = {f: np.asarray(v, np.float32).astype(np.float64) for f, v in st.items()}
    s = agcm.State(agcm.Grid(I, J, K), agcm.AGCM_FP32)
    s.set_stage_kernel(agcm.STAGE_ROW)
    s.load(st)
    got = {f: v.double().cpu().numpy() for f, v in s.tendency().items()}
    s.close()
    return got, oracle.Oracle(I, J, K).tendency(st)


@pytest.mark.parametrize("grid", [(256, 128, 30), (405, 203, 20)], ids=lambda g: "%dx%dx%d" % g)
def test_rows_share_no_large_factor(cuda_ok, grid):
    """A tendency is one factor of its row times sums: what a row's values have
    in common is the rounding of that factor and of the tables behind its
    leading terms, two of 2.5e-8 each (the root mean square of a rounding), at
    most.  Root mean square over the rows of a field: 4e-8."""
    got, want = _tendency(*grid)
    for f in ("U", "V", "Phi"):
        e = got[f] - want[f]
        k = (e * want[f]).sum((0, 2)) / (want[f] ** 2).sum((0, 2))
        # what the values' own roundings (1e-7 of the largest term, a few times the tendency) leave of it
        noise = np.sqrt((e ** 2).sum((0, 2)) / (want[f] ** 2).sum((0, 2)) / want[f][:, 0].size)
        assert np.sqrt((k ** 2).mean()) <= 4e-8 + 3 * noise.mean(), (f, np.sqrt((k ** 2).mean()), noise.mean())


def test_the_hydrostatic_sum_over_many_levels(cuda_ok):
    """At rest, U's tendency is the difference of two hydrostatic sums.  The
    same sums in FP32 on the CPU, Phi of mean 200 and deviation 50 over 120
    levels: a difference is 2.8e-6 of the root mean square off where a sum is
    one chain, 1.3e-6 where it is kept in groups of eight levels."""
    agcm.build()
    I, J, K = 256, 128, 120
    st = {"U": np.zeros((K, J, I)), "V": np.zeros((K, J - 1, I)), "pi": np.zeros((J, I)), "phis": np.zeros((J, I)),
          "Phi": np.random.default_rng(5).normal(200.0, 50.0, (K, J, I)).astype(np.float32).astype(np.float64)}
    s = agcm.State(agcm.Grid(I, J, K), agcm.AGCM_FP32)
    s.load(st)
    got = s.tendency()["U"].double().cpu().numpy()
    s.close()
    want = oracle.Oracle(I, J, K).tendency(st)["U"]
    # rows on segments: the column body sums differences
    rows = agcm.Grid(I, J, K).leap()[0] < 30
    assert np.sqrt(((got - want)[:, rows] ** 2).mean() / (want[:, rows] ** 2).mean()) <= 2e-6
