"""A repeated agcm_tendency_static call finds its tables and its work items in
place: what the host does for it does not grow with the grid."""
import ctypes
import time

import numpy as np
import pytest

from paper_2103_10114_gb300 import agcm, inputs

pytestmark = pytest.mark.gpu


def test_repeated_calls_do_not_plan_again(cuda_ok):
    """The quickest of 50 calls on a grid of 4096 rows against one of 64: a
    plan of the rows takes a millisecond there, a call's two launches some ten
    microseconds on either; five times as long leaves room for both."""
    import torch

    agcm.build()

    def quickest(I, J, K):
        st = inputs.random_state(I, J, K, seed=1, terrain=False)
        g = agcm.Grid(I, J, K, leap_u=np.ones(J, np.int32), leap_v=np.ones(J - 1, np.int32))
        x = [torch.as_tensor(st[f], dtype=torch.float32, device="cuda") for f in agcm.FIELDS]
        out = [torch.empty_like(t) for t in x]
        args = [ctypes.c_void_p(t.data_ptr()) for t in x + out]
        times = []
        for _ in range(50):
            torch.cuda.synchronize()
            t0 = time.perf_counter()
            agcm.check(agcm.lib().agcm_tendency_static(g.handle, agcm.AGCM_FP32, *args, agcm._stream_ptr()))
            times.append(time.perf_counter() - t0)
        torch.cuda.synchronize()
        return min(times)

    small, large = quickest(64, 64, 1), quickest(64, 4096, 1)
    assert large <= 5 * small, (small, large)
