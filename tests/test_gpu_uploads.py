"""Tables that a call uploads on its own (the adjoint's row items, the
persistent ensemble's) are there before its first launch, whatever stream that
is on: torch's side streams do not wait for the stream that copies."""
import os
import re

import pytest

from paper_2103_10114_gb300 import agcm, inputs
from paper_2103_10114_gb300.ensemble import Ensemble

SOURCE = os.path.join(os.path.dirname(os.path.dirname(__file__)), "paper_2103_10114_gb300", "csrc", "agcm_api.cu")


def test_every_upload_is_waited_for():
    """The one synchronous copy from host memory stands in upload(), which waits for it."""
    text = re.sub(r"//[^\n]*", "", open(SOURCE).read())
    copies = [m.start() for m in re.finditer(r"\bcudaMemcpy\(", text)]
    a = text.index("bool upload(")
    b = text.index("\n}", a)
    assert len(copies) == 1 and a < copies[0] < b
    assert "cudaStreamSynchronize(" in text[copies[0]:b]


@pytest.mark.gpu
@pytest.mark.parametrize("grid", [(97, 45, 5), (256, 128, 6)], ids=lambda g: "%dx%dx%d" % g)
def test_first_adjoint_on_a_side_stream(cuda_ok, grid):
    import torch

    agcm.build()
    I, J, K = grid
    st = inputs.random_state(I, J, K, seed=I)
    lam = inputs.random_direction(I, J, K, seed=2)
    g = agcm.Grid(I, J, K, phis=st["phis"])
    dt = 0.1 * g.dt(100.0)
    outs = []
    for stream in (torch.cuda.Stream(), torch.cuda.default_stream()):
        s = agcm.State(g, agcm.AGCM_FP32)
        s.load(st)
        d = {f: torch.as_tensor(lam[f], dtype=torch.float32, device="cuda") for f in agcm.FIELDS}
        torch.cuda.synchronize()
        outs.append(s.step_adjoint(d, dt, stream=stream))
        torch.cuda.synchronize()
        s.close()
    assert all(torch.equal(outs[0][f], outs[1][f]) for f in agcm.FIELDS)


@pytest.mark.gpu
def test_first_persistent_step_on_a_side_stream(cuda_ok):
    import torch

    agcm.build()
    outs = []
    for stream in (torch.cuda.Stream(), torch.cuda.default_stream()):
        states = []
        for I, J, K in ((96, 48, 5), (200, 100, 4)):
            st = inputs.random_state(I, J, K, seed=I)
            states.append(agcm.State(agcm.Grid(I, J, K, phis=st["phis"]), agcm.AGCM_FP32))
            states[-1].load(st)
        torch.cuda.synchronize()
        e = Ensemble(states)
        e.configure(8, 0, 1)
        e.step(2, [0.1 * s.grid.dt(100.0) for s in states], stream=stream)
        e.status(stream)
        outs.append([s.store() for s in states])
        torch.cuda.synchronize()
        e.close()
        for s in states:
            s.close()
    assert all(torch.equal(a[f], b[f]) for a, b in zip(*outs) for f in agcm.FIELDS)


@pytest.mark.gpu
def test_first_adjoint_beside_a_capture(cuda_ok):
    """The workspace of a first reverse step is made while another thread
    captures a graph on a stream of its own: neither disturbs the other."""
    import threading

    import torch

    agcm.build()
    I, J, K = 96, 48, 4
    st = inputs.random_state(I, J, K, seed=1)
    lam = inputs.random_direction(I, J, K, seed=2)
    a, b, c = (agcm.State(agcm.Grid(I, J, K, phis=st["phis"]), agcm.AGCM_FP32) for _ in range(3))
    side = torch.cuda.Stream()
    lam = {f: torch.as_tensor(lam[f], dtype=torch.float32, device="cuda") for f in agcm.FIELDS}
    for s in (a, b, c):
        s.load(st)
    a.step(1, 1.0)
    out = b.empty()
    torch.cuda.synchronize()
    errors = []

    def other():
        try:
            args = [(agcm._vp * 4)(*[t[f].data_ptr() for f in agcm.FIELDS]) for t in (lam, out)]
            agcm.check(agcm.lib().agcm_step_adjoint(b.handle, *args, 1.0, agcm._stream_ptr(side)))
            side.synchronize()
        except Exception as e:  # reported by the test's own thread
            errors.append(e)

    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, capture_error_mode="thread_local"):
        a.step(1, 1.0)
        t = threading.Thread(target=other)
        t.start()
        t.join()
    assert not errors, errors
    g.replay()
    want = c.step_adjoint(lam, 1.0)
    torch.cuda.synchronize()
    assert all(torch.equal(out[f], want[f]) for f in agcm.FIELDS)
