"""An allocator hook that returns memory of little alignment: the library's
tables and workspaces are read by 16-byte loads and copies all the same."""
import ctypes
import subprocess

import pytest

from paper_2103_10114_gb300 import agcm, inputs

FIELDS = agcm.FIELDS


class Hook:
    """alloc / free through `take` and `give`, 8 bytes past what they hand out."""

    def __init__(self, take, give):
        self.live, self.asked = {}, []

        def alloc(n, ctx):
            p = take(int(n) + 8)
            self.asked.append(int(n))
            self.live[p + 8] = p
            return p + 8

        def free(p, ctx):
            give(self.live.pop(p))  # KeyError for an address that alloc did not return

        self.cbs = agcm._ALLOC_T(alloc), agcm._FREE_T(free)

    def __enter__(self):
        a, f = (ctypes.cast(c, ctypes.c_void_p) for c in self.cbs)
        agcm.check(agcm.lib().agcm_set_allocator(a, f, None))
        return self

    def __exit__(self, *exc):
        agcm.check(agcm.lib().agcm_set_allocator(None, None, None))
        agcm._alloc_cbs = None


PROGRAM = r"""
#include <cstdlib>
#include <set>
#include "agcm_host.h"
int main() {
  for (size_t shift : {0u, 8u, 16u, 4u, 248u, 1u}) {
    std::set<void*> live;
    char* const room = (char*)(((uintptr_t)std::malloc(1 << 14) + 255) & ~(uintptr_t)255);
    size_t given = 0;
    auto take = [&](size_t n) { given = n; live.insert(room + shift); return (void*)(room + shift); };
    auto give = [&](void* p) { if (!live.erase(p)) std::exit(2); };
    agcm::AlignedBlocks b;
    char* const q = (char*)b.take(1000, take, give);
    if ((uintptr_t)q % 16 || q < room + shift || q + 1000 > room + shift + given || live.size() != 1) return 1;
    give(b.release(q));
    if (!live.empty()) return 3;
    if (b.release(q) != q) return 4;
  }
  agcm::AlignedBlocks b;
  return b.take(8, [](size_t) { return (void*)nullptr; }, [](void*) { std::exit(2); }) ? 5 : 0;
}
"""


def test_blocks_are_aligned_and_given_back(tmp_path):
    src, exe = tmp_path / "main.cpp", tmp_path / "main"
    src.write_text(PROGRAM)
    subprocess.check_call(["g++", "-std=c++17", "-I", agcm._CSRC, "-o", str(exe), str(src)])
    assert subprocess.run([str(exe)]).returncode == 0


@pytest.mark.gpu
@pytest.mark.parametrize("prec", [agcm.AGCM_FP64, agcm.AGCM_FP32])
def test_same_results_from_memory_of_little_alignment(cuda_ok, prec):
    import torch

    agcm.build()
    I, J, K = 256, 128, 5
    st = inputs.random_state(I, J, K, seed=3)
    lam = inputs.random_direction(I, J, K, seed=2)

    def run():
        g = agcm.Grid(I, J, K, phis=st["phis"])
        s = agcm.State(g, prec, torch_alloc=False)
        s.load(st)
        dt = 0.1 * g.dt(100.0)
        out = [s.tendency(), s.step_adjoint(lam, dt)]
        s.step(2, dt)
        out += [s.store(), s.diagnostics()]
        torch.cuda.synchronize()
        s.close()
        g.close()
        return out

    with Hook(torch.cuda.caching_allocator_alloc, torch.cuda.caching_allocator_delete) as hook:
        got = run()
        assert hook.asked and not hook.live
    want = run()
    assert all(torch.equal(a[f], b[f]) for a, b in zip(got[:3], want) for f in FIELDS) and got[3] == want[3]
    agcm.use_torch_allocator()
