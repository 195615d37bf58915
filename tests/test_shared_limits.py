"""The limit on a kernel's dynamic shared memory belongs to a device and to
every thread that launches there: raised on each device on its own, and never
lowered by a thread that needs less."""
import os
import re
import subprocess

import pytest

from paper_2103_10114_gb300 import agcm, inputs

PROGRAM = r"""
#include <thread>
#include <vector>
#include "agcm_host.h"
int main() {
  agcm::SharedLimits l;
  const int kernels[2] = {};
  size_t limit[2][2] = {};  // what the devices hold
  bool lowered = false;
  auto need = [&](int dev, int k, size_t n) {
    const int rc = l.raise(dev, &kernels[k], n, [&](size_t b) {
      lowered = lowered || b < limit[dev][k];
      limit[dev][k] = b;
      return 0;
    });
    return rc == 0 && limit[dev][k] >= n;
  };
  if (!need(0, 0, 1000) || !need(1, 0, 1000) || !need(0, 1, 10) || !need(0, 0, 500)) return 1;
  if (l.raise(1, &kernels[1], 9, [](size_t) { return 3; }) != 3 || !need(1, 1, 5)) return 2;  // a failure is not kept
  std::vector<std::thread> t;
  std::vector<char> ok(8, 1);
  for (int q = 0; q < 8; ++q)
    t.emplace_back([&, q] {
      for (int i = 1; i <= 2000; ++i)
        if (l.raise(0, &kernels[0], 1000 + (size_t)i * (q + 1), [&](size_t b) {
              lowered = lowered || b < limit[0][0];
              limit[0][0] = b;
              return 0;
            }))
          ok[q] = 0;
    });
  for (auto& x : t) x.join();
  for (char c : ok)
    if (!c) return 3;
  return lowered || limit[0][0] != 1000 + 2000 * 8 ? 4 : 0;
}
"""


def test_limits_are_per_device_and_only_raised(tmp_path):
    src, exe = tmp_path / "main.cpp", tmp_path / "main"
    src.write_text(PROGRAM)
    subprocess.check_call(["g++", "-std=c++17", "-pthread", "-I", agcm._CSRC, "-o", str(exe), str(src)])
    assert subprocess.run([str(exe)]).returncode == 0


def test_the_library_sets_the_attribute_in_one_place():
    text = re.sub(r"//[^\n]*", "", open(os.path.join(agcm._CSRC, "agcm_api.cu")).read())
    calls = [m.start() for m in re.finditer(r"cudaFuncSetAttribute\(", text)]
    a = text.index("cudaError_t allow_shared(")
    assert len(calls) == 1 and a < calls[0] < text.index("\n}", a)


@pytest.mark.gpu
def test_threads_with_different_level_counts(cuda_ok):
    """States whose kernels need different amounts, stepped by a thread each."""
    import threading

    import torch

    agcm.build()
    I, J = 96, 48
    errors = []

    def work(K):
        try:
            s = agcm.State(agcm.Grid(I, J, K), agcm.AGCM_FP32)
            st = inputs.random_state(I, J, K, seed=K)
            lam = inputs.random_direction(I, J, K, seed=K)
            with torch.cuda.stream(torch.cuda.Stream()):
                for _ in range(5):
                    s.load(st)
                    s.filter()
                    s.step_adjoint(lam, 1.0)
                    s.step(1, 1.0)
                torch.cuda.current_stream().synchronize()
            s.close()
        except Exception as e:  # reported by the test's own thread
            errors.append(e)

    threads = [threading.Thread(target=work, args=(K,)) for K in (3, 40, 17, 64)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors
