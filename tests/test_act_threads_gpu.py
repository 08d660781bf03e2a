"""The shared memory that a long activation row asks for does not depend on the calls before it or beside it: host
threads quantize rows of growing length at once, in a process of its own (no earlier call has asked for the
room), and every launch is accepted.  The threads are C++ ones that start each round together: Python's own take
turns and hardly ever overlap inside the call."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

HAMMER = r"""
#include <atomic>
#include <cstdint>
#include <thread>
#include <vector>
typedef int (*act_fn)(void*, int64_t, int64_t, const float*, const float*, const float*, void*, uint8_t*, float*, int32_t*,
                      int32_t*, int32_t*, const void*);
// threads x rounds calls: in round r thread k takes a row of first + 8 (r n + k) columns; returns the refused ones
extern "C" int hammer(act_fn fn, int n, int first, int last, const float* X, void* Xq, float* h, int32_t* z, const void* cfg) {
  std::atomic<int> gate{0}, bad{0};
  const int rounds = ((last - first) / 8 + 1) / n;
  auto work = [&](int k) {
    for (int r = 0; r < rounds; ++r) {
      gate.fetch_add(1);
      while (gate.load() < n * (r + 1)) {}
      if (fn(nullptr, 1, first + 8 * (r * n + (k + r) % n), X, nullptr, nullptr, Xq, nullptr, h, z, z, z, cfg)) bad.fetch_add(1);
    }
  };
  std::vector<std::thread> ts;
  for (int k = 0; k < n; ++k) ts.emplace_back(work, k);
  for (auto& t : ts) t.join();
  return bad.load();
}
"""

SCRIPT = """
import ctypes, sys
sys.path.insert(0, %r)
import torch
from paper_2308_13137_gb300 import _lib
X, Xq = torch.randn(32768, device="cuda"), torch.empty(32768, device="cuda", dtype=torch.bfloat16)
h, z = torch.empty(4, device="cuda"), torch.empty(4, device="cuda", dtype=torch.int32)
p, cfg = lambda t: ctypes.c_void_p(t.data_ptr()), _lib.make_cfg(abits=4)
f = ctypes.cast(_lib.lib().omq_act_quant_per_token, ctypes.c_void_p)
bad = ctypes.CDLL(%r).hammer(f, 4, 10248, 32768, p(X), p(Xq), p(h), p(z), ctypes.byref(cfg))
torch.cuda.synchronize()
print("refused:", bad)
sys.exit(1 if bad else 0)
"""


def test_row_lengths_from_threads(cuda_lib, tmp_path):
    src, so = tmp_path / "hammer.cpp", tmp_path / "hammer.so"
    src.write_text(HAMMER)
    subprocess.run(["g++", "-O2", "-std=c++17", "-shared", "-fPIC", "-pthread", str(src), "-o", str(so)], check=True)
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    for _ in range(3):
        r = subprocess.run([sys.executable, "-c", SCRIPT % (root, str(so))], capture_output=True, text=True, timeout=120)
        assert r.returncode == 0, r.stdout + r.stderr
