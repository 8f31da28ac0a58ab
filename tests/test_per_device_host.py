"""Function attributes and launch limits are prepared per device, not once per process (CPU): a second
device of a process would otherwise miss them, and its first launch would be refused."""
import os
import re
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2005_06104_gb300", "csrc")

PROGRAM = r"""
#include "common.cuh"
std::atomic<long long> g_kernel_launches{0};
int main() {
  int calls = 0;
  auto f = [&](int dev) { return once_per_device(dev, [&] { return 10 * ++calls; }); };
  bool ok = f(0) == 10 && f(1) == 20 && f(0) == 10 && f(1) == 20 && calls == 2;
  int other = 0;  // another call site has its own values
  ok = ok && once_per_device(0, [&] { return ++other; }) == 1 && calls == 2;
  int tries = 0, failed = 0, value = 0;  // a call that throws is tried again
  for (int k = 0; k < 2; ++k) {
    try {
      value = once_per_device(2, [&] { return ++tries == 1 ? throw TdvpError(TDVP_ERR_CUDA, "x") : 7; });
    } catch (const TdvpError&) {
      ++failed;
    }
  }
  ok = ok && value == 7 && failed == 1;
  bool refused = false;
  try { f(kMaxDevices); } catch (const TdvpError&) { refused = true; }
  return ok && refused ? 0 : 1;
}
"""


def test_no_attribute_is_set_once_per_process():
    for name in sorted(os.listdir(CSRC)):
        text = open(os.path.join(CSRC, name)).read()
        for m in re.finditer(r"cudaFuncSetAttribute|cudaDevAttrMultiProcessorCount", text):
            before = text[:m.start()]
            start = max(before.rfind("static const"), before.rfind("per_device("))
            inside = before[start:].count("{") > before[start:].count("}")
            assert not (inside and before[start:].startswith("static const")), (name, before[-200:])


def test_once_per_device(tmp_path):
    from paper_2005_06104_gb300 import build
    src = tmp_path / "per_device.cu"
    src.write_text(PROGRAM)
    exe = tmp_path / "per_device"
    r = subprocess.run([build._nvcc(), *build.ARCH, "-std=c++17", "-I", CSRC, "-o", str(exe), str(src)],
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    assert subprocess.run([str(exe)], timeout=60).returncode == 0
