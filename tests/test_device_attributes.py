"""Kernel attributes are set once per thread and device (a thread may drive
handles on several devices): the set of prepared devices, and that every
launcher goes through it (CPU)."""
import os
import re
import subprocess

import paper_1905_00689_gb300 as package

CSRC = os.path.join(os.path.dirname(package.__file__), "csrc")

PROGRAM = """
#include "device_set.h"
int main() {
  lstm_approx_impl::DeviceSet s;
  if (s.has(0) || s.has(63) || s.has(-1)) return 1;
  s.add(0);
  if (!s.has(0) || s.has(1) || s.has(64)) return 2;   // a second device is not prepared by the first
  s.add(63);
  if (!s.has(63) || s.has(62) || !s.has(0)) return 3;
  s.add(64);
  s.add(-1);
  return s.has(64) || s.has(1) || s.has(-1) ? 4 : 0;
}
"""


def test_device_set(tmp_path):
    (tmp_path / "p.cpp").write_text(PROGRAM)
    subprocess.run(["g++", "-std=c++17", "-I", CSRC, str(tmp_path / "p.cpp"), "-o", str(tmp_path / "p")], check=True)
    assert subprocess.run([str(tmp_path / "p")]).returncode == 0


def test_every_launcher_sets_attributes_per_device():
    sites = 0
    for name in sorted(os.listdir(CSRC)):
        with open(os.path.join(CSRC, name)) as f:
            text = f.read()
        assert not re.search(r"static thread_local bool", text), name
        for m in re.finditer(r"cudaFuncSetAttribute", text):
            sites += 1
            # inside a once_per_device call, or (k_dense.cu) on every launch
            before = text[text.rindex("template <", 0, m.start()) if "template <" in text[:m.start()] else 0:m.start()]
            assert "once_per_device" in before or name == "k_dense.cu", (name, m.start())
    assert sites >= 10
