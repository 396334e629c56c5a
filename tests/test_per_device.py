"""Function attributes are set once per device: the host helper, against a fake of the call that sets them."""
import os
import subprocess

from paper_2608_13076_gb300 import _build

PROGRAM = r"""
#include <cstdio>
#include "per_device.h"
int main() {
  static spade::OncePerDevice once;
  int set[2] = {0, 0}, other = 0;
  bool ok = true;
  for (int pass = 0; pass < 3; ++pass)
    for (int dev = 0; dev < 2; ++dev) ok &= once(dev, [&] { ++set[dev]; return 0; }) == 0;
  ok &= set[0] == 1 && set[1] == 1;
  // a failed call is made again, and its error comes back
  int calls = 0;
  ok &= once(2, [&] { ++calls; return 7; }) == 7;
  ok &= once(2, [&] { ++calls; return 0; }) == 0;
  ok &= once(2, [&] { ++calls; return 0; }) == 0 && calls == 2;
  // past the table: nothing is remembered
  for (int i = 0; i < 2; ++i) ok &= once(spade::kMaxDevices, [&] { ++other; return 0; }) == 0;
  ok &= other == 2;
  puts(ok ? "ok" : "wrong");
}
"""


def test_once_per_device(tmp_path):
    src, exe = tmp_path / "t.cpp", tmp_path / "t"
    src.write_text(PROGRAM)
    subprocess.run([os.environ.get("CXX", "g++"), "-std=c++17", "-I", _build.CSRC, str(src), "-o", str(exe)], check=True)
    assert subprocess.run([str(exe)], capture_output=True, text=True).stdout == "ok\n"


def test_every_launcher_uses_it():
    """No source sets the attribute by itself, under a flag for the whole process."""
    for path in _build.sources():
        with open(path) as f:
            text = f.read()
        assert "cudaFuncAttributeMaxDynamicSharedMemorySize" not in text and "static bool configured" not in text, path
