"""State kept for a device (csrc/per_device.h): work done once on one device is still to be done on
another.  The header is host code; a small program runs it here."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1708_09689_gb300", "csrc")


def _run(tmp_path, body):
    cxx = shutil.which("g++")
    if cxx is None:
        pytest.skip("no host compiler")
    src, exe = str(tmp_path / "unit.cpp"), str(tmp_path / "unit")
    with open(src, "w") as f:
        f.write('#include <cstdio>\n#include "per_device.h"\nusing namespace pvsc;\n'
                '#define CHECK(c) do { if (!(c)) { std::printf("line %d: %s\\n", __LINE__, #c); return 1; } } while (0)\n'
                "int main() {\n" + body + "\n  return 0;\n}\n")
    subprocess.run([cxx, "-std=c++17", "-Wall", "-Werror", "-I", CSRC, src, "-o", exe, "-lpthread"], check=True)
    r = subprocess.run([exe], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout


def test_a_kernel_attribute_is_set_once_per_device(tmp_path):
    _run(tmp_path, """
  OncePerDevice<int> once;
  int calls = 0, rc = 0;
  auto set = [&]() { ++calls; return rc; };
  CHECK(once.run(0, 7, set) == 0 && calls == 1);
  CHECK(once.run(0, 7, set) == 0 && calls == 1);   // done on device 0
  CHECK(once.run(1, 7, set) == 0 && calls == 2);   // not yet on device 1
  CHECK(once.run(1, 8, set) == 0 && calls == 3);
  CHECK(once.run(1, 7, set) == 0 && calls == 3);
  rc = -5;
  CHECK(once.run(2, 7, set) == -5 && calls == 4);  // a failure is not remembered
  rc = 0;
  CHECK(once.run(2, 7, set) == 0 && calls == 5);
""")
