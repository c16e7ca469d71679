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


def test_every_device_has_its_own_streams(tmp_path):
    _run(tmp_path, """
  struct Pool { int device = -1; };
  PerDevice<Pool> pools;
  int made = 0, rc = 0, dev = 0;
  auto make = [&](Pool& p) { ++made; p.device = dev; return rc; };
  Pool *a = nullptr, *b = nullptr, *c = nullptr;
  CHECK(pools.get(0, &a, make) == 0 && a->device == 0 && made == 1);
  dev = 1;
  CHECK(pools.get(1, &b, make) == 0 && b->device == 1 && made == 2 && a != b);
  CHECK(pools.get(0, &c, make) == 0 && c == a && made == 2);
  rc = -5;
  dev = 2;
  CHECK(pools.get(2, &c, make) == -5 && made == 3);  // nothing kept of a failure
  rc = 0;
  CHECK(pools.get(2, &c, make) == 0 && made == 4 && c->device == 2);
  CHECK(a->device == 0 && b->device == 1);
""")
