"""What the launches keep per device (csrc/device_cache.h), compiled for the host
with calls that count: a second device gets its own attributes, a failed query
is asked again, a limit is only raised."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

MAIN = r"""
#include <cstdio>
#include <tuple>
#include "device_cache.h"
#define CHECK(x) do { if (!(x)) { std::printf("line %d: %s\n", __LINE__, #x); return 1; } } while (0)
int main() {
  gw::DeviceCache<std::tuple<int, long>, int> c;
  int made = 0, v = 0;
  auto ok = [&](int* p) { *p = ++made; return true; };
  auto bad = [&](int*) { ++made; return false; };
  CHECK(c.get(0, {7, 100}, &v, ok) && v == 1);
  CHECK(c.get(0, {7, 100}, &v, ok) && v == 1 && made == 1);
  CHECK(c.get(1, {7, 100}, &v, ok) && v == 2);             // another device
  CHECK(c.get(0, {7, 101}, &v, ok) && v == 3);
  CHECK(!c.get(0, {8, 100}, &v, bad) && made == 4);
  CHECK(c.get(0, {8, 100}, &v, ok) && v == 5);             // a failure is not kept
  gw::DeviceCache<int, unsigned long> r;
  int set = 0;
  auto up = [&](unsigned long) { ++set; return 0; };
  auto no = [&](unsigned long) { ++set; return 9; };
  CHECK(r.raise(0, 0, 10ul, up) == 0 && set == 1);
  CHECK(r.raise(0, 0, 9ul, up) == 0 && set == 1);          // never lowered
  CHECK(r.raise(1, 0, 9ul, up) == 0 && set == 2);          // another device
  CHECK(r.raise(0, 0, 11ul, no) == 9 && set == 3);
  CHECK(r.raise(0, 0, 11ul, up) == 0 && set == 4);
  return 0;
}
"""


def test_values_belong_to_a_device(tmp_path):
    cxx = shutil.which("g++") or shutil.which("c++")
    if not cxx:
        pytest.skip("no C++ compiler")
    (tmp_path / "m.cpp").write_text(MAIN)
    subprocess.run([cxx, "-std=c++17", "-O1", "-I" + os.path.join(ROOT, "paper_1408_3036_gb300", "csrc"),
                    str(tmp_path / "m.cpp"), "-o", str(tmp_path / "m"), "-lpthread"], check=True)
    r = subprocess.run([str(tmp_path / "m")], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout


@pytest.mark.parametrize("name", ["kernels_col.cu", "kernels_cg.cu", "kernels_tc.cu"])
def test_launch_attributes_belong_to_a_device(name):
    """cudaFuncSetAttribute holds on the current device: kept once per process it
    leaves every other device without it (one GPU here, so this reads the source)."""
    src = open(os.path.join(ROOT, "paper_1408_3036_gb300", "csrc", name)).read()
    assert "cudaFuncSetAttribute" in src and "DeviceCache<" in src
    assert "static std::mutex" not in src and "static cudaError_t attr" not in src
