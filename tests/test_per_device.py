"""A kernel's attributes are set once per device, not once per process: the helper that does it, on a fake of the call that
names the current device."""
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

PROGRAM = r"""
#include "per_device.h"
#include <cstdio>
static int g_dev = 0;
static cudaError_t g_answer = cudaSuccess;
extern "C" cudaError_t cudaGetDevice(int *dev) { *dev = g_dev; return g_answer; }
int main() {
  algproj::OncePerDevice once, other;
  int sets = 0;
  cudaError_t result = cudaSuccess;
  auto call = [&](algproj::OncePerDevice &o, int dev) { g_dev = dev; return o([&] { ++sets; return result; }); };
#define CHECK(cond) do { if (!(cond)) { std::printf("line %d: %s\n", __LINE__, #cond); return 1; } } while (0)
  CHECK(call(once, 0) == cudaSuccess && sets == 1);
  CHECK(call(once, 0) == cudaSuccess && sets == 1);
  CHECK(call(once, 1) == cudaSuccess && sets == 2);    // a second device gets its own
  CHECK(call(once, 63) == cudaSuccess && sets == 3);
  CHECK(call(once, 1) == cudaSuccess && call(once, 63) == cudaSuccess && sets == 3);
  CHECK(call(other, 0) == cudaSuccess && sets == 4);   // and every kernel
  CHECK(call(once, 64) == cudaSuccess && call(once, 64) == cudaSuccess && sets == 6);
  result = cudaErrorInvalidValue;
  CHECK(call(once, 2) == result && call(once, 2) == result && sets == 8);   // not done while it fails
  result = cudaSuccess;
  CHECK(call(once, 2) == cudaSuccess && call(once, 2) == cudaSuccess && sets == 9);
  g_answer = cudaErrorNoDevice;
  CHECK(call(once, 3) == cudaErrorNoDevice && sets == 9);
  return 0;
}
"""


def test_attributes_are_set_once_per_device(tmp_path):
    src, exe = tmp_path / "p.cpp", tmp_path / "p"
    src.write_text(PROGRAM)
    cuda = os.environ.get("CUDA_HOME", "/usr/local/cuda")
    subprocess.check_call(["g++", "-std=c++17", "-I", os.path.join(ROOT, "paper_2609_32814_b200", "csrc"), "-I", os.path.join(cuda, "include"),
                           str(src), "-o", str(exe)])
    out = subprocess.run([str(exe)], capture_output=True, text=True)
    assert out.returncode == 0, out.stdout


def test_no_launcher_remembers_an_attribute_for_the_process():
    """Every cudaFuncSetAttribute either runs on each launch or inside a OncePerDevice."""
    csrc = os.path.join(ROOT, "paper_2609_32814_b200", "csrc")
    for name in sorted(os.listdir(csrc)):
        text = open(os.path.join(csrc, name)).read()
        assert "static bool attr" not in text, name
