"""Programmatic dependent launches: their error handling, on the CPU."""
import os
import re
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
PKG = os.path.join(ROOT, "paper_2406_13651_gb300")
NVCC = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"

# launch_after against a runtime (fakes.cpp) that refuses every second launch with status 9.
CALLS = r"""
#include "clamp_kernels.cuh"
#include <cstdio>
extern int last;
void kernel(int) {}
int main() {
  const cudaError_t a = clamp::launch_after(kernel, dim3(1), 256, 0, (cudaStream_t)0, 1);
  std::printf("%d %d ", (int)a, last);
  const cudaError_t b = clamp::launch_after(kernel, dim3(1), 256, 0, (cudaStream_t)0, 1);
  std::printf("%d %d\n", (int)b, last);
  return 0;
}
"""
FAKES = r"""
int last = 0;
static int launches = 0;
extern "C" int cudaLaunchKernelExC(const void*, const void*, void**) {
  const int e = launches++ % 2 ? 0 : 9;
  if (e) last = e;
  return e;
}
extern "C" int cudaGetLastError() {
  const int e = last;
  last = 0;
  return e;
}
"""


def test_refused_launch_is_reported_once(tmp_path):
    if not os.path.exists(NVCC):
        pytest.skip("no nvcc")
    (tmp_path / "calls.cu").write_text(CALLS)
    (tmp_path / "fakes.cpp").write_text(FAKES)
    exe = str(tmp_path / "calls")
    r = subprocess.run([NVCC, "-gencode=arch=compute_103a,code=sm_103a", "-std=c++17", "-cudart", "shared",
                        "-Xlinker", "-rpath,/usr/local/cuda/lib64",
                        "-I" + os.path.join(ROOT, "include"), "-I" + os.path.join(PKG, "csrc"), "-o", exe,
                        str(tmp_path / "calls.cu"), str(tmp_path / "fakes.cpp")], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    out = subprocess.run([exe], capture_output=True, text=True, timeout=120)
    assert out.stdout.split() == ["9", "0", "0", "0"], out.stdout   # the refusal, and no error left for the next call


# What a kernel of such a chain may read through the non-coherent path (__ldg): data that nothing in the
# chain writes.  The kernel may be resident while the one before it still runs, and only what is read-only for as
# long as it is resident may be read so.
READ_ONLY = ("a.t.", "a.window", "c.window", "tw")


def _bodies(text):
    """Bodies of the functions that call after_previous()."""
    at = 0
    while (at := text.find("  after_previous();", at)) >= 0:
        depth, end = 1, at
        while depth:
            depth += {"{": 1, "}": -1}.get(text[end], 0)
            end += 1
        yield text[at:end]
        at = end


def test_dependent_kernels_read_the_chains_data_coherently():
    seen = 0
    for name in sorted(os.listdir(os.path.join(PKG, "csrc"))):
        with open(os.path.join(PKG, "csrc", name)) as f:
            for body in _bodies(f.read()):
                seen += 1
                for arg in re.findall(r"__ldg\(\s*&?\s*([\w.\->]+)", body):
                    assert arg.startswith(READ_ONLY), (name, arg)
    assert seen >= 5   # the band passes and the fused pass
