"""Which device-side addresses a kernel may take itself (csrc/dg_pointer.h), without a GPU: only this device's own
memory; another GPU's (no peer access), managed, host and unknown memory go through copies."""
import subprocess

import pytest

from paper_2301_11238_gb300 import build

PROGRAM = """
#include <cstdio>
#include "dg_pointer.h"
int main() {
  const cudaMemoryType types[] = {cudaMemoryTypeUnregistered, cudaMemoryTypeHost, cudaMemoryTypeDevice,
                                  cudaMemoryTypeManaged};
  for (auto t : types)
    for (int owner = 0; owner < 2; ++owner) {
      cudaPointerAttributes a{};
      a.type = t;
      a.device = owner;
      std::printf("%d", dgswe::kernel_addressable(a, 0) ? 1 : 0);
    }
}
"""


def test_only_this_devices_memory(tmp_path):
    src = tmp_path / "rule.cu"
    src.write_text(PROGRAM)
    exe = str(tmp_path / "rule")
    try:
        nvcc = build._nvcc()
    except RuntimeError:
        pytest.skip("no nvcc")
    subprocess.run([nvcc, "-std=c++17", "-I", build.CSRC, str(src), "-o", exe], check=True)
    assert subprocess.run([exe], capture_output=True, text=True, check=True).stdout == "00001000"
