"""The reductions over CTAs refuse, at compile time, more values than their slots hold."""
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_2403_09133_gb300", "csrc")

SOURCE = r"""
#include "lorads_device.cuh"
__global__ void k(lorads::GridScope s, double* v) {
  s.init();
  s.reduce<VALUES>(v);
  s.reduce_each<VALUES>(v, [=](int i, double x) { v[i] = x; });
}
"""


@pytest.mark.parametrize("values", ["SLOT", "SLOT + 1"])
def test_more_values_than_slots_do_not_compile(tmp_path, values):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("no nvcc")
    src = tmp_path / "k.cu"
    src.write_text(SOURCE.replace("VALUES", values.replace("SLOT", "lorads::SLOT_VALUES")))
    r = subprocess.run([nvcc, "-std=c++17", "-gencode", "arch=compute_103a,code=sm_103a", "-I",
                        CSRC, "-c", str(src), "-o", str(tmp_path / "k.o")], capture_output=True,
                       text=True)
    if values == "SLOT":
        assert r.returncode == 0, r.stderr
    else:
        assert r.returncode != 0 and "a set of slots holds a reduction's values" in r.stderr
