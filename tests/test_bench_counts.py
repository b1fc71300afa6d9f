"""What bench.py reports of a run: the kernels it launches and the bytes of its result copy."""
import os
import subprocess
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
sys.path.insert(0, ROOT)

import bench  # noqa: E402
from paper_2406_06488_gb300 import workloads  # noqa: E402


def _spec(n, stat="ed", sigma=1.0, B=100):
    return workloads.TwoSampleSpec(nx=n // 2, ny=n - n // 2, p=4, stat=stat, sigma=sigma, B=B)


def test_launches_of_a_run():
    # the launch lists in profiles/: highdim 10 kernels, the batch 11, 15 windows 97
    assert bench._kernels([_spec(5000)]) == 10
    assert bench._kernels([_spec(1024)]) == 8 and bench._kernels([_spec(1025)]) == 10
    assert bench._kernels([_spec(5000, "mmd", -1.0)]) == 16 and bench._kernels([_spec(200, "mmd", -1.0)]) == 14
    assert bench._kernels([_spec(5000, "mmd", 2.0)]) == 10
    assert bench._kernels([_spec(300), _spec(4000)]) == 11 and bench._kernels([_spec(300), _spec(400)]) == 9
    assert bench._kernels([_spec(60000)], windows=15) == 97


def test_bytes_of_the_result_copy(tmp_path):
    assert bench._result_bytes([_spec(200, B=1000)]) == 256 + 256 + 8 * 1001
    assert bench._result_bytes([_spec(200, B=10)] * 40) == 5120 + 512 + 8 * 11 * 40
    src = tmp_path / "size.cu"
    src.write_text('#include <cstdio>\n#include "ept_internal.cuh"\n'
                   'int main() { printf("%zu", sizeof(ept::Counters)); }\n')
    inc = os.path.join(ROOT, "paper_2406_06488_gb300", "csrc")
    try:
        subprocess.run([os.environ.get("NVCC", "nvcc"), "-std=c++17", "-I" + inc, "-o", str(tmp_path / "size"), str(src)],
                       check=True, capture_output=True)
    except OSError as e:
        pytest.skip("nvcc not usable here: %s" % e)
    size = subprocess.run([str(tmp_path / "size")], check=True, capture_output=True, text=True).stdout
    assert int(size) == bench.COUNTERS_BYTES
