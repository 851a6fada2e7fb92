"""CPU check of the path kernels' step-cap test, which lets a lane take a whole
visit of steps without looking at the cap: exact up to the largest cap that
pdds_set_step_cap takes (2^31 - 1; larger defaults are cut to it), where the sum
of the steps taken and those ahead no longer fits 32 bits.  A wrapped sum would
let a path that never leaves its patch step on for ever."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
TOP = 2 ** 31 - 1


def test_step_cap_is_exact_up_to_the_largest_cap(tmp_path):
    cxx = shutil.which("g++")
    if cxx is None or not os.path.isdir("/usr/local/cuda/include"):
        pytest.skip("needs g++ and the CUDA headers")
    exe = str(tmp_path / "probe")
    subprocess.run([cxx, "-std=c++17", "-O2", "-I", "/usr/local/cuda/include", "-I",
                    os.path.join(ROOT, "paper_2301_05780_gb300", "csrc"), "-I",
                    os.path.join(ROOT, "include"), os.path.join(ROOT, "tests", "step_cap_probe.cpp"),
                    "-o", exe], check=True)
    cases = [(n, more, kmax) for kmax in (1, 2, 17, 1000, TOP - 1, TOP) for more in (4, 16, 64)
             for n in {0, kmax // 2, *(kmax - d for d in (1, 3, 4, 5, 15, 16, 17, 63, 64, 65, 66))}
             if 0 <= n < kmax]
    inp = "".join(f"{n} {m} {k}\n" for n, m, k in cases)
    out = subprocess.run([exe], input=inp, capture_output=True, text=True, check=True).stdout
    assert [int(x) for x in out.split()] == [int(n + m < k) for n, m, k in cases]
