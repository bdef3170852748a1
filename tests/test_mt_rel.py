"""The visibility rays' relative FP32 pre-test (``mt_rel_classify``) never
contradicts the FP64 test, on the 1.6M seeded, mostly adversarial segments of
``mt_pretest_check.cpp`` (CPU only), and leaves less undecided than the
pre-test over absolute coordinates, which is what it is for."""
import os
import re
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CUDA_INC = os.path.join(os.environ.get("CUDA_HOME", "/usr/local/cuda"), "include")


def run(tmp_path, source):
    exe = tmp_path / source.replace(".cpp", "")
    subprocess.run([shutil.which("g++"), "-O2", "-ffp-contract=off", "-std=c++17",
                    "-I", os.path.join(ROOT, "include"), "-I", os.path.join(ROOT, "tests"),
                    "-I", os.path.join(ROOT, "paper_2208_10939_gb300", "csrc"), "-I", CUDA_INC,
                    os.path.join(ROOT, "tests", source), "-o", str(exe)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=300)
    m = re.search(r"cases (\d+) violations (\d+) decided (\d+)", r.stdout)
    assert m, r.stdout + r.stderr
    return tuple(map(int, m.groups())) + (r.stdout,)


def test_relative_pretest_decides_only_what_fp64_decides(tmp_path):
    if shutil.which("g++") is None or not os.path.exists(os.path.join(CUDA_INC, "cuda_runtime.h")):
        pytest.skip("g++ or the CUDA headers are missing")
    cases, violations, decided, out = run(tmp_path, "mt_rel_check.cpp")
    assert cases == 1_600_000 and violations == 0, out
    assert decided > run(tmp_path, "mt_pretest_check.cpp")[2]
