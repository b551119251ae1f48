"""The FP64 cutoff bits that teno7_f64math.cuh decides in FP32 (it compiles for the
host too) against the FP64 evaluation: windows of every magnitude FP32 holds and
beyond, and windows next to the cutoff's thresholds."""
import shutil
import subprocess
from pathlib import Path

import pytest

ROOT = Path(__file__).resolve().parent.parent


@pytest.fixture(scope="module")
def results(tmp_path_factory):
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("no host compiler")
    exe = tmp_path_factory.mktemp("f64math") / "range_check"
    subprocess.run([gxx, "-O2", "-ffp-contract=off", "-std=c++17", "-I",
                    str(ROOT / "paper_1808_00037_gb300" / "csrc"), str(ROOT / "tests" / "f64math_range_check.cpp"),
                    "-o", str(exe)], check=True)
    out = subprocess.run([str(exe)], check=True, capture_output=True, text=True, timeout=300).stdout
    return {k: (int(n), int(bad)) for k, n, bad in (line.split() for line in out.splitlines())}


@pytest.mark.parametrize("what", ["scale", "threshold"])
def test_same_bits_as_fp64(results, what):
    n, bad = results[what]
    assert n > 100000 and bad == 0
