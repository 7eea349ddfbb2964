"""Range and accuracy of the FP64 transforms' fixed-point engines (csrc/fx.cuh), line by line on the CPU:
``host/lines.cpp`` compiles the kernels' own headers for the host and runs a line's threads in turn.

* Accuracy: the fixed-point engine replaces an FP64 engine, so its rms error against long double may
  be no larger than that of the same plan in FP64, on forward lines of six kinds of fields and on
  inverse lines of their spectra times a Green spectrum, at 10 and 25 nodes per wave.
* Range: no sum and no factor leaves its words on lines at the full scale, aligned with each
  frequency in turn so that the whole headroom is used.
* Outputs that cancel exactly are zero, and conversions give the nearest FP64 value down to the
  smallest subnormal.
"""
import os
import platform
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_2301_12836_gb300", "csrc")

pytestmark = pytest.mark.skipif(shutil.which("g++") is None, reason="needs a host compiler")


@pytest.fixture(scope="module")
def lines(tmp_path_factory):
    """Rows (as lists of words) of `lines <what>`."""
    exe = str(tmp_path_factory.mktemp("lines") / "lines")
    fma = []   # the FP64 yardstick uses fused multiply-adds, as the GPU does
    if platform.machine() == "x86_64" and "fma" in open("/proc/cpuinfo").read().split():
        fma = ["-mfma"]
    subprocess.run(["g++", "-std=c++17", "-O2", "-w", "-ffp-contract=fast", *fma, "-I", os.path.join(HERE, "host"), "-I", CSRC,
                    os.path.join(HERE, "host", "lines.cpp"), "-o", exe], check=True)

    def run(what):
        out = subprocess.run([exe, what], check=True, capture_output=True, text=True).stdout
        return [r.split() for r in out.splitlines()]
    return run


def test_accuracy_no_worse_than_fp64(lines):
    rows = lines("accuracy")
    assert len(rows) >= 37 * 12
    worse = [r for r in rows if float(r[3]) > float(r[4])]
    assert not worse, worse


def test_full_scale_lines_stay_in_range(lines):
    rows = lines("range")
    assert len(rows) >= 37 * 4
    assert all(int(r[4]) == 0 for r in rows), rows


def test_exact_cancellations_are_zero(lines):
    rows = lines("zeros")
    assert len(rows) >= 37 * 2
    assert all(int(r[2]) == 0 for r in rows), rows


def test_conversion_to_fp64_is_nearest(lines):
    (bad, subnormal), = lines("convert")
    assert int(subnormal) > 5000
    assert int(bad) == 0
