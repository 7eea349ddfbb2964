"""The tuner's input field.  The FP64 transforms' time depends on the values: a line of zeros takes the
careful conversion of its results.  ``lsm_autotune`` reads nothing from the caller and returns only the
variants it kept, so its source is checked: the field is the white field of csrc/common.cuh, written
before anything is timed; and that field is checked by value, compiled for the host.
"""
import os
import re
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_2301_12836_gb300", "csrc")


def _body(text, head):
    i = text.index("{", text.index(head))
    depth, j = 1, i + 1
    while depth:
        depth += {"{": 1, "}": -1}.get(text[j], 0)
        j += 1
    return text[i:j]


def test_timed_on_the_white_field():
    text = re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, "lsm.cu")).read())
    tune, top = _body(text, "static lsm_status tune_one("), _body(text, 'extern "C" lsm_status lsm_autotune(')
    assert "cudaMemset" not in tune + top
    assert tune.index("launch_white((T*)u, 6 * s->d.N") < tune.index("launch_apply<T>(")


@pytest.mark.skipif(shutil.which("g++") is None, reason="needs a host compiler")
def test_white_field_values(tmp_path):
    src = tmp_path / "white.cpp"
    src.write_text('''#include "common.cuh"
#include <cstdio>
int main() {
    const int n = 1 << 20;
    double s = 0, q = 0, c = 0, prev = 0, top = 0;
    int zeros = 0;
    for (int i = 0; i < n; ++i) {
        const double v = lsm::white(i);
        s += v, q += v * v, c += v * prev;
        top = std::max(top, std::fabs(v));
        zeros += (float)v == 0.0f;
        prev = v;
    }
    std::printf("%d %.6f %.6f %.6f %.9f\\n", zeros, s / n, q / n, c / n, top);
}
''')
    exe = str(tmp_path / "white")
    subprocess.run(["g++", "-std=c++17", "-O1", "-w", "-I", os.path.join(HERE, "host"), "-I", CSRC, str(src), "-o", exe], check=True)
    zeros, mean, var, corr, top = (float(v) for v in subprocess.run([exe], check=True, capture_output=True, text=True).stdout.split())
    # standard errors of the three averages at 2^20 samples: 0.00056, 0.00029, 0.00033; five of each
    assert zeros == 0 and abs(mean) < 0.0029 and abs(var - 1 / 3) < 0.0015 and abs(corr) < 0.0017 and top < 1
