"""Arithmetic that host planning and device code share, compiled for the host, at the ends of its range."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

COPY_END = r"""
#include <cstdio>
#include "tc_conv_plan.h"
int main() {
    for (long long x_end : {5ll, 4096ll, 2147483640ll, 2147483645ll, 2147483646ll, 2147483647ll}) {
        const int x_whole = (int)(x_end & ~3ll);
        for (long long last = x_end > 40 ? x_end - 40 : 1; last <= x_end; ++last) {
            const long long up = (last + 3) & ~3ll, want = up < x_whole ? up : x_whole;
            const int got = onnxb::fp32_conv_copy_end((int)last, x_whole);
            if (got != want) return std::printf("%lld of %lld: %d, not %lld\\n", last, x_end, got, want), 1;
        }
    }
    return 0;
}
"""


@pytest.mark.skipif(shutil.which("g++") is None, reason="no host compiler")
def test_copies_end_inside_x(tmp_path):
    (tmp_path / "t.cpp").write_text(COPY_END)
    csrc = os.path.join(ROOT, "paper_2008_08272_b200", "csrc")
    subprocess.run(["g++", "-std=c++17", "-fsanitize=signed-integer-overflow", "-fno-sanitize-recover", "-I" + csrc, str(tmp_path / "t.cpp"), "-o",
                    str(tmp_path / "t")], check=True)
    run = subprocess.run([str(tmp_path / "t")], capture_output=True, text=True)
    assert run.returncode == 0, run.stdout + run.stderr
