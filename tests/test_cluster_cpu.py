"""The rule that steps a thread-block cluster down to what a device can hold,
against a stand-in for the device (CPU)."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

SOURCE = """
#include "cluster.h"
#include <cstdio>
int main()
{
    for (int want = 1; want <= 16; want *= 2)
        for (int most = 0; most <= 16; ++most)   // a device that holds `most` CTAs, or answers with an error (0)
            std::printf("%d %d %d\\n", want, most,
                        mg::cluster_step_down(want, [&](int c) { return c <= most; }));
}
"""


def test_cluster_steps_down_to_what_is_resident(tmp_path):
    cxx = shutil.which("g++") or shutil.which("c++")
    if cxx is None:
        pytest.skip("no C++ compiler")
    src, exe = tmp_path / "rule.cpp", tmp_path / "rule"
    src.write_text(SOURCE)
    subprocess.run([cxx, "-std=c++17", "-I" + os.path.join(ROOT, "paper_1008_2801_gb300", "csrc"),
                    str(src), "-o", str(exe)], check=True)
    out = subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout
    rows = [tuple(map(int, r.split())) for r in out.splitlines()]
    assert len(rows) == 5 * 17
    for want, most, got in rows:
        assert got == max([c for c in (1, 2, 4, 8, 16) if c <= min(want, most)], default=1)
