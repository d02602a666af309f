"""Host rules of the launches, compiled with the host compiler.

Clusters of 16 CTAs are beyond the size that every device takes: the launch class of a system's
outputs is the largest one that fits the device, down to single CTAs.
"""
import os
import re
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2403_10343_gb300", "csrc")


def run(tmp_path, body):
    cxx = shutil.which("g++")
    if cxx is None:
        pytest.skip("no host C++ compiler")
    src, exe = tmp_path / "r.cc", tmp_path / "r"
    src.write_text(f'#include <cstdio>\n#include <initializer_list>\n#include "rix_rules.h"\nusing namespace rix;\nint main() {{\n{body}\n}}\n')
    subprocess.run([cxx, "-std=c++17", "-I", CSRC, str(src), "-o", str(exe)], check=True)
    return [int(x) for x in subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout.split()]


def test_class_is_capped_by_what_fits(tmp_path):
    got = run(tmp_path, 'for (int most : {16, 8, 4, 1})\n  for (int want = 0; want < 5; want++)\n'
                        '    printf("%d ", fitting_class(want, [&](int n) { return n <= most; }));')
    assert got == [0, 1, 2, 3, 4, 0, 1, 2, 3, 3, 0, 1, 2, 2, 2, 0, 0, 0, 0, 0]


def test_class_follows_the_longest_output(tmp_path):
    # one output of n equal ones: an even share of the 152 SMs holds n / 152 of them
    got = run(tmp_path, 'for (double n : {1.0, 20.0, 40.0, 100.0, 303.0, 304.0})\n'
                        '  printf("%d ", cluster_class(1.0, n, 4));')
    assert got == [4, 4, 3, 2, 1, 0]


def test_one_name_for_the_number_of_SMs():
    for f in sorted(os.listdir(CSRC)):
        for line in open(os.path.join(CSRC, f)):
            code = line.split("//")[0]
            assert f == "rix_rules.h" or not re.search(r"\b152\b", code), (f, line)
