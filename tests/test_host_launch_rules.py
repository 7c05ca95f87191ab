"""The rules by which launches choose between kernel variants (no GPU): compiled from the library's own header and held
against measured times.  A call must not get a variant with which it takes more than 5 % longer than in the form that
took every such call before the variants."""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1510_08318_gb300", "csrc")


def _run(tmp_path, expr, n_arg, rows):
    """expr, over long long x[0], x[1], ..., of each row of whole numbers."""
    cxx = shutil.which("g++") or shutil.which("c++")
    if cxx is None:
        pytest.skip("no C++ compiler")
    src, exe = str(tmp_path / "rule.cpp"), str(tmp_path / "rule")
    with open(src, "w") as f:
        f.write('#include "launch_rules.h"\n#include <cstdio>\nint main() {\n    long long x[16];\n    for (;;) {\n'
                '        for (int i = 0; i < %d; ++i)\n            if (std::scanf("%%lld", x + i) != 1) return 0;\n'
                '        std::printf("%%lld\\n", (long long)(%s));\n    }\n}\n' % (n_arg, expr))
    subprocess.run([cxx, "-std=c++17", "-I" + CSRC, "-o", exe, src], check=True)
    text = "\n".join(" ".join(map(str, r)) for r in rows)
    return [int(v) for v in subprocess.run([exe], input=text, capture_output=True, text=True, check=True).stdout.split()]


def test_correlator_roles(tmp_path):
    """(FP16, samples): us before, in the short and in the long form (antennas, (channel, pol) varied, 152 SMs)."""
    measured = [((1, 64), (16.6, 16.8, 22.7)), ((1, 96), (18.6, 18.6, 22.7)), ((1, 96), (43.3, 28.8, 33.0)),
                ((1, 96), (65.4, 47.3, 65.3)), ((1, 128), (12.5, 12.4, 16.5)), ((1, 256), (100.6, 64.8, 78.4)),
                ((1, 384), (78.1, 65.1, 62.0)), ((1, 512), (154.9, 103.2, 103.7)),
                ((1, 1024), (285.3, 184.7, 183.2)), ((0, 64), (39.3, 26.8, 30.9)),
                ((0, 128), (47.3, 37.0, 39.1)), ((0, 128), (58.3, 56.8, 71.7)), ((0, 192), (39.0, 37.0, 41.1)),
                ((0, 256), (86.7, 89.7, 82.8)), ((0, 1024), (129.5, 130.9, 108.6)),
                ((0, 1024), (216.0, 213.0, 168.4))]
    got = _run(tmp_path, "epic::xeng_short(x[0] != 0, int(x[1]))", 2, [m[0] for m in measured])
    for short, (case, (before, t_short, t_long)) in zip(got, measured):
        assert (t_short if short else t_long) <= 1.05 * before, case
