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


def test_lag_planes_per_group(tmp_path):
    """(N_p, entries of the lag table, planes): us before, and by planes per group."""
    measured = [
        ((128, 3400, 33), 33.6, {2: 74.0, 4: 51.4, 8: 41.1, 16: 35.1, 32: 33.1}),
        ((128, 95256, 5), 30.6, {2: 35.0, 4: 33.0, 8: 28.7}),
        ((128, 95256, 8), 30.4, {2: 41.1, 4: 32.9, 8: 29.7, 16: 28.7}),
        ((128, 95256, 16), 34.4, {2: 59.6, 4: 42.5, 8: 34.7, 16: 30.9, 32: 30.9}),
        ((128, 95256, 33), 50.4, {2: 88.3, 4: 61.6, 8: 49.3, 16: 45.3, 32: 41.1}),
        ((128, 95256, 64), 47.4, {2: 167.9, 4: 97.8, 8: 65.0, 16: 46.2, 32: 39.1}),
        ((128, 95256, 128), 62.0, {2: 308.4, 4: 168.6, 8: 102.9, 16: 65.8, 32: 51.4}),
        ((128, 52000, 5), 28.7, {2: 34.7, 4: 31.9, 8: 28.4}),
        ((128, 52000, 8), 28.5, {2: 41.1, 4: 33.0, 8: 28.8, 16: 28.8}),
        ((128, 52000, 16), 30.9, {2: 57.6, 4: 41.2, 8: 32.9, 16: 28.9, 32: 30.9}),
        ((128, 52000, 33), 42.9, {2: 86.3, 4: 59.6, 8: 49.3, 16: 44.8, 32: 40.2}),
        ((128, 52000, 64), 41.2, {2: 160.4, 4: 94.6, 8: 63.8, 16: 45.3, 32: 39.1}),
        ((128, 52000, 128), 51.2, {2: 293.9, 4: 162.3, 8: 100.1, 16: 63.7, 32: 49.4}),
        ((128, 168480, 5), 34.4, {2: 34.5, 4: 32.7, 8: 30.4}),
        ((128, 168480, 8), 34.5, {2: 42.5, 4: 32.3, 8: 29.7, 16: 30.5}),
        ((128, 168480, 16), 40.3, {2: 61.5, 4: 43.1, 8: 35.0, 16: 30.9, 32: 35.0}),
        ((128, 168480, 33), 68.3, {2: 90.4, 4: 63.7, 8: 51.4, 16: 47.3, 32: 43.2}),
        ((128, 168480, 64), 61.8, {2: 176.8, 4: 100.7, 8: 65.8, 16: 47.3, 32: 41.2}),
        ((128, 168480, 128), 82.2, {2: 325.0, 4: 174.8, 8: 106.9, 16: 69.9, 32: 55.5}),
        ((128, 409050, 8), 46.3, {2: 45.5, 4: 34.4, 8: 32.8, 16: 36.5}),
        ((128, 409050, 16), 54.9, {2: 71.4, 4: 46.6, 8: 36.6, 16: 36.6, 32: 44.5}),
        ((128, 409050, 33), 112.8, {2: 102.6, 4: 72.4, 8: 59.6, 16: 53.4, 32: 55.5}),
        ((128, 409050, 64), 109.3, {2: 213.8, 4: 119.3, 8: 76.1, 16: 55.5, 32: 49.4}),
        ((128, 32896, 5), 36.5, {2: 40.8, 4: 36.8, 8: 36.8}),
        ((128, 32896, 8), 36.5, {2: 44.8, 4: 36.9, 8: 34.2, 16: 36.9}),
        ((128, 32896, 16), 38.7, {2: 63.7, 4: 45.2, 8: 39.1, 16: 37.1, 32: 41.2}),
        ((128, 32896, 33), 52.2, {2: 96.5, 4: 67.8, 8: 55.5, 16: 49.4, 32: 47.3}),
        ((128, 32896, 64), 57.9, {2: 169.9, 4: 102.1, 8: 69.2, 16: 52.1, 32: 46.7}),
        ((128, 32896, 128), 87.0, {2: 337.9, 4: 200.7, 8: 131.8, 16: 93.6, 32: 75.0}),
        ((128, 2664576, 8), 234.4, {2: 83.9, 4: 61.4, 8: 67.1, 16: 87.7}),
        ((128, 2664576, 33), 600.8, {2: 232.1, 4: 162.7, 8: 131.6, 16: 125.1, 32: 181.1}),
        ((64, 52000, 8), 31.0, {2: 24.8, 4: 24.8, 8: 24.8, 16: 26.8}),
        ((64, 52000, 33), 51.5, {2: 39.1, 4: 30.9, 8: 28.9, 16: 30.9, 32: 35.1}),
    ]
    got = _run(tmp_path, "epic::fx_planes_per_group(int(x[2]), int(x[0]), x[1])", 3, [m[0] for m in measured])
    for g, (case, before, by_width) in zip(got, measured):
        assert by_width[g] <= 1.05 * before, case
    assert _run(tmp_path, "epic::fx_planes_per_group(int(x[2]), int(x[0]), x[1])", 3, [(128, 10, 1), (64, 10, 1)]) == [1, 1]
