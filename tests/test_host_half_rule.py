"""The rules that choose between the two forms at N_p = 256 (no GPU): compiled from the library's own header and held
against measured times.  A call must not be sent to the half-image kernels where the clusters, which took every call
before them, were more than 5 % faster."""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1510_08318_gb300", "csrc")

# (mapping entries, samples, channels): us forward in halves, in clusters; us adjoint in halves, in clusters (152 SMs)
MEASURED = {
    (331, 38, 1): (41.3, 36.5, 34.6, 40.1), (331, 76, 1): (58.7, 43.6, 35.8, 54.9),
    (331, 152, 1): (70.4, 60.1, 56.9, 85.1), (331, 228, 1): (79.5, 75.1, 77.5, 114.8),
    (331, 608, 1): (139.2, 151.1, 184.1, 263.5), (331, 1, 152): (95.6, 109.3, 62.7, 102.7),
    (331, 4, 38): (59.5, 70.2, 57.7, 89.4), (331, 128, 4): (118.3, 134.8, 164.8, 232.5),
    (2979, 60, 1): (49.6, 37.4, 36.2, 41.2), (2979, 304, 1): (94.6, 88.7, 102.3, 148.6),
    (2979, 1, 76): (47.7, 68.0, 38.2, 66.9), (16219, 152, 1): (76.4, 62.1, 75.6, 101.6),
    (16219, 160, 1): (74.1, 62.1, 106.5, 102.4), (16219, 608, 1): (153.2, 160.7, 259.9, 319.9),
    (40051, 140, 1): (70.0, 64.1, 100.2, 110.2), (40051, 608, 1): (172.4, 200.4, 358.4, 427.6),
    (50176, 76, 1): (63.4, 56.3, 69.7, 93.4), (50176, 160, 1): (96.3, 80.5, 174.5, 148.2),
    (50176, 240, 1): (109.7, 105.0, 227.4, 201.4), (50176, 608, 1): (187.7, 222.6, 441.4, 468.1),
    (74475, 76, 1): (63.4, 76.4, 81.9, 119.7), (74475, 160, 1): (98.6, 113.5, 219.1, 193.3),
    (74475, 608, 1): (203.5, 335.1, 561.3, 627.7), (230400, 76, 1): (80.9, 230.0, 191.3, 274.7),
    (230400, 160, 1): (151.4, 370.6, 538.6, 450.1), (230400, 608, 1): (331.4, 1209.4, 1420.6, 1509.1),
    (297900, 76, 1): (84.4, 316.5, 211.2, 372.8), (297900, 304, 1): (212.2, 908.2, 804.7, 1094.6),
}
# the same forward, where sums begin and end in the middle of a worker's share
MEASURED_FWD = {
    (1525, 38, 4): (61.6, 57.6),
    (1525, 14, 13): (82.1, 67.0),
    (6775, 30, 4): (55.5, 52.5),
    (6775, 22, 5): (70.4, 54.6),
    (6775, 29, 5): (72.6, 61.8),
    (6775, 20, 6): (70.4, 52.1),
    (6775, 24, 6): (71.3, 53.5),
    (6775, 76, 8): (153.1, 160.0),
    (6775, 35, 13): (126.7, 123.5),
    (6775, 7, 16): (71.4, 54.6),
    (6775, 38, 16): (154.2, 161.3),
    (9216, 152, 4): (145.1, 160.4),
    (9216, 5, 24): (71.9, 55.6),
    (74475, 20, 6): (84.4, 94.6),
}
# far enough apart that the halves have to be taken: where they save more than a fifth of the call
CLEAR = 0.8


def _compiled(tmp_path_factory, body):
    cxx = shutil.which("g++") or shutil.which("c++")
    if cxx is None:
        pytest.skip("no C++ compiler")
    d = tmp_path_factory.mktemp("rule")
    src, exe = str(d / "rule.cpp"), str(d / "rule")
    with open(src, "w") as f:
        f.write('#include "half_rule.h"\n#include <cstdio>\nint main() {\n    long long e, n, c, m, o;\n%s}\n' % body)
    subprocess.run([cxx, "-std=c++17", "-I" + CSRC, "-o", exe, src], check=True)
    return exe


@pytest.fixture(scope="module")
def rule(tmp_path_factory):
    exe = _compiled(tmp_path_factory, '    while (std::scanf("%lld %lld %lld", &e, &n, &c) == 3)\n'
                    '        std::printf("%d %d\\n", epic::half_pays_fwd(n, 152, double(e), c), '
                    'epic::half_pays_bwd(n, 152, double(e)));\n')
    cases = list(MEASURED) + list(MEASURED_FWD)
    text = "".join("%d %d %d\n" % (e, t * c, c) for e, t, c in cases)
    out = subprocess.run([exe], input=text, capture_output=True, text=True, check=True).stdout.split()
    return {k: (out[2 * i] == "1", out[2 * i + 1] == "1") for i, k in enumerate(cases)}


@pytest.mark.parametrize("case", list(MEASURED), ids=lambda c: "x".join(map(str, c)))
def test_choice(rule, case):
    for half, (h, c) in zip(rule[case], (MEASURED[case][:2], MEASURED[case][2:])):
        assert (h if half else c) <= 1.05 * c
        if h < CLEAR * c and case[1] * case[2] > 38:
            assert half


@pytest.mark.parametrize("case", list(MEASURED_FWD), ids=lambda c: "x".join(map(str, c)))
def test_choice_by_sums(rule, case):
    h, c = MEASURED_FWD[case]
    assert (h if rule[case][0] else c) <= 1.05 * c


@pytest.mark.parametrize("items, n_ent, n_cp, cap, one_buffer, want", [
    (4096, 3000, 32, 0, 0, (1, 0)),          # no cap
    (4096, 3000, 32, 76, 0, (1, 76)),        # half images on 76 SMs
    (4096, 3000, 32, 76, 1, (0, 19)),        # the same SMs as clusters of four
    (4096, 3000, 32, 114, 1, (0, 28)),
    (30, 3000, 1, 114, 0, (0, 28)),          # few images: clusters
    (30, 3000, 1, 3, 0, (0, 1)),
    (30, 3000, 1, 0, 0, (0, 0)),
    (76, 3000, 19, 0, 0, (1, 0)),            # one wave of halves on 152 SMs, two on 76
    (76, 3000, 19, 76, 0, (1, 76)),
    (77, 3000, 4, 76, 0, (0, 19)),           # three waves of halves and five of clusters
    (1 << 30, 3000, 32, 0, 0, (0, 0)),       # too many half images to number
])
def test_cap_in_sms(tmp_path_factory, items, n_ent, n_cp, cap, one_buffer, want):
    """A launch is capped in SMs, whichever form it takes, and the rule counts the SMs under the cap."""
    exe = _compiled(tmp_path_factory, '    std::scanf("%lld %lld %lld %lld %lld", &n, &e, &c, &m, &o);\n'
                    '    const epic::HalfChoice f = epic::half_choice(n, 152, double(e), c, int(m), o != 0);\n'
                    '    std::printf("%d %d\\n", f.half, f.cap);\n')
    out = subprocess.run([exe], input="%d %d %d %d %d" % (items, n_ent, n_cp, cap, one_buffer), capture_output=True,
                         text=True, check=True).stdout.split()
    assert tuple(map(int, out)) == want
