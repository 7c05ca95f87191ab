"""Host logic of the gridding by cell pairs (no GPU): the tables that the library's own builders make for the
tensor-core form at N_p = 128, the half-image kernels at 256 and the two-pass form at 512, walked as the kernels walk
them; see tests/host/pair_tables_check.cu for what is checked.  Mappings: dense and sparse, complex weights, a ragged
grid, many antennas, nearly empty ones, and one antenna in the grid's corners."""
import os
import shutil
import subprocess

import numpy as np
import pytest

from oracle import moff
from paper_1510_08318_gb300 import synth

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
NVCC = shutil.which("nvcc") or ("/usr/local/cuda/bin/nvcc" if os.path.exists("/usr/local/cuda/bin/nvcc") else None)


@pytest.fixture(scope="module")
def checker(tmp_path_factory):
    if NVCC is None:
        pytest.skip("nvcc not available")
    out = str(tmp_path_factory.mktemp("pt") / "pair_tables_check")
    cmd = [NVCC, "-std=c++17", "--expt-relaxed-constexpr", "-gencode", "arch=compute_103a,code=sm_103a",
           "-o", out, os.path.join(ROOT, "tests", "host", "pair_tables_check.cu")]
    r = subprocess.run(cmd, capture_output=True, text=True)
    assert r.returncode == 0, r.stderr[-2000:]
    return out


def _mapping(case, side):
    """n_grid and the mapping of one layout on a grid of at most side x side cells."""
    rng = np.random.default_rng(side)
    n_grid = {"ragged": side - 27}.get(case, side)
    n_ant = {"many": 1400, "few": 3, "one": 1, "dense": 40}.get(case, 150)
    pos = rng.uniform(1.5, n_grid - 2.5, (n_ant, 2))
    kerns = [synth.kernel_square(rng.uniform(0.5, 2.5), 1 / 3) for _ in range(n_ant)]
    if case == "dense":
        pos = rng.uniform(13.0, n_grid - 14.0, (n_ant, 2))
        kerns = [synth.kernel_square(24.0, 1.0)] * n_ant
    if case == "one":
        pos, kerns = np.zeros((1, 2)), [synth.kernel_point()]
    if case == "corners":
        pos[:4] = [[0, 0], [n_grid - 1, 0], [0, n_grid - 1], [n_grid - 1, n_grid - 1]]
        kerns[:4] = [synth.kernel_point()] * 4
    ptr, dxdy, w = synth.pack_kernels(kerns)
    if case == "complex":
        w = w * np.exp(1j * rng.uniform(0, 2 * np.pi, w.shape))
    return n_grid, moff.map_antennas(pos, ptr, dxdy, w, 1.0, np.zeros(2), n_grid)


@pytest.mark.parametrize("side", [64, 128, 256])
@pytest.mark.parametrize("case", ["plain", "complex", "ragged", "many", "dense", "few", "one", "corners"])
def test_every_entry_once(checker, tmp_path, case, side):
    n_grid, M = _mapping(case, side)
    M = M.tocsr()
    M.sort_indices()
    rows = np.repeat(np.arange(M.shape[0]), np.diff(M.indptr))
    cell = (rows // n_grid) * side + rows % n_grid
    order = np.argsort(cell, kind="stable")
    ptr = np.concatenate([[0], np.cumsum(np.bincount(cell, minlength=side * side))])
    path = str(tmp_path / "map.txt")
    with open(path, "w") as f:
        f.write("%d %d\n" % (side * side, M.nnz))
        f.write(" ".join(map(str, ptr)) + "\n")
        f.write(" ".join(map(str, M.indices[order])) + "\n")
        f.write(" ".join("%.9g" % v for v in np.float32(M.data.real[order])) + "\n")
        f.write(" ".join("%.9g" % v for v in np.float32(M.data.imag[order])) + "\n")
    r = subprocess.run([checker, path], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout + r.stderr
