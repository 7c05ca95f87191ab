"""The transforms that bench.py's cross-polarisation mode asks for exist at its plan's size with those products (CPU
only): the library refuses the reduced-precision and the N_p = 256 forms there."""
import bench
from paper_1510_08318_gb300 import epic


def test_cross_polarisation_forms():
    assert [xf for _, xf in bench.XPOL_FORMS] == ["fft", "dftgemm"]
    assert all(xf in epic.XFORMS for _, xf in bench.XPOL_FORMS)
