"""The correlator's kernel variants (GPU only) on both sides of the line between short and long integrations (FP16:
768 samples, 4+4 bits read one by one: 224), with antennas that leave rows and columns of a block empty.

Voltages are whole numbers of -7..7 (FP16 too), so every product is a whole number and every sum below 2^24 exact; the
result is that sum times the FP32 number next to 1/T: two roundings, 2^-23 of each component."""
import numpy as np
import pytest

from paper_1510_08318_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def epic():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1510_08318_gb300 import build, epic as ep
    build.build()
    ep.load()
    return ep


@pytest.mark.parametrize("vdtype, n_ant, n_time, n_chan, n_pol", [
    ("f16", 33, 5, 3, 1), ("f16", 130, 768, 2, 2), ("f16", 130, 769, 2, 2), ("f16", 256, 800, 60, 1),
    ("f16", 100, 64, 200, 1), ("ci4", 127, 1, 2, 1), ("ci4", 130, 224, 40, 2), ("ci4", 130, 225, 40, 2),
    ("ci4", 129, 40, 5, 1), ("ci4", 300, 33, 9, 2), ("ci4", 4, 300, 3, 2), ("ci4", 132, 65, 60, 2),
])
def test_exact_sums(epic, vdtype, n_ant, n_time, n_chan, n_pol):
    rng = np.random.default_rng([n_ant, n_time])
    re, im = rng.integers(-7, 8, (2, n_time, n_chan, n_pol, n_ant))
    if vdtype == "ci4":
        raw = torch.from_numpy(((re & 15) << 4 | (im & 15)).astype(np.uint8))
    else:
        raw = torch.from_numpy(np.stack([re, im], -1).astype(np.float16))
    ptr, dxdy, w = synth.pack_kernels([synth.kernel_point()] * n_ant)
    plan = epic.Plan(rng.uniform(1, 30, (n_ant, 2)), ptr, dxdy, w, 1.0, np.zeros(2), 32, 64, n_chan, n_pol, vdtype, 0)
    got = plan.correlate(raw.cuda()).cpu().numpy()
    v = (re + 1j * im).transpose(1, 2, 3, 0)
    want = v @ v.conj().swapaxes(-1, -2) / n_time
    for g, x in ((got.real, want.real), (got.imag, want.imag)):
        assert (np.abs(g - x) <= 1.001 * 2.0 ** -23 * np.abs(x)).all()
