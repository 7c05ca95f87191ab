"""The tensor-core form at N_p = 128 (GPU only) where its two-image pipeline can go wrong: one image, odd
and even image counts, (channel, pol) changing inside a pair of images, more and fewer images than SMs,
antenna counts around the gridding threads' shares (176 antennas a round, 352 prefetched) and past the
count that fits two voltage buffers (about 1,900), arrays whose footprints leave most cells empty or
reach the grid's corner, complex weights, gains, powers and continued integrations.

Against the oracle in float64.  Operands carry about 22 bits (relative 2^-22 each) and FP32 sums of at
most 192 products round at 2^-24 each: 1e-5 of the image's norm bounds the field's error doubled by the
square."""
import numpy as np
import pytest

from oracle import moff
from paper_1510_08318_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
TOL = 1e-5


@pytest.fixture(scope="module")
def epic():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1510_08318_gb300 import build, epic as ep
    build.build()
    ep.load()
    return ep


def _workload(n_ant, n_time, n_chan, n_pol, vdtype, complex_w=False, seed=0):
    rng = np.random.default_rng([n_ant, n_time, seed])
    n_grid, n_pad = 64, 128
    pos = rng.uniform(1.0, n_grid - 2.0, (n_ant, 2))
    pos[0] = 0.0                                        # an antenna on the grid's corner cell
    kerns = [synth.kernel_point()] + [synth.kernel_square(rng.uniform(0.5, 2.0), 0.5) for _ in range(n_ant - 1)]
    ptr, dxdy, w = synth.pack_kernels(kerns)
    if complex_w:
        w = w * np.exp(1j * rng.uniform(0, 2 * np.pi, w.shape))
    wl = synth.Workload("dg128", pos, ptr, dxdy, w, 1.0, np.zeros(2), n_grid, n_pad, np.full(n_chan, 1e8), n_pol,
                        n_time, vdtype)
    shape = (n_time, n_chan, n_pol, n_ant)
    return synth._finish(wl, rng.standard_normal(shape) + 1j * rng.standard_normal(shape), vdtype)


@pytest.mark.parametrize("n_ant, n_time, n_chan, n_pol, vdtype, complex_w", [
    (1, 1, 1, 1, "c64", False),
    (3, 1, 5, 2, "f16", False),
    (176, 3, 2, 2, "ci4", False),
    (177, 2, 1, 1, "c64", True),
    (353, 5, 3, 1, "ci4", False),
    (40, 409, 3, 1, "f16", True),
    (2000, 2, 2, 1, "f16", False),
    (2448, 1, 3, 1, "ci4", False),
])
def test_image_and_power(epic, n_ant, n_time, n_chan, n_pol, vdtype, complex_w):
    wl = _workload(n_ant, n_time, n_chan, n_pol, vdtype, complex_w)
    g = synth.random_gains(np.random.default_rng(n_ant), (n_chan, n_pol, n_ant))
    plan = epic.Plan.from_workload(wl).set_transform("dftgemm")
    volt, gains = torch.from_numpy(wl.volt_raw).cuda(), torch.from_numpy(g).cuda()
    out = plan.image(volt, gains, want_autocorr=True)
    plan.sync()
    M = moff.map_antennas(wl.pos, wl.kern_ptr, wl.kern_dxdy, wl.kern_w, wl.dx, wl.origin, wl.n_grid)
    want = moff.moff_image(M, wl.volt, g.astype(np.complex128), wl.n_grid, wl.n_pad)
    got = out["image"].cpu().numpy()
    for c in range(n_chan):
        for p in range(n_pol):
            assert np.linalg.norm(got[c, p] - want[c, p]) < TOL * np.linalg.norm(want[c, p]), (c, p)
    power = (np.abs(wl.volt * g.astype(np.complex128)) ** 2).sum(0)
    assert np.abs(out["power"].cpu().numpy() - power).max() < 1e-5 * power.max()
    # a second block continues the integration
    again = plan.image(volt, gains, accum=out["accum"], power=out["power"], t_prev=n_time)
    plan.sync()
    assert np.linalg.norm(again["image"].cpu().numpy() - want) < TOL * np.linalg.norm(want)


def test_cross_products_over_a_pair_of_images(epic):
    """Three samples per virtual pol: every pair of images but one in three spans two of them."""
    wl = _workload(60, 3, 2, 2, "ci4")
    plan = epic.Plan.from_workload(wl).set_transform("dftgemm")
    out = plan.image_xpol(torch.from_numpy(wl.volt_raw).cuda())
    plan.sync()
    M = moff.map_antennas(wl.pos, wl.kern_ptr, wl.kern_dxdy, wl.kern_w, wl.dx, wl.origin, wl.n_grid)
    want = moff.moff_image(M, wl.volt, None, wl.n_grid, wl.n_pad)
    assert np.linalg.norm(out["image"].cpu().numpy() - want) < TOL * np.linalg.norm(want)
