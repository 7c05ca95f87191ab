"""The half-image kernels at N_p = 256 (GPU only) where they can go wrong: unit ranges that cut a (channel,
pol) or a half, one image, image counts on both sides of the rule that takes a call to the cluster kernels
(39 to 76 images and most counts above take the halves), antenna counts around the 512 threads' shares and
the shared-memory limit (1,471 the most; the cluster kernels beyond), arrays that leave most cells empty or
reach the grid's corners, complex weights, every voltage format, powers and continued integrations, the
adjoint, and lists of plans (batches).

Against the oracle in float64.  FP32 transforms of 256 points round at most 16 times at 2^-24 in each
direction: 1e-5 of the image's norm, and of the gradient's 1e-4 (it sums signed terms of an image-sized
spread)."""
import numpy as np
import pytest

from oracle import moff
from paper_1510_08318_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
TOL, TOL_GRAD = 1e-5, 1e-4


@pytest.fixture(scope="module")
def epic():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1510_08318_gb300 import build, epic as ep
    build.build()
    ep.load()
    return ep


def _workload(n_ant, n_time, n_chan, n_pol, vdtype, complex_w=False, n_grid=128):
    rng = np.random.default_rng([n_ant, n_time, n_chan])
    pos = rng.uniform(1.0, n_grid - 2.0, (n_ant, 2))
    pos[0] = 0.0                                     # the grid's corner cells
    pos[-1] = n_grid - 1.0
    kerns = [synth.kernel_point()] + [synth.kernel_square(rng.uniform(0.5, 2.0), 0.5) for _ in range(n_ant - 2)]
    kerns += [synth.kernel_point()] * (n_ant - len(kerns))
    ptr, dxdy, w = synth.pack_kernels(kerns)
    if complex_w:
        w = w * np.exp(1j * rng.uniform(0, 2 * np.pi, w.shape))
    wl = synth.Workload("half256", pos, ptr, dxdy, w, 1.0, np.zeros(2), n_grid, 256, np.full(n_chan, 1e8), n_pol,
                        n_time, vdtype)
    shape = (n_time, n_chan, n_pol, n_ant)
    return synth._finish(wl, rng.standard_normal(shape) + 1j * rng.standard_normal(shape), vdtype)


def _map(wl):
    return moff.map_antennas(wl.pos, wl.kern_ptr, wl.kern_dxdy, wl.kern_w, wl.dx, wl.origin, wl.n_grid)


@pytest.mark.parametrize("n_ant, n_time, n_chan, n_pol, vdtype, complex_w, n_grid", [
    (1, 40, 1, 1, "c64", False, 128),
    (2, 7, 3, 2, "f16", False, 101),
    (513, 21, 2, 1, "ci4", True, 128),
    (60, 103, 2, 1, "f16", False, 128),
    (331, 77, 1, 1, "f16", False, 128),
    (1471, 40, 1, 1, "f16", False, 128),
    (1472, 40, 1, 1, "f16", False, 128),
    (3, 1, 1, 1, "c64", False, 128),
])
def test_image_power_gradient(epic, n_ant, n_time, n_chan, n_pol, vdtype, complex_w, n_grid):
    wl = _workload(n_ant, n_time, n_chan, n_pol, vdtype, complex_w, n_grid)
    rng = np.random.default_rng(n_ant)
    g = synth.random_gains(rng, (n_chan, n_pol, n_ant))
    G = rng.standard_normal((n_chan, n_pol, 256, 256)).astype(np.float32)
    plan, M, gg = epic.Plan.from_workload(wl), _map(wl), g.astype(np.complex128)
    volt, gains = torch.from_numpy(wl.volt_raw).cuda(), torch.from_numpy(g).cuda()
    out = plan.image(volt, gains, want_autocorr=True)
    want = moff.moff_image(M, wl.volt, gg, wl.n_grid, 256)
    got = out["image"].cpu().numpy()
    for c in range(n_chan):
        for p in range(n_pol):
            assert np.linalg.norm(got[c, p] - want[c, p]) < TOL * np.linalg.norm(want[c, p]), (c, p)
    power = (np.abs(wl.volt * gg) ** 2).sum(0)
    assert np.abs(out["power"].cpu().numpy() - power).max() < TOL * power.max()
    again = plan.image(volt, gains, accum=out["accum"], power=out["power"], t_prev=n_time)
    assert np.linalg.norm(again["image"].cpu().numpy() - want) < TOL * np.linalg.norm(want)
    grad = plan.image_backward(volt, gains, torch.from_numpy(G).cuda()).cpu().numpy()
    want_g = moff.grad_gains(M, wl.volt, gg, wl.n_grid, 256, G.astype(np.float64))
    assert np.linalg.norm(grad - want_g) < TOL_GRAD * np.linalg.norm(want_g)


def test_lists_of_plans(epic):
    """A batch of three plans of different sizes (one past the half-image kernels' antennas in a second list):
    units cut at plan, channel and half boundaries."""
    for sizes in [(5, 90, 600), (40, 1500)]:
        wls = [_workload(a, 7, 1 + i, 1, "f16") for i, a in enumerate(sizes)]
        plans = [epic.Plan.from_workload(w) for w in wls]
        batch = epic.Batch(plans)
        acc, img = batch.alloc()
        batch.image([torch.from_numpy(w.volt_raw).cuda() for w in wls], acc, img)
        torch.cuda.synchronize()
        for w, im in zip(wls, img):
            want = moff.moff_image(_map(w), w.volt, None, w.n_grid, 256)
            assert np.linalg.norm(im.cpu().numpy() - want) < TOL * np.linalg.norm(want), sizes
