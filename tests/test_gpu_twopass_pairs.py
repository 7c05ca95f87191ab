"""The two-pass form's kernels at N_p = 512 (GPU only) where they can go wrong: one item, odd item counts, sample
pairs that cut a (channel, pol) or a sub-array, item counts on both sides of the column pass's groups (19 on 152
SMs) and of a chunk of scratch (4 per SM), antenna counts on both sides of the row pass's forms (665: two CTAs an
SM; 1,587: one; beyond: one sample at a time), arrays that leave most cells empty or reach the grid's corners,
complex weights, every voltage format, powers and continued integrations.

Against the oracle in float64.  FP32 transforms of 512 points round at most 18 times at 2^-24 in each direction:
1e-5 of the image's norm."""
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


def _workload(n_ant, n_time, n_chan, n_pol, vdtype, complex_w=False, n_grid=256):
    rng = np.random.default_rng([n_ant, n_time, n_chan])
    pos = rng.uniform(1.0, n_grid - 2.0, (n_ant, 2))
    pos[0] = 0.0                                     # the grid's corner cells
    pos[-1] = n_grid - 1.0
    kerns = [synth.kernel_point()] + [synth.kernel_square(rng.uniform(0.5, 2.0), 0.5) for _ in range(n_ant - 2)]
    kerns += [synth.kernel_point()] * (n_ant - len(kerns))
    ptr, dxdy, w = synth.pack_kernels(kerns)
    if complex_w:
        w = w * np.exp(1j * rng.uniform(0, 2 * np.pi, w.shape))
    wl = synth.Workload("twopass", pos, ptr, dxdy, w, 1.0, np.zeros(2), n_grid, 512, np.full(n_chan, 1e8), n_pol,
                        n_time, vdtype)
    shape = (n_time, n_chan, n_pol, n_ant)
    return synth._finish(wl, rng.standard_normal(shape) + 1j * rng.standard_normal(shape), vdtype)


def _map(wl):
    return moff.map_antennas(wl.pos, wl.kern_ptr, wl.kern_dxdy, wl.kern_w, wl.dx, wl.origin, wl.n_grid)


@pytest.mark.parametrize("n_ant, n_time, n_chan, n_pol, vdtype, complex_w, n_grid", [
    (1, 1, 1, 1, "c64", False, 256),
    (2, 3, 3, 2, "f16", False, 199),
    (300, 19, 1, 1, "ci4", True, 256),
    (60, 305, 2, 1, "f16", False, 130),
    (665, 7, 1, 2, "f16", False, 256),
    (666, 7, 3, 1, "ci4", False, 256),
    (1587, 5, 2, 1, "c64", True, 256),
    (1588, 5, 2, 1, "c64", False, 256),
])
def test_image_power(epic, n_ant, n_time, n_chan, n_pol, vdtype, complex_w, n_grid):
    wl = _workload(n_ant, n_time, n_chan, n_pol, vdtype, complex_w, n_grid)
    g = synth.random_gains(np.random.default_rng(n_ant), (n_chan, n_pol, n_ant))
    plan, gg = epic.Plan.from_workload(wl).set_transform("fft_twopass"), g.astype(np.complex128)
    volt, gains = torch.from_numpy(wl.volt_raw).cuda(), torch.from_numpy(g).cuda()
    out = plan.image(volt, gains, want_autocorr=True)
    got, want = out["image"].cpu().numpy(), moff.moff_image(_map(wl), wl.volt, gg, wl.n_grid, 512)
    for c in range(n_chan):
        for p in range(n_pol):
            assert np.linalg.norm(got[c, p] - want[c, p]) < TOL * np.linalg.norm(want[c, p]), (c, p)
    power = (np.abs(wl.volt * gg) ** 2).sum(0)
    assert np.abs(out["power"].cpu().numpy() - power).max() < TOL * power.max()
    again = plan.image(volt, gains, accum=out["accum"], power=out["power"], t_prev=n_time)
    assert np.linalg.norm(again["image"].cpu().numpy() - want) < TOL * np.linalg.norm(want)


@pytest.mark.parametrize("sizes", [(5, 300, 90), (40, 1000), (1600, 40)])
def test_lists_of_plans(epic, sizes):
    """A batch of plans of odd sample counts, complex and real weights mixed, in the form that the autotuner keeps,
    equals calls of each plan in the cluster form."""
    wls = [_workload(a, 7, 1 + 2 * i, 1, "f16", complex_w=i == 1) for i, a in enumerate(sizes)]
    plans, volts = [epic.Plan.from_workload(w) for w in wls], [torch.from_numpy(w.volt_raw).cuda() for w in wls]
    refs = [p.image(v)["image"].cpu().numpy() for p, v in zip(plans, volts)]
    batch = epic.Batch(plans)
    acc, img = batch.alloc()
    batch.autotune(volts, acc)
    for a in acc:
        a.zero_()
    batch.image(volts, acc, img)
    torch.cuda.synchronize()
    for w, im, ref in zip(wls, img, refs):
        assert np.linalg.norm(im.cpu().numpy() - ref) < TOL * np.linalg.norm(ref), sizes
