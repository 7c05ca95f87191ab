"""Images of the half-image kernels at N_p = 256 (GPU only) at sample counts that the rule for their choice gives to
them (csrc/half_rule.h: many images, or fewer over several (channel, pol)): units that cut a half or a (channel,
pol), one sample each, antenna counts around the 512 threads' shares and the shared-memory limit (1,471), arrays that
leave most cells empty or reach the grid's corners, complex weights, every voltage format, powers, the
auto-correlation term and continued integrations.

Against the oracle in float64.  FP32 transforms of 256 points round at most 16 times at 2^-24 in each direction:
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


@pytest.mark.parametrize("n_ant, n_time, n_chan, n_pol, vdtype, complex_w, n_grid", [
    (1, 1, 76, 1, "c64", False, 128),
    (2, 2, 19, 2, "f16", False, 101),
    (513, 3, 25, 1, "ci4", True, 128),
    (60, 103, 5, 2, "f16", False, 128),
    (331, 608, 1, 1, "f16", False, 128),
    (1471, 15, 5, 1, "f16", False, 128),
    (1025, 152, 4, 1, "c64", True, 90),
])
def test_image_power(epic, n_ant, n_time, n_chan, n_pol, vdtype, complex_w, n_grid):
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
    wl = synth._finish(wl, rng.standard_normal(shape) + 1j * rng.standard_normal(shape), vdtype)
    g = synth.random_gains(rng, (n_chan, n_pol, n_ant))
    gg = g.astype(np.complex128)
    plan = epic.Plan.from_workload(wl)
    M = moff.map_antennas(wl.pos, wl.kern_ptr, wl.kern_dxdy, wl.kern_w, wl.dx, wl.origin, wl.n_grid)
    volt, gains = torch.from_numpy(wl.volt_raw).cuda(), torch.from_numpy(g).cuda()
    out = plan.image(volt, gains, want_autocorr=True)
    want = moff.moff_image(M, wl.volt, gg, wl.n_grid, 256)
    got = out["image"].cpu().numpy()
    for c in range(n_chan):
        for p in range(n_pol):
            assert np.linalg.norm(got[c, p] - want[c, p]) < TOL * np.linalg.norm(want[c, p]), (c, p)
    power = (np.abs(wl.volt * gg) ** 2).sum(0)
    assert np.abs(out["power"].cpu().numpy() - power).max() < TOL * power.max()
    if n_ant <= 100:
        ac = moff.autocorr_term(M, wl.volt, gg, wl.n_grid, 256)
        assert np.linalg.norm(out["autocorr"].cpu().numpy() - ac) < TOL * np.linalg.norm(ac)
    again = plan.image(volt, gains, accum=out["accum"], power=out["power"], t_prev=n_time)
    assert np.linalg.norm(again["image"].cpu().numpy() - want) < TOL * np.linalg.norm(want)
