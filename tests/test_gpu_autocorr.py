"""The auto-correlation term (GPU only) at the sizes where its kernel can go wrong: every cluster size (1, 2, 4, 8 CTAs
per (channel, pol), chosen by antennas, (channel, pol) and pixels), antennas that do not divide over the cluster,
footprints of one cell, continued integrations; and footprints up to the widest that a plan admits, where shared
memory is full (N_p = 512: 25 cells up to 2,110 antennas, 24 cells beyond).

Against the oracle in float64.  All its sums are FP32: P_a from T samples, U(d) from A antennas, and two transforms of
L lags each (two fused multiply-adds a lag), with single roundings of the tables.  Every partial sum is bounded by
sum_a P_a (sum |w_a|)^2, which is the term at the image's centre for positive weights, so a pixel is off by at most
(A + T + 4 L + 16) 2^-24 of that."""
import numpy as np
import pytest

from oracle import moff
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


def _workload(pos, kerns, n_pad, n_time, n_chan, n_pol, complex_w=False):
    rng = np.random.default_rng([len(pos), n_pad, n_chan])
    ptr, dxdy, w = synth.pack_kernels(kerns)
    if complex_w:
        w = w * np.exp(1j * rng.uniform(0, 2 * np.pi, w.shape))
    wl = synth.Workload("autocorr", pos, ptr, dxdy, w, 1.0, np.zeros(2), n_pad // 2, n_pad, np.full(n_chan, 1e8), n_pol,
                        n_time, "c64")
    shape = (n_time, n_chan, n_pol, len(pos))
    return synth._finish(wl, rng.standard_normal(shape) + 1j * rng.standard_normal(shape), "c64")


def _bound(wl, L, peak):
    return (wl.volt.shape[3] + wl.volt.shape[0] + 4 * L + 16) * 2.0 ** -24 * peak


@pytest.mark.parametrize("n_pad, n_ant, n_chan, n_pol, kind", [
    (64, 3, 1, 1, "squares"),
    (64, 7, 1, 1, "complex"),
    (64, 13, 3, 1, "squares"),
    (64, 37, 1, 2, "complex"),
    (64, 37, 50, 2, "squares"),
    (64, 37, 160, 1, "points"),
    (32, 37, 155, 2, "squares"),
    (128, 300, 1, 1, "squares"),
    (256, 18, 2, 1, "points"),
])
def test_cluster_sizes(epic, n_pad, n_ant, n_chan, n_pol, kind):
    rng = np.random.default_rng(n_ant)
    pos = rng.uniform(2.0, n_pad // 2 - 3.0, (n_ant, 2))
    kerns = [synth.kernel_point() if kind == "points" else synth.kernel_square(rng.uniform(0.5, 2.5), 1 / 3)
             for _ in range(n_ant)]
    wl = _workload(pos, kerns, n_pad, 6, n_chan, n_pol, kind == "complex")
    g = synth.random_gains(rng, (n_chan, n_pol, n_ant))
    plan, gains, volt = epic.Plan.from_workload(wl), torch.from_numpy(g).cuda(), torch.from_numpy(wl.volt_raw).cuda()
    M = moff.map_antennas(wl.pos, wl.kern_ptr, wl.kern_dxdy, wl.kern_w, wl.dx, wl.origin, wl.n_grid)
    want = moff.autocorr_term(M, wl.volt, g.astype(np.complex128), wl.n_grid, n_pad)
    P = (np.abs(wl.volt * g) ** 2).mean(0)
    peak = (P * np.asarray(np.abs(M).sum(0)).reshape(-1) ** 2).sum(-1)[..., None, None]
    full = plan.image(volt, gains, want_autocorr=True)
    part = plan.image(volt[:2].contiguous(), gains, want_image=False, want_autocorr=True)
    rest = plan.image(volt[2:].contiguous(), gains, accum=part["accum"], power=part["power"], t_prev=2,
                      want_autocorr=True)
    only = plan.image(volt, gains, want_image=False, want_autocorr=True)
    for out in (full, rest, only):
        err = np.abs(out["autocorr"].cpu().numpy() - want)
        assert (err <= _bound(wl, plan.info["lag_side"], peak)).all(), (err / peak).max()
    # the image of the same launch is accum / T, one rounding
    for out in (full, rest):
        assert torch.equal(out["image"], (out["accum"] * (1.0 / 6)).float())


@pytest.mark.parametrize("cells, n_ant", [(25, 1), (25, 2110), (24, 993)])
def test_widest_footprints(epic, cells, n_ant):
    """Shared memory full: antennas of one footprint on whole cells, so that the term is sum_a P_a |K(k)|^2."""
    rng = np.random.default_rng(n_ant)
    off = np.arange(cells) - cells // 2
    kern = (np.array([(x, y) for y in off for x in off], dtype=np.float64), rng.uniform(0.5, 1.5, cells ** 2) / cells ** 2)
    pos = rng.integers(13, 243, (n_ant, 2)).astype(np.float64)
    wl = _workload(pos, [kern] * n_ant, 512, 2, 1, 1)
    plan, volt = epic.Plan.from_workload(wl), torch.from_numpy(wl.volt_raw).cuda()
    assert plan.info["lag_side"] == 2 * cells - 1
    one = moff.map_antennas(pos[:1], *synth.pack_kernels([kern]), 1.0, np.zeros(2), 256)
    P = (np.abs(wl.volt) ** 2).mean(0).sum()
    want = P * np.abs(moff.footprint_transforms(one, 256, 512)[0]) ** 2
    bound = _bound(wl, 2 * cells - 1, P * np.abs(kern[1]).sum() ** 2)
    out = plan.image(volt, want_autocorr=True)
    assert np.abs(out["autocorr"].cpu().numpy()[0, 0] - want).max() <= bound
    assert torch.equal(out["image"], (out["accum"] * 0.5).float())
    accum, power = torch.empty_like(out["accum"]), torch.empty_like(out["power"])
    image, term = torch.empty_like(out["image"]), torch.empty_like(out["autocorr"])
    epic.epic_image_noalloc(plan._h, volt.data_ptr(), 2, None, accum.data_ptr(), power.data_ptr(), 0, image.data_ptr(),
                            term.data_ptr(), 16, torch.cuda.current_stream().cuda_stream)
    torch.cuda.synchronize()
    assert np.abs(term.cpu().numpy()[0, 0] - want).max() <= bound
    assert torch.equal(image, (accum * 0.5).float())


def test_footprints_wider_than_the_tables(epic):
    """26 cells at N_p = 512 (and 25 with more antennas than fit) have no tables: refused before anything is launched."""
    rng = np.random.default_rng(5)
    for cells, n_ant in [(26, 1), (25, 2111)]:
        off = np.arange(cells) - cells // 2
        kern = (np.array([(x, y) for y in off for x in off], dtype=np.float64), np.full(cells ** 2, 1.0 / cells ** 2))
        wl = _workload(rng.integers(13, 243, (n_ant, 2)).astype(np.float64), [kern] * n_ant, 512, 1, 1, 1)
        plan = epic.Plan.from_workload(wl)
        assert plan.info["lag_side"] == 0
        with pytest.raises(epic.EpicError) as e:
            plan.image(torch.from_numpy(wl.volt_raw).cuda(), want_autocorr=True)
        assert e.value.status == epic.EPIC_EUNSUPPORTED
