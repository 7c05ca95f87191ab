"""FX imaging (GPU only) for few antennas, whose lag planes are gathered in wide groups: one plane, plane counts around
the group widths, odd ones among them, visibilities that are not Hermitian.

Against I(k) = Re sum_ab V_ab K_a(k) conj(K_b(k)) in float64, K_a the transform of antenna a's footprint.  In FP32 every
pixel sums A^2 pairs' entries and a transform of 128 lags a side: a pixel is off by at most (entries of a lag cell + 40)
2^-24 of sum_ab |V_ab| (sum |w_a|)(sum |w_b|), with at most A^2 entries in a cell."""
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


@pytest.mark.parametrize("n_ant", [1, 9])
@pytest.mark.parametrize("n_chan, n_pol", [(1, 1), (1, 2), (3, 1), (5, 1), (4, 2), (17, 1), (33, 1), (35, 2)])
def test_few_antennas(epic, n_ant, n_chan, n_pol):
    rng = np.random.default_rng([n_ant, n_chan])
    pos = rng.uniform(2.0, 60.0, (n_ant, 2))
    ptr, dxdy, w = synth.pack_kernels([synth.kernel_square(rng.uniform(0.5, 2.5), 1 / 3) for _ in range(n_ant)])
    plan = epic.Plan(pos, ptr, dxdy, w, 1.0, np.zeros(2), 64, 128, n_chan, n_pol, "ci4", 0)
    vis = rng.standard_normal((n_chan, n_pol, n_ant, n_ant, 2)).astype(np.float32)
    got = plan.fx_image(torch.view_as_complex(torch.from_numpy(vis)).contiguous().cuda()).cpu().numpy()
    M = moff.map_antennas(pos, ptr, dxdy, w, 1.0, np.zeros(2), 64)
    K = moff.footprint_transforms(M, 64, 128)
    V = vis[..., 0].astype(np.float64) + 1j * vis[..., 1]
    want = np.einsum("cpab,aij,bij->cpij", V, K, K.conj(), optimize=True).real
    norm = np.asarray(np.abs(M).sum(0)).reshape(-1)
    bound = (n_ant ** 2 + 40) * 2.0 ** -24 * np.einsum("cpab,a,b->cp", np.abs(V), norm, norm)
    assert (np.abs(got - want) <= bound[..., None, None]).all()
