"""From r = 256 on the weight field stays transformed along z alone, and its
sums are taken in the y passes: the scalars of Eq. 4 and W~ as it is read back
against FP64, for clouds that touch some y-blocks, all of them, or plane 0, and
with a cluster size asked for, where the same passes run."""
import numpy as np
import pytest

from paper_2106_03452_gb300 import synth
from test_gpu_empty_tiles import _cloud

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2106_03452_gb300 import build
    build.build()


@pytest.mark.parametrize("path", [None, "4"])
def test_scalars_and_weights(oracle, monkeypatch, path):
    import torch
    from paper_2106_03452_gb300 import libdpsr as L
    from paper_2106_03452_gb300.dpsr import Plan
    if path:
        monkeypatch.setenv("DPSR_PLANE_PATH", path)
    r, sigma = 256, 2.0
    rng = synth.Rng(41)
    plan = Plan(r, sigma)
    for kind, n in (("full", 20000), ("corner", 500), ("line_z", 500), ("slab_x", 700)):
        if kind == "full":
            pts, nrm = rng.uniform(n, 3).astype(np.float32), rng.normal(n, 3).astype(np.float32)
        else:
            pts, nrm = _cloud(kind, r, n, rng)
        plan.forward(torch.from_numpy(pts).cuda(), torch.from_numpy(nrm).cuda())
        assert plan.sync() == 0, kind
        got = L.dpsr_debug_read_spectrum(plan.handle, 2, r)
        w = np.fft.fft(np.fft.rfft(oracle.splat(r, pts.astype(np.float64)).reshape(r, r, r), axis=2), axis=1)
        assert np.max(np.abs(got - w)) <= 5e-6 * np.max(np.abs(w)), kind
        _, chip, mu, s = oracle.forward(r, sigma, pts, nrm, full=True)
        sc = plan.scalars()
        top = np.max(np.abs(chip))  # the bound of chi: 1e-5 of its largest entry
        assert abs(sc[0] - mu) <= 1e-5 * top and abs(sc[1] - s) <= 2e-5 * top, (kind, sc, mu, s, top)
    assert L.dpsr_plan_clusters(plan.handle) == [0, 0, 0, 0]
    plan.close()
