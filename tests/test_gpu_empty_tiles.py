"""Clouds that leave most of the domain empty, where the passes skip the tiles
and planes without points: corners and slabs across the periodic wrap, a line
of points along each axis, a lone cell. Each follows a cloud that filled the
whole domain on the same plan, so that what is skipped holds that cloud's
spectra and a tile that is wrongly left out, or read, shows. Against the FP64
oracle, both plane paths, with the spectra of the splat read back."""
import numpy as np
import pytest

from paper_2106_03452_gb300 import synth

pytestmark = pytest.mark.gpu

KINDS = ["corner", "slab_x", "slab_y", "line_x", "line_y", "line_z", "cell", "far_apart"]


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2106_03452_gb300 import build
    build.build()


def _cloud(kind, r, n, rng):
    """Points, and normals that point away from the cloud's centre, axis or
    plane: chi' then has one sign on the points, and Eq. 4's scale (chi'(0)
    minus its mean there) does not cancel."""
    u = rng.uniform(n, 3)
    c = np.zeros((n, 3))                    # where the normals point away from
    if kind == "corner":                    # all eight corner cells of the wrap
        p = (u - 0.5) * (3.0 / r)
    elif kind in ("slab_x", "slab_y"):      # across 0 of one axis
        a = "xy".index(kind[-1])
        p = u.copy()
        p[:, a] = (u[:, 2] - 0.5) * (2.5 / r)
        p[:, 2] = rng.uniform(n)
        c = np.where(np.arange(3) == a, 0.0, p)
    elif kind.startswith("line"):           # one row of cells along an axis, on a block's last row
        a = "xyz".index(kind[-1])
        p = (16 - 0.5) / r + (u - 0.5) * (0.9 / r)
        p[:, a] = u[:, a]
        c = np.where(np.arange(3) == a, p, (16 - 0.5) / r)
    elif kind == "cell":                    # one cell, its second row in the next block
        p = (np.array([r // 2, 15, 3]) + u) / r
        c = np.broadcast_to((np.array([r // 2, 15, 3]) + 0.5) / r, p.shape)
    else:                                   # two small balls
        c = np.where(rng.uniform(n, 1) < 0.5, 0.05, 0.8) * np.ones((1, 3))
        p = c + (u - 0.5) * 0.1
    d = p - c
    return p.astype(np.float32), (d / np.linalg.norm(d, axis=1, keepdims=True)).astype(np.float32)


@pytest.mark.parametrize("path", ["0", "1"])
@pytest.mark.parametrize("r", [32, 64, 128])
def test_sparse_clouds_match_the_oracle(oracle, monkeypatch, r, path):
    import torch
    from gpu_util import gpu_fwd_bwd, relmax
    from paper_2106_03452_gb300 import libdpsr as L
    from paper_2106_03452_gb300.dpsr import Plan
    monkeypatch.setenv("DPSR_PLANE_PATH", path)
    sigma, n = 2.0, 400
    rng = synth.Rng(5200 + r)
    plan = Plan(r, sigma)
    full = rng.uniform(40 * r, 3).astype(np.float32), rng.normal(40 * r, 3).astype(np.float32)
    dchi = synth.upstream_grad(rng, r)
    for kind in KINDS:
        assert gpu_fwd_bwd(r, sigma, *full, dchi, plan)["bstatus"] == 0  # leaves every tile filled
        pts, nrm = _cloud(kind, r, n, rng)
        out = gpu_fwd_bwd(r, sigma, pts, nrm, None, plan)
        assert out["status"] == 0, kind
        chi, chip, mu, s = oracle.forward(r, sigma, pts, nrm, full=True)
        # FP32 rounding of the scale (see the parity tests), amplified by max|chi'| / |s|
        slack = 2.0 ** -24 * float(np.max(np.abs(chip))) / abs(s)
        assert relmax(out["chi"], chi) <= 1e-5 + slack, kind
        w = np.fft.fft(np.fft.rfft(oracle.splat(r, pts.astype(np.float64)).reshape(r, r, r), axis=2), axis=1)
        got = L.dpsr_debug_read_spectrum(plan.handle, 2, r)
        assert np.max(np.abs(got - w)) <= 5e-6 * np.max(np.abs(w)), kind
        rdp, rdn = oracle.backward(r, sigma, pts, nrm, dchi)
        for _ in range(2):  # any number of backward passes follows a forward
            dp, dn = plan.backward(torch.from_numpy(dchi).cuda())
            assert plan.sync() == 0
            assert relmax(dp.cpu().numpy(), rdp) <= 1e-4 + slack, kind
            assert relmax(dn.cpu().numpy(), rdn) <= 1e-4 + slack, kind
    plan.close()


@pytest.mark.parametrize("r", [256, 512])
def test_sparse_clouds_on_the_largest_grids(r):
    """The tuned paths against the layer in plain FP64 GPU operations."""
    import torch
    import bench
    from gpu_util import relmax
    from paper_2106_03452_gb300.dpsr import Plan
    rng = synth.Rng(90 + r)
    plan = Plan(r, 3.0)
    gen = torch.Generator("cuda").manual_seed(r)
    full = [torch.rand((60000, 3), device="cuda", generator=gen) for _ in range(2)]
    d = torch.randn((r, r, r), device="cuda", generator=gen)
    for kind in ("corner", "slab_y", "line_y", "far_apart"):
        plan.forward(*full)
        plan.backward(d)
        pts, nrm = (torch.from_numpy(x).cuda() for x in _cloud(kind, r, 3000, rng))
        chi = plan.forward(pts, nrm)
        dp, dn = plan.backward(d)
        assert plan.sync() == 0, kind
        p64, n64 = pts.double().requires_grad_(True), nrm.double().requires_grad_(True)
        ref = bench.torch_ops_dpsr(p64, n64, r, 3.0)
        rdp, rdn = torch.autograd.grad(ref, (p64, n64), d.double())
        _, s, a = plan.scalars()
        slack = 2.0 ** -24 * float(ref.detach().abs().max()) / (a * abs(s))
        cpu = lambda t: t.detach().cpu().numpy()  # noqa: E731
        assert relmax(cpu(chi), cpu(ref)) <= 1e-5 + slack, kind
        assert relmax(cpu(dp), cpu(rdp)) <= 1e-4 + slack and relmax(cpu(dn), cpu(rdn)) <= 1e-4 + slack, kind
        del ref, rdp, rdn
    plan.close()


@pytest.mark.parametrize("n", [1023, 1025, 303105])
def test_point_counts_at_the_edges_of_the_binning_blocks(n):
    """r = 256: one point short of and past a block of 1 024, and past the
    last point that the grid's blocks take one each (296 of them)."""
    import torch
    import bench
    from gpu_util import relmax
    from paper_2106_03452_gb300.dpsr import Plan
    pts, nrm = (torch.from_numpy(x).cuda() for x in synth.sphere_cloud(synth.Rng(n), n))
    plan = Plan(256, 2.0)
    chi = plan.forward(pts, nrm)
    assert plan.sync() == 0
    with torch.no_grad():
        ref = bench.torch_ops_dpsr(pts.double(), nrm.double(), 256, 2.0)
    assert relmax(chi.cpu().numpy(), ref.cpu().numpy()) <= 1e-5
    plan.close()
