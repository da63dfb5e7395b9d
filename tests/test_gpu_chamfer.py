"""The Chamfer distance by the box tree against FP64 brute force, at the sizes
where its packets, leaves, box levels and cell grids begin and end, and with
equal points, points far from the other set and points that are not finite."""
import numpy as np
import pytest

from paper_2106_03452_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2106_03452_gb300 import build
    build.build()


def _run(a, b):
    import torch
    from paper_2106_03452_gb300.optimize import chamfer
    A = torch.from_numpy(a).cuda().requires_grad_(True)
    loss = chamfer(A, torch.from_numpy(b).cuda())
    (g,) = torch.autograd.grad(loss, A)
    return float(loss.detach()), g.cpu().numpy()


def _reference(a, b):
    """Brute force in FP64 on neighbours picked as in FP32 (ties to the lowest index)."""
    def nearest(q, t):
        idx = np.empty(len(q), np.int64)
        for k in range(0, len(q), 256):
            d = (q[k:k + 256, None, :] - t[None]).astype(np.float64)
            v = np.float32(d[..., 2] ** 2)  # fma(dx, dx, fma(dy, dy, dz * dz)) in FP32
            for c in (1, 0):
                v = np.float32(d[..., c] ** 2 + v)
            idx[k:k + 256] = v.argmin(1)
        return idx
    i, j = nearest(a, b), nearest(b, a)
    a64, b64 = a.astype(np.float64), b.astype(np.float64)
    loss = ((a64 - b64[i]) ** 2).sum(1).mean() + ((b64 - a64[j]) ** 2).sum(1).mean()
    g = 2.0 * (a64 - b64[i]) / len(a)
    np.add.at(g, j, 2.0 * (a64[j] - b64) / len(b))
    return loss, g


SIZES = [(1, 1), (1, 1000), (16, 17), (31, 33), (1024, 1025), (32768, 40), (70, 32769), (5001, 3003)]


@pytest.mark.parametrize("na,nb", SIZES)
@pytest.mark.parametrize("kind", ["surface", "volume", "grid", "apart"])
def test_tree_matches_bruteforce(na, nb, kind):
    rng = synth.Rng(na * 7 + nb + len(kind))
    if kind == "surface":
        a, b = (synth.sphere_cloud(rng, n, jitter=0.01)[0] for n in (na, nb))
    elif kind == "volume":
        a, b = rng.uniform(na, 3) * 2 - 1, rng.uniform(nb, 3) * 2 - 1
    elif kind == "grid":  # equal points and equal distances everywhere
        a, b = (np.floor(rng.uniform(n, 3) * 9) for n in (na, nb))
    else:  # the sets far from each other, one of them flat, and a stray point
        a, b = rng.uniform(na, 3) * [1, 1, 0], rng.uniform(nb, 3) + [40, 0, 0]
        a[0] = [-1e6, 3, 5]
    a, b = a.astype(np.float32), b.astype(np.float32)
    loss, g = _run(a, b)
    rloss, rg = _reference(a, b)
    # FP32 squared distances (relative 2^-22), and sums of at most nb + 1 terms per gradient
    assert abs(loss - rloss) <= 1e-6 * rloss
    assert np.max(np.abs(g - rg)) <= 1e-5 * np.max(np.abs(rg))


def test_points_that_are_not_finite():
    rng = synth.Rng(5)
    a, b = rng.uniform(700, 3).astype(np.float32), rng.uniform(900, 3).astype(np.float32)
    a[3, 1], a[200, 0], b[17, 2], b[500] = np.nan, np.inf, np.nan, -np.inf
    loss, g = _run(a, b)
    fa, fb = np.isfinite(a).all(1), np.isfinite(b).all(1)
    _, rg = _reference(a[fa], b[fb])
    assert not np.isfinite(loss) and np.isnan(g[~fa]).all()
    # the finite points' neighbours are the finite ones; the weights count every point
    i = np.nonzero(fa)[0]
    d = a[fa][:, None, :].astype(np.float64) - b[fb][None]
    ab, ba = (d ** 2).sum(-1).argmin(1), (d ** 2).sum(-1).argmin(0)
    want = 2.0 * (a[fa] - b[fb][ab].astype(np.float64)) / len(a)
    np.add.at(want, ba, 2.0 * (a[fa][ba].astype(np.float64) - b[fb]) / len(b))
    assert np.max(np.abs(g[i] - want)) <= 1e-5 * np.max(np.abs(want))


def test_workspace_is_checked():
    from paper_2106_03452_gb300 import libdpsr as L
    assert L.dpsr_chamfer_ws_bytes(0, 5) == 0 and L.dpsr_chamfer_ws_bytes(5, 2 ** 31) == 0
    n = L.dpsr_chamfer_ws_bytes(10, 10)
    lib = L.load()
    for ws, nb in ((256, n - 1), (264, n), (0, n)):  # too small, misaligned, NULL: refused before any launch
        assert lib.dpsr_chamfer_tree(256, 10, 256, 10, ws or None, nb, 256, 256, None, None) == L.DPSR_EINVAL


def _hard(kind, n=20000):
    """Sets that a grid of equal cells over the bounding box cannot split."""
    rng = synth.Rng(len(kind))
    a, b = (synth.sphere_cloud(rng, n, jitter=0.01)[0] for _ in range(2))
    if kind == "outlier":
        a[7] = 1e6
    elif kind == "outliers in both":
        a[7], b[n - 9] = 1e6, -1e6
    elif kind == "cluster in a large box":
        box = rng.uniform(n // 4, 3) * 1000
        a[::4], b[::4] = box, box + 0.5
    elif kind == "one place":
        b[:] = 0.25
    elif kind == "two places":
        a[:], b[:] = 0.75, 0.25
    elif kind == "half in one place":
        a[::2], b[1::2] = 0.5, 0.5
    elif kind == "far apart":
        b += 1e6
    elif kind == "scales":
        s = 10.0 ** np.floor(rng.uniform(n, 1) * 8 - 4)
        a, b = rng.normal(n, 3) * s, rng.normal(n, 3) * s
    elif kind == "axes":
        k, (u, v) = np.arange(n) % 3, rng.uniform(2, n)
        a, b = np.zeros((n, 3)), np.zeros((n, 3))
        a[np.arange(n), k], b[np.arange(n), k] = u, v
    return np.ascontiguousarray(a, np.float32), np.ascontiguousarray(b, np.float32)


@pytest.mark.parametrize("kind", ["outlier", "outliers in both", "cluster in a large box", "one place", "two places",
                                  "half in one place", "far apart", "scales", "axes"])
def test_hard_sets_equal_bruteforce_and_cost_no_more(kind):
    import torch
    from paper_2106_03452_gb300 import libdpsr as L
    a, b = (torch.from_numpy(x).cuda() for x in _hard(kind))
    n, st = a.shape[0], torch.cuda.current_stream().cuda_stream
    ws = torch.empty(L.dpsr_chamfer_ws_bytes(n, n), dtype=torch.uint8, device="cuda")
    idx, d2 = torch.empty(2 * n, dtype=torch.int32, device="cuda"), torch.empty(2 * n, device="cuda")
    out = []
    for tree in (True, False):
        g, loss = torch.empty_like(a), torch.empty(1, dtype=torch.float64, device="cuda")

        def call():
            if tree:
                L.dpsr_chamfer_tree(a.data_ptr(), n, b.data_ptr(), n, ws.data_ptr(), ws.numel(), g.data_ptr(),
                                    loss.data_ptr(), 0, st)
            else:
                L.dpsr_chamfer(a.data_ptr(), n, b.data_ptr(), n, idx.data_ptr(), d2.data_ptr(), g.data_ptr(),
                               loss.data_ptr(), st)
        call()
        ms = []
        for _ in range(5):
            e = [torch.cuda.Event(enable_timing=True) for _ in range(2)]
            e[0].record()
            call()
            e[1].record()
            e[1].synchronize()
            ms.append(e[0].elapsed_time(e[1]))
        out.append((loss.item(), g.cpu().double(), sorted(ms)[2]))
    (l1, g1, t1), (l0, g0, t0) = out
    # the same neighbours: sums of the same terms in another order
    assert abs(l1 - l0) <= 1e-6 * abs(l0)
    assert float((g1 - g0).abs().max()) <= 1e-5 * float(g0.abs().max())
    assert t1 <= t0, (t1, t0)


def test_bruteforce_with_points_that_are_not_finite():
    """dpsr_chamfer's points without a neighbour are nobody's, as the tree's
    (their index is -1; buffers with guards around them stay as they are)."""
    import torch
    from paper_2106_03452_gb300 import libdpsr as L
    rng = synth.Rng(6)
    a, b = (torch.from_numpy(rng.uniform(n, 3).astype(np.float32)).cuda() for n in (500, 600))
    a[0, 1], a[7, 0], a[20] = np.nan, np.inf, 3e38
    b[0], b[5, 2] = np.nan, -np.inf
    st = torch.cuda.current_stream().cuda_stream
    g = torch.full((500 + 20, 3), 7.0, device="cuda")
    loss = torch.empty(1, dtype=torch.float64, device="cuda")
    idx, d2 = torch.empty(1100, dtype=torch.int32, device="cuda"), torch.empty(1100, device="cuda")
    L.dpsr_chamfer(a.data_ptr(), 500, b.data_ptr(), 600, idx.data_ptr(), d2.data_ptr(), g[10:].data_ptr(),
                   loss.data_ptr(), st)
    assert bool((g[:10] == 7).all()) and bool((g[510:] == 7).all())
    ws = torch.empty(L.dpsr_chamfer_ws_bytes(500, 600), dtype=torch.uint8, device="cuda")
    t = torch.empty_like(a)
    L.dpsr_chamfer_tree(a.data_ptr(), 500, b.data_ptr(), 600, ws.data_ptr(), ws.numel(), t.data_ptr(), loss.data_ptr(),
                        0, st)
    g = g[10:510]
    bad = torch.isnan(g)
    assert torch.equal(bad, torch.isnan(t)) and bool(bad[[0, 7, 20]].all()) and int(bad.any(1).sum()) == 3
    assert float((g - t)[~bad].abs().max()) <= 1e-5 * float(t[~bad].abs().max())
    assert not np.isfinite(loss.item())
