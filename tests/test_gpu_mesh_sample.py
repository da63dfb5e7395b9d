"""Sampling on a triangle soup at the edges of its scan blocks (1 024
triangles), of its searches and of its vector loads, against FP64 on the same
draws."""
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


@pytest.mark.parametrize("offset", [0, 1])  # of the soup in floats: off a 16-byte boundary too
@pytest.mark.parametrize("T", [1, 2, 1023, 1024, 1025, 4099, 2048 * 1024 + 5])
def test_sample_matches_fp64(T, offset):
    import torch
    from paper_2106_03452_gb300.mesh import sample
    rng = synth.Rng(T + offset)
    M, seed = 3001, 77 + T
    tris = (rng.uniform(min(T, 5000), 3, 3) - 0.3).astype(np.float32)
    tris = np.tile(tris, (-(-T // len(tris)), 1, 1))[:T]
    tris[T // 2] = tris[T // 2, 0]  # a triangle without area
    if T == 1:
        tris[0] = [[0, 0, 0], [1, 0, 0], [0, 1, 0]]
    nrm = rng.normal(T, 3).astype(np.float32)
    buf = torch.empty(9 * T + 4, device="cuda")
    t = buf[offset:offset + 9 * T].view(T, 3, 3)
    t.copy_(torch.from_numpy(tris))
    P, N = (x.cpu().numpy().astype(np.float64) for x in sample(t, torch.from_numpy(nrm).cuda(), M, seed))
    t64 = tris.astype(np.float64)
    area = 0.5 * np.linalg.norm(np.cross(t64[:, 1] - t64[:, 0], t64[:, 2] - t64[:, 0]), axis=1)
    cum = np.cumsum(area)
    def u01(i):
        z = np.uint64(seed) + np.uint64(0x9E3779B97F4A7C15) * (i.astype(np.uint64) + np.uint64(1))
        z = (z ^ (z >> np.uint64(30))) * np.uint64(0xBF58476D1CE4E5B9)
        z = (z ^ (z >> np.uint64(27))) * np.uint64(0x94D049BB133111EB)
        return ((z ^ (z >> np.uint64(31))) >> np.uint64(11)).astype(np.float64) / 2.0 ** 53
    i = np.arange(M)
    x = u01(3 * i) * cum[-1]
    k = np.minimum(np.searchsorted(cum, x, side="right"), T - 1)
    # a draw within rounding of a boundary (1e-12 of the total) may fall to either side
    clear = np.minimum(np.abs(cum[k] - x), np.abs(x - np.where(k > 0, cum[k - 1], 0))) > 1e-12 * cum[-1]
    assert clear.sum() > 0.99 * M
    u, v = u01(3 * i + 1), u01(3 * i + 2)
    flip = u + v > 1
    u, v = np.where(flip, 1 - u, u)[:, None], np.where(flip, 1 - v, v)[:, None]
    c = t64[k]
    want = c[:, 0] + u * (c[:, 1] - c[:, 0]) + v * (c[:, 2] - c[:, 0])
    # FP32 edge vectors and one rounding of the point: 3 x 2^-24 of coordinates below 1
    assert np.max(np.abs(P - want)[clear]) <= 3e-7
    assert np.array_equal(N[clear], nrm.astype(np.float64)[k][clear])


def _hard_roots(count):
    """Pairs of whole numbers whose y^2 + z^2 (exact in FP64) has a root within
    2^-13 of the middle between two doubles."""
    rng = np.random.default_rng(7)
    y, z = (rng.integers(2 ** 22, 2 ** 24, 4_000_000).astype(np.float64) for _ in range(2))
    s = y * y + z * z
    r = np.sqrt(s)
    c = r * 134217729.0  # Veltkamp's split: r * r = p + e exactly
    hi = c - (c - r)
    lo = r - hi
    p = r * r
    e = ((hi * hi - p) + 2 * hi * lo) + lo * lo
    off = np.abs((s - p) - e) / (2 * r) / np.spacing(r)  # distance of the root from its rounding, in ulps
    k = np.argsort(np.abs(off - 0.5))[:count]
    return y[k].astype(np.float32), z[k].astype(np.float32), s[k]


def test_areas_are_correctly_rounded():
    """Areas 0.5 sqrt(y^2 + z^2) at the hardest roots, bit for bit: the sums in
    the workspace start at each block of 1 024 triangles, here one with an area."""
    import torch
    from paper_2106_03452_gb300 import libdpsr as L
    y, z, s = _hard_roots(1000)
    T = 1024 * len(y)
    tris = torch.zeros((len(y), 1024, 3, 3), device="cuda")
    tris[:, 0, 1, 0] = 1.0  # edges (1, 0, 0) and (0, y, z): cross (0, -z, y)
    tris[:, 0, 2, 1:] = torch.from_numpy(np.stack([y, z], 1)).cuda()
    ws = torch.empty(T + len(y) + 1, dtype=torch.float64, device="cuda")
    out = torch.empty((2, 8, 3), device="cuda")
    nrm = torch.zeros((T, 3), device="cuda")
    L.dpsr_mesh_sample(tris.data_ptr(), nrm.data_ptr(), T, 8, 1, ws.data_ptr(), out[0].data_ptr(), out[1].data_ptr(),
                       torch.cuda.current_stream().cuda_stream)
    got = ws[:T].view(-1, 1024)[:, 0].cpu().numpy()
    assert np.array_equal(got, 0.5 * np.sqrt(s))


@pytest.mark.parametrize("T", [1000, 3000, 2048 * 1024 + 5])
@pytest.mark.parametrize("bad", [np.nan, np.inf])
def test_areas_that_are_not_finite(T, bad):
    """Without a total area there is nothing to search for: every sample falls
    on the last triangle, however many scan blocks there are."""
    import torch
    from paper_2106_03452_gb300.mesh import sample
    tris = torch.rand((T, 3, 3), device="cuda")
    tris[10, 1, 2] = bad
    nrm = torch.arange(T, device="cuda", dtype=torch.float32)[:, None].expand(T, 3).contiguous()
    _, n = sample(tris, nrm, 500, 3)
    assert torch.equal(n, nrm[-1].expand(500, 3))


@pytest.mark.parametrize("T", [1, 2, 1025, 2048 * 1024 + 5])
def test_many_samples_are_the_few(T):
    """A draw depends on its index alone: calls of few and of many samples (blocks
    of 64 and of 128 threads, one and several samples a thread) share theirs."""
    import torch
    from paper_2106_03452_gb300.mesh import sample
    g = torch.Generator("cuda").manual_seed(T)
    tris, nrm = torch.rand((T, 3, 3), device="cuda", generator=g), torch.rand((T, 3), device="cuda", generator=g)
    few = sample(tris, nrm, 68096, 9)
    for M in (1, 68097, 300001):
        many = sample(tris, nrm, M, 9)
        n = min(M, 68096)
        assert torch.equal(many[0][:n], few[0][:n]) and torch.equal(many[1][:n], few[1][:n])
