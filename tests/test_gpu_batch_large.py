"""Batches of large grids against solo solves, and batches whose launches are refused."""
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


def _rel(a, b):
    return float((a.double() - b.double()).abs().max() / b.double().abs().max())


def _batch(rs, ns, seed=0):
    """A bound batch and its tensors (points, normals, dchi, chi, dp, dn) per instance."""
    import torch
    from paper_2106_03452_gb300.dpsr import Batch
    b, io = Batch(rs, [2.0] * len(rs), ns), []
    for i, (r, n) in enumerate(zip(rs, ns)):
        rng = synth.Rng(100 * seed + i)
        p, d = (torch.from_numpy(x).cuda() for x in synth.sphere_cloud(rng, n, radius=0.2 + 0.02 * i))
        g = torch.from_numpy(rng.normal(r, r, r).astype(np.float32)).cuda()
        out = [torch.empty((r, r, r), device="cuda"), torch.empty_like(p), torch.empty_like(p)]
        b.bind(i, p, d, out[0], g, out[1], out[2])
        io.append((p, d, g, *out))
    return b, io


def _solo(r, p, d, g):
    from paper_2106_03452_gb300.dpsr import Plan
    plan = Plan(r, 2.0)
    chi = plan.forward(p, d).clone()
    dp, dn = plan.backward(g)
    assert plan.sync() == 0
    plan.close()
    return chi, dp, dn


def _agree(io, rs):
    """chi and gradients of every instance against its solo solve: two solves of
    one cloud differ by the order of their splats' sums."""
    for r, (p, d, g, *out) in zip(rs, io):
        for x, y, tol in zip(out, _solo(r, p, d, g), (1e-5, 1e-4, 1e-4)):
            assert _rel(x, y) <= tol


def test_a_refused_run_leaves_the_batch_usable(monkeypatch):
    """A plane path that does not exist fails each run after the binning has
    counted; the run after the path is gone starts from cleared counters."""
    from paper_2106_03452_gb300 import libdpsr as L
    rs = [64, 64]
    b, io = _batch(rs, [3000, 5000])
    monkeypatch.setenv("DPSR_PLANE_PATHS_64", "2,2,2,2")
    for graph in (False, True, False):
        with pytest.raises(L.DPSRError):
            b.run(graph=graph)
    monkeypatch.delenv("DPSR_PLANE_PATHS_64")
    for graph in (False, True):
        b.run(graph=graph)
        assert b.sync() == 0
        _agree(io, rs)
    b.close()


@pytest.mark.parametrize("path", [None, "4"])
def test_large_grids_in_a_batch(monkeypatch, path):
    """r = 256 and 512 in one batch, their Solve read from the device table: the
    solo solves' results by plain launches, capture and replay, the paths and
    launches that ran (the pencil passes, asked for by a cluster size or not)."""
    if path:
        monkeypatch.setenv("DPSR_PLANE_PATH", path)
    else:
        monkeypatch.delenv("DPSR_PLANE_PATH", raising=False)
    rs = [256, 512, 256] if path is None else [256, 256]  # no cluster size is accepted at r = 512
    b, io = _batch(rs, [20000, 30000, 700][:len(rs)], seed=1)
    for graph in (False, True, True):
        for t in io:
            for x in t[3:]:
                x.fill_(float("nan"))
        b.run(graph=graph)
        assert b.sync() == 0
        _agree(io, rs)
    assert all(list(b.paths(r)) == [0] * 4 for r in set(rs))
    assert b.launches(False) == len(set(rs)) * 7 and b.launches() == len(set(rs)) * 13
    b.close()
