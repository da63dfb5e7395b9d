"""How the C++ entries of the hot calls sit in a Python program: what other
threads may do meanwhile."""
import threading
import time

import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2106_03452_gb300 import build
    build.build()


def _cloud(n=3000, seed=0):
    import torch
    g = torch.Generator("cuda").manual_seed(seed)
    d = torch.nn.functional.normalize(torch.randn((n, 3), device="cuda", generator=g), dim=1)
    return (0.5 + 0.3 * d).contiguous(), d


def _ball(r=32):
    import torch
    t = torch.arange(r, device="cuda") / r - 0.5
    return ((t[:, None, None] ** 2 + t[None, :, None] ** 2 + t[None, None, :] ** 2).sqrt() - 0.3).contiguous()


@pytest.mark.parametrize("call", ["extract", "mesh_points", "layer", "forward"])
def test_other_threads_run_while_a_call_waits(call):
    """A call that waits for queued work (the count of an extraction, a plan
    whose workspace grows) leaves the interpreter to other threads."""
    import torch
    from paper_2106_03452_gb300.dpsr import Plan, dpsr
    from paper_2106_03452_gb300.mesh import MeshPoints, extract
    chi, plan = _ball(), Plan(32, 2.0)
    plan.forward(*_cloud(64))
    p, n = _cloud(100000)
    fn = {"extract": lambda: extract(chi), "mesh_points": lambda: MeshPoints.apply(chi, 0.0, 100, 1),
          "layer": lambda: dpsr(p, n, plan), "forward": lambda: plan.forward(p, n)}[call]
    if call in ("extract", "mesh_points"):
        fn()
    torch.cuda._sleep(1000)
    torch.cuda.synchronize()
    stop, gap = threading.Event(), [0.0]

    def count():
        last = time.perf_counter()
        while not stop.is_set():
            now = time.perf_counter()
            gap[0], last = max(gap[0], now - last), now

    thread = threading.Thread(target=count)
    thread.start()
    time.sleep(0.02)
    torch.cuda._sleep(800_000_000)  # some 0.4 s
    t0 = time.perf_counter()
    fn()
    took = time.perf_counter() - t0
    stop.set()
    thread.join()
    torch.cuda.synchronize()
    plan.close()
    if call in ("extract", "mesh_points"):
        assert took > 0.1  # the call did wait
    assert gap[0] <= 0.1, (took, gap[0])
