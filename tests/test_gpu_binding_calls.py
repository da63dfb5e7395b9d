"""How the C++ entries of the hot calls sit in a Python program: what other
threads may do meanwhile, subclasses of the classes that call them, streams."""
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


def test_subclasses_answer_for_themselves():
    """A subclass of a function or of the plan keeps its own methods."""
    import torch
    from paper_2106_03452_gb300.dpsr import DPSRFunction, Plan, dpsr
    from paper_2106_03452_gb300.loop import GridSample
    from paper_2106_03452_gb300.mesh import MeshPoints
    from paper_2106_03452_gb300.optimize import ChamferLoss
    p, n = _cloud()
    calls = []

    class Own(Plan):
        def forward(self, points, normals, chi_out=None):
            calls.append("forward")
            return super().forward(points, normals, chi_out)

        def backward(self, dchi, dpoints=None, dnormals=None):
            calls.append("backward")
            return super().backward(dchi, dpoints, dnormals)

        def _bind_stream(self):
            calls.append("stream")
            super()._bind_stream()

    plan = Own(32, 2.0)
    a = p.clone().requires_grad_(True)
    dpsr(a, n, plan).sum().backward()
    assert calls == ["forward", "stream", "backward", "stream"]
    plan.close()

    def zeros(base, k):
        class Zero(base):
            @staticmethod
            def backward(ctx, *g):
                return (torch.zeros_like(ctx.x),) + (None,) * k

            @staticmethod
            def forward(ctx, x, *rest):
                ctx.x = x
                return base.forward(ctx, x, *rest)
        return Zero

    plan, chi = Plan(32, 2.0), _ball()
    for fn, k, x, rest in ((DPSRFunction, 2, p, (n, plan)), (GridSample, 1, chi, (p,)), (ChamferLoss, 1, p, (p + 0.1,)),
                           (MeshPoints, 3, chi, (0.0, 0, 0))):
        x = x.clone().requires_grad_(True)
        out = zeros(fn, k).apply(x, *rest)
        (g,) = torch.autograd.grad((out[0] if isinstance(out, tuple) else out).sum(), x)
        assert not g.any(), fn
    plan.close()


@pytest.mark.parametrize("r", [32, 64, 256])
def test_a_side_stream_waits_for_its_own_inputs(r):
    """The inputs are written on a side stream, behind a long kernel, right before
    the call: work on any other stream would read what was there before. The
    upstream gradient is random: the layer is well conditioned then, and two solves
    of one cloud differ by some 5e-7 of the largest value (their splats' sums run
    in no fixed order), where chi.square().sum() turns the same rounding into 1e-4."""
    import torch
    from paper_2106_03452_gb300.dpsr import Plan, dpsr
    from paper_2106_03452_gb300.optimize import chamfer
    (p, n), (p0, n0) = _cloud(3000, 1), _cloud(3000, 2)
    w = torch.randn((r, r, r), device="cuda", generator=torch.Generator("cuda").manual_seed(r))
    plan = Plan(r, 2.0)

    def step(a, b, g, q):
        chi = dpsr(a, b, plan)
        return [chi.detach(), *torch.autograd.grad(chi, (a, b), g), *torch.autograd.grad(chamfer(a, q), a)]

    def inputs(p, n, w, q):
        return p.clone().requires_grad_(True), n.clone().requires_grad_(True), w.clone(), q.clone()

    want = step(*inputs(p, n, w, p0))
    late = inputs(p0, n0, torch.zeros_like(w), p)
    other = step(*inputs(p0, n0, w, p))
    st = torch.cuda.Stream()
    st.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(st):
        torch.cuda._sleep(100_000_000)  # some 50 ms
        with torch.no_grad():
            for x, y in zip(late, (p, n, w, p0)):
                x.copy_(y)
        got = step(*late)
    torch.cuda.current_stream().wait_stream(st)
    for x, y, z in zip(got, want, other):
        scale = float(y.abs().max())
        assert float((x - y).abs().max()) <= 1e-5 * scale
        assert float((z - y).abs().max()) >= 1e-2 * scale  # the inputs before would have shown
    plan.close()


def test_a_plan_without_a_name_answers_as_another():
    """The graph keeps a plan that went out of scope; with a random upstream
    gradient (see above)."""
    import gc
    import torch
    from paper_2106_03452_gb300.dpsr import Plan, dpsr
    p, n = _cloud()
    w = torch.randn((32, 32, 32), device="cuda")
    a = p.clone().requires_grad_(True)
    plan = Plan(32, 2.0)
    (want,) = torch.autograd.grad(dpsr(a, n, plan), a, w)
    chi = dpsr(a, n, Plan(32, 2.0))
    gc.collect()
    (got,) = torch.autograd.grad(chi, a, w)
    assert float((got - want).abs().max()) <= 1e-5 * float(want.abs().max())
    plan.close()


def test_threads_with_plans_of_their_own(tmp_path):
    """Eight threads solve at once from the first call of a process on, each with
    its plan and stream (the kernels' set-up is shared): the results of one thread."""
    import os
    import subprocess
    import sys
    code = """
import sys, threading
import torch
from paper_2106_03452_gb300.dpsr import Plan, dpsr
from paper_2106_03452_gb300.mesh import MeshPoints
from paper_2106_03452_gb300.optimize import chamfer
def cloud(k):
    g = torch.Generator("cuda").manual_seed(k)
    d = torch.nn.functional.normalize(torch.randn((2000 + 300 * k, 3), device="cuda", generator=g), dim=1)
    return (0.5 + 0.3 * d).contiguous(), d, torch.randn((R[k],) * 3, device="cuda", generator=g)
R = (32, 64, 128, 256, 32, 64, 128, 256)
def solve(k, plan):
    p, d, w = IN[k]
    a = p.clone().requires_grad_(True)
    chi = dpsr(a, d, plan)
    (g,) = torch.autograd.grad(chi, a, w)
    m, _ = MeshPoints.apply(chi.detach(), 0.0, 500, k)
    return [chi.detach(), g, chamfer(p, p.flip(0) + 0.01), torch.tensor(float(m.shape[0]))]
IN = [cloud(k) for k in range(8)]
torch.cuda.synchronize()
out, err, go = [None] * 8, [], threading.Barrier(8)
def work(k):
    try:
        st = torch.cuda.Stream()
        with torch.cuda.stream(st):
            plan = Plan(R[k], 2.0)
            go.wait()
            for _ in range(5):
                out[k] = solve(k, plan)
            st.synchronize()
            assert plan.sync() == 0
    except BaseException as e:
        err.append(repr(e))
        go.abort()
ts = [threading.Thread(target=work, args=(k,)) for k in range(8)]
[t.start() for t in ts]
[t.join() for t in ts]
assert not err, err
for k in range(8):
    for x, y in zip(out[k], solve(k, Plan(R[k], 2.0))):
        assert float((x - y).abs().max()) <= 1e-5 * float(y.abs().max()), k
print("fine")
"""
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    for tune in ("1", "0"):
        r = subprocess.run([sys.executable, "-c", code], cwd=root, capture_output=True, text=True, timeout=300,
                           env={**os.environ, "DPSR_TUNE": tune, "PYTHONPATH": root})
        assert r.returncode == 0 and "fine" in r.stdout, r.stderr[-3000:]
