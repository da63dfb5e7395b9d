"""The C++ autograd functions of the hot calls against the Python classes that
answer for everything they do not take: the same values and gradients, the
same errors, and plans, graphs and streams used as a program may use them."""
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


def _python(fn, *args):
    """The Python class' own path, whatever the binding would take."""
    import torch
    return super(fn, fn).apply(*args) if issubclass(fn, torch.autograd.Function) else fn(*args)


def _rel(a, b):
    return float((a.double() - b.double()).abs().max() / b.double().abs().max())


def test_layer_equals_the_python_path():
    import torch
    from paper_2106_03452_gb300 import libdpsr as L
    from paper_2106_03452_gb300.dpsr import DPSRFunction, Plan, dpsr
    p, n = _cloud()
    plan = Plan(32, 2.0)
    assert L.binding().layer(p, n, plan) is not None
    w = torch.randn((32, 32, 32), device="cuda")
    out = []
    for call in (lambda a, b: dpsr(a, b, plan), lambda a, b: _python(DPSRFunction, a, b, plan)):
        a, b = p.clone().requires_grad_(True), n.clone().requires_grad_(True)
        scale = torch.full((1,), 1.5, device="cuda", requires_grad=True)
        chi = call(a * 1.0, b * scale)          # not leaves
        (chi * w).sum().backward(retain_graph=True)
        first = a.grad.clone()
        (chi * w).sum().backward()              # any number of backward passes
        assert _rel(a.grad, 2 * first) <= 1e-5
        out.append((chi.detach(), a.grad, b.grad, scale.grad))
    # two solves of one cloud differ by the order of their splats' atomic sums
    assert _rel(out[0][0], out[1][0]) <= 1e-5
    assert all(_rel(x, y) <= 1e-4 for x, y in zip(out[0][1:3], out[1][1:3]))
    # a gradient that is expanded, not dense
    a = p.clone().requires_grad_(True)
    (g,) = torch.autograd.grad(dpsr(a, n, plan).sum(), a)
    (h,) = torch.autograd.grad(_python(DPSRFunction, a, n, plan).sum(), a)
    assert _rel(g, h) <= 1e-4
    plan.close()


def test_plan_state_is_the_python_path_s():
    import torch
    from paper_2106_03452_gb300 import libdpsr as L
    from paper_2106_03452_gb300.dpsr import Plan, dpsr
    p, n = _cloud()
    plan = Plan(32, 2.0)
    with pytest.raises(L.DPSRError):
        plan.backward(torch.zeros((32, 32, 32), device="cuda"))
    a = p.clone().requires_grad_(True)
    chi = dpsr(a, n, plan)
    g0 = plan.generation
    dp, _ = plan.backward(torch.ones((32, 32, 32), device="cuda"))  # the plan's own backward follows
    assert dp.shape == p.shape and plan.generation == g0
    plan.forward(p, n)
    assert plan.generation == g0 + 1
    with pytest.raises(RuntimeError, match="another forward pass"):
        chi.sum().backward()
    with torch.no_grad():
        assert not dpsr(a, n, plan).requires_grad
    chi = dpsr(a, n, plan)
    plan.close()
    with pytest.raises(L.DPSRError) as e:
        chi.sum().backward()
    assert e.value.code == L.DPSR_EINVAL
    with pytest.raises(L.DPSRError):
        dpsr(a, n, plan)


def test_plan_outlives_its_name():
    """The graph keeps the plan: a plan that went out of scope still answers."""
    import gc
    import torch
    from paper_2106_03452_gb300.dpsr import Plan, dpsr
    p, n = _cloud()
    a = p.clone().requires_grad_(True)
    plan = Plan(32, 2.0)
    (want,) = torch.autograd.grad(dpsr(a, n, plan).square().sum(), a)
    chi = dpsr(a, n, Plan(32, 2.0))
    gc.collect()
    (got,) = torch.autograd.grad(chi.square().sum(), a)
    assert _rel(got, want) <= 1e-4


def test_what_was_refused_is_refused():
    import torch
    from paper_2106_03452_gb300 import libdpsr as L
    from paper_2106_03452_gb300.dpsr import Plan, dpsr
    from paper_2106_03452_gb300.loop import GridSample
    from paper_2106_03452_gb300.mesh import MeshPoints, extract
    from paper_2106_03452_gb300.optimize import chamfer
    p, n = _cloud(64)
    plan = Plan(32, 2.0)
    for bad, err in (((p.cpu(), n.cpu()), TypeError), ((p.double(), n.double()), TypeError),
                     ((p, n[:-1]), ValueError), ((p[:, :2], n[:, :2]), ValueError), ((p[:0], n[:0]), L.DPSRError)):
        with pytest.raises(err):
            dpsr(*bad, plan)
    q = p.requires_grad_(True)
    with pytest.raises(RuntimeError), torch.autograd.forward_ad.dual_level():
        dpsr(torch.autograd.forward_ad.make_dual(p.detach(), n), n, plan)
    with pytest.raises(RuntimeError):
        torch.func.vmap(lambda x: dpsr(x, n, plan))(torch.stack([p.detach(), p.detach()]))
    with pytest.raises(ValueError):
        extract(torch.zeros((8, 8, 8)))
    with pytest.raises(L.DPSRError):
        GridSample.apply(torch.zeros((12, 12, 12), device="cuda"), p.detach())  # not a power of two
    with pytest.raises(L.DPSRError):
        MeshPoints.apply(torch.zeros((12, 12, 12), device="cuda"))
    with pytest.raises(L.DPSRError):
        chamfer(q[:0], p)
    # accepted before, and still: another layout goes the Python way
    t = torch.empty((3, 64), device="cuda").t()
    t.copy_(p.detach())
    assert L.binding().layer(t, n, plan) is None
    assert _rel(dpsr(t, n, plan), dpsr(p.detach(), n, plan)) <= 1e-5

    class Sub(torch.Tensor):
        pass

    assert L.binding().layer(p.detach().as_subclass(Sub), n, plan) is None
    plan.close()


def test_losses_equal_the_python_path():
    import torch
    from paper_2106_03452_gb300.loop import GridSample
    from paper_2106_03452_gb300.mesh import MeshPoints, extract, sample
    from paper_2106_03452_gb300.optimize import ChamferLoss
    g = torch.Generator("cuda").manual_seed(3)
    q = torch.rand((5000, 3), device="cuda", generator=g)
    t = (torch.arange(32, device="cuda") / 32 - 0.5)
    chi = ((t[:, None, None] ** 2 + t[None, :, None] ** 2 + t[None, None, :] ** 2).sqrt() - 0.3).contiguous()
    w = torch.randn(5000, device="cuda", generator=g)
    for native in (True, False):
        c = chi.clone().requires_grad_(True)
        v = GridSample.apply(c, q) if native else _python(GridSample, c, q)
        (d,) = torch.autograd.grad(v, c, w)
        a = q.clone().requires_grad_(True)
        loss = ChamferLoss.apply(a, q[:3000] + 0.01) if native else _python(ChamferLoss, a, q[:3000] + 0.01)
        (da,) = torch.autograd.grad(loss * 2.0, a)
        c = chi.clone().requires_grad_(True)
        p, n = MeshPoints.apply(c) if native else _python(MeshPoints, c, 0.0, 0, 0)
        assert not n.requires_grad and p.requires_grad and p.shape == n.shape
        (m,) = torch.autograd.grad((p - 0.5).square().sum(), c)
        if native:
            kept = v.detach(), d, loss.detach(), da, m, p.shape[0]
        else:
            # sums of float atomics, in any order: the two agree to their rounding
            assert torch.equal(v.detach(), kept[0]) and _rel(d, kept[1]) <= 1e-5
            assert _rel(loss.detach(), kept[2]) <= 1e-6 and _rel(da, kept[3]) <= 1e-5
            assert _rel(m, kept[4]) <= 1e-5 and p.shape[0] == kept[5]
    tris, nrm = extract(chi)
    s1, s2 = sample(tris, nrm, 999, seed=-7), sample(tris.transpose(1, 2).contiguous().transpose(1, 2), nrm, 999, seed=-7)
    assert torch.equal(s1[0], s2[0]) and torch.equal(s1[1], s2[1])
    p, n = MeshPoints.apply(chi, 0.0, 500, 11)
    assert p.shape == (500, 3) and n.shape == (500, 3)


def test_on_another_stream():
    import torch
    from paper_2106_03452_gb300.dpsr import Plan, dpsr
    p, n = _cloud()
    plan = Plan(64, 2.0)
    a = p.clone().requires_grad_(True)
    (want,) = torch.autograd.grad(dpsr(a, n, plan).square().sum(), a)
    st = torch.cuda.Stream()
    st.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(st):
        for _ in range(3):
            (got,) = torch.autograd.grad(dpsr(a, n, plan).square().sum(), a)
    torch.cuda.current_stream().wait_stream(st)
    assert _rel(got, want) <= 1e-4
    plan.close()
