"""The sum of the L_DPSR loss (Eq. 9) against FP64 on the grids that the kernel
reads: what a long FP32 sum per thread would lose has to be there."""
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


@pytest.mark.parametrize("r", [8, 32, 64, 128, 256])
def test_loss_keeps_small_terms(r):
    """Differences of 1 among others of 2^-13, whose squares vanish in an FP32 sum
    that holds a large one. Eight squares are summed in FP32 (a product and three
    levels of sums: a relative error of 4 * 2^-24 at most), the rest in pairs of
    floats; eight float4 in FP32 would lose 31 * 2^-26."""
    import torch
    from paper_2106_03452_gb300.dpsr import Plan
    p, n = synth.sphere_cloud(synth.Rng(r), 2000, jitter=0.01)
    plan = Plan(r, 2.0)
    chi = plan.forward(torch.from_numpy(p).float().cuda(), torch.from_numpy(n).float().cuda())
    for first in (True, False):
        d = torch.full((r ** 3,), 2.0 ** -13, device="cuda")
        if first:
            d[: r ** 3 // 8: 4] = 1.0  # the first float4 of each thread that takes eight, strided
        else:
            d[::32] = 1.0
        target = chi - d.view_as(chi)
        dchi = plan.mse_grad(target)
        diff = (chi - target).double()
        want = (diff * diff).mean().item()
        assert abs(plan.loss() - want) <= 4 * 2.0 ** -24 * want
        assert torch.equal(dchi, (chi - target) * (2.0 / r ** 3))
    plan.close()
