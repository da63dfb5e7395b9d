"""Mesh extraction of one grid at an aligned and at an odd address: the two read
and share out the cubes differently, by size, and cut the same triangles."""
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2106_03452_gb300 import build
    build.build()


def _cut(chi, level):
    """(sorted triangles with normals, count) by dpsr_mesh_extract."""
    import torch
    from paper_2106_03452_gb300 import libdpsr as L
    r = chi.shape[0]
    st = torch.cuda.current_stream().cuda_stream
    n = torch.zeros(1, dtype=torch.int64, device="cuda")
    L.dpsr_mesh_extract(chi.data_ptr(), r, level, 0, 0, 0, n.data_ptr(), st)
    count = int(n.item())
    tris, nrm = torch.empty((max(count, 1), 9), device="cuda"), torch.empty((max(count, 1), 3), device="cuda")
    L.dpsr_mesh_extract(chi.data_ptr(), r, level, tris.data_ptr(), nrm.data_ptr(), count, n.data_ptr(), st)
    assert int(n.item()) == count
    return torch.cat([tris, nrm], 1)[:count].cpu().unique(dim=0), count


@pytest.mark.parametrize("r", [2, 4, 8, 32, 64])
def test_aligned_and_odd_addresses_agree(r):
    import torch
    g = torch.Generator("cuda").manual_seed(r)
    for chi, level in ((torch.randn((r, r, r), device="cuda", generator=g), 0.0),
                       (torch.rand((r, r, r), device="cuda", generator=g), 0.97), (torch.ones((r, r, r), device="cuda"), 0.0)):
        odd = torch.empty(r ** 3 + 1, device="cuda")[1:].view(r, r, r)
        odd.copy_(chi)
        (a, na), (b, nb) = _cut(chi, level), _cut(odd, level)
        assert na == nb and torch.equal(a, b)
