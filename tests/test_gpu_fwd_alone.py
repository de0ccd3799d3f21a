"""A projection is the same, bit for bit, whichever views are rendered beside it: one view alone against the same view
in a call of many, at sizes whose launches have few and many thread blocks, for each tile size."""
import pytest
import torch

from test_gpu_bin_routes import _views

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("tile", [8, 16, 32])
@pytest.mark.parametrize("n,edge,P", [(3000, 128, 2), (3000, 512, 40), (20_000, 256, 40)])
def test_a_view_alone_and_among_others(n, edge, P, tile):
    import paper_2506_22280_gb300 as pkg
    g = torch.Generator(device="cuda").manual_seed(n)
    d = torch.randn(n, 3, generator=g, device="cuda")
    x = 60.0 * d / d.norm(dim=1, keepdim=True) * torch.rand(n, 1, generator=g, device="cuda") ** (1 / 3)
    s = 1.0 + torch.rand(n, 3, generator=g, device="cuda")
    q = torch.randn(n, 4, generator=g, device="cuda")
    rho = 0.01 * torch.rand(n, generator=g, device="cuda")
    lat = {"nx": 8, "ny": 8, "nz": 8, "R": 1, "origin": (-100.0,) * 3, "spacing": (28.0,) * 3}
    phi = torch.randn(1, 8, 8, 8, 3, generator=g, device="cuda")
    w = torch.randn(P, 1, generator=g, device="cuda")
    views, p = _views(P, edge, 200.0 / edge), P // 2
    many = pkg.Projector(lat, views, tile=tile).forward(x, s, q, rho, phi, w)
    one = pkg.Projector(lat, views[p:p + 1], tile=tile).forward(x, s, q, rho, phi, w[p:p + 1].contiguous())
    assert float(one.abs().max()) > 0 and torch.equal(one[0], many[p])
