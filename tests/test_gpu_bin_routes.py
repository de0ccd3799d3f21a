"""The prefix sum and the tile lists take one of several routes by size: one tile of counts, blocks that add up the
sums before theirs, a launch in between (more than 4096 tiles of 4096 counts); list ranges formed with the launch
order (up to 4096 lists) or by themselves.  A call over several views and calls over single views take different
routes to the same lists; their images agree within the projections' bound of 1e-5 (a list's split over warps may
differ)."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


def _views(P, n, pitch):
    out = []
    for p in range(P):
        a = 0.1 + 2 * np.pi * p / P
        cs, sn = float(np.cos(a)), float(np.sin(a))
        out.append({"src": (1000.0 * cs, 1000.0 * sn, 0.0), "det_c": (-500.0 * cs, -500.0 * sn, 0.0),
                    "e_u": (-sn, cs, 0.0), "e_v": (0.0, 0.0, 1.0), "du": pitch, "dv": pitch, "off_u": 0.0,
                    "off_v": 0.0, "nu": n, "nv": n, "parallel": False, "scan": 0})
    return out


@pytest.mark.parametrize("n,edge,P", [(200, 64, 2),        # 32 counts against 16: one tile
                                      (3000, 256, 2),      # 6144 counts against 3072: two tiles, one
                                      (20_000, 256, 17),   # 4352 lists against 256
                                      (500_000, 512, 9)])  # 18.0 M counts: more than 4096 tiles
def test_views_together_equal_views_alone(n, edge, P):
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
    views = _views(P, edge, 200.0 / edge)
    both = pkg.Projector(lat, views, tile=16).forward(x, s, q, rho, phi, w)
    assert float(both.abs().max()) > 0
    for p in range(P):
        one = pkg.Projector(lat, views[p:p + 1], tile=16).forward(x, s, q, rho, phi, w[p:p + 1].contiguous())
        assert float((one[0] - both[p]).norm()) <= 1e-5 * float(both[p].norm())
