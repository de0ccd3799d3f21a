"""The forward raster's launch shapes (list splits per tile size, on both sides of the line between them) against
the FP64 oracle, from an empty tile list to lists that end inside a batch of 32.  Bound: the projections' 1e-5."""
import numpy as np
import pytest
import torch

import synth
from oracle import digs_oracle as O

pytestmark = pytest.mark.gpu


def T(a):
    return torch.as_tensor(np.asarray(a), dtype=torch.float32, device="cuda").contiguous()


@pytest.mark.parametrize("tile,views,edge", [(8, 2, 64), (8, 5, 512), (16, 3, 72), (16, 9, 512), (32, 2, 100), (32, 17, 512)])
@pytest.mark.parametrize("n", [1, 33, 400])
def test_forward_launch_shapes(n, tile, views, edge):
    import paper_2506_22280_gb300 as pkg
    wl = synth.tiny(seed=n, n=n, n_proj=views, nu=edge, nv=edge - 5, du=102.4 / edge, dv=102.4 / edge)
    pj = pkg.Projector(wl.lattice, wl.views, tile=tile)
    args = [T(wl.mu0), T(wl.scale), T(wl.quat), T(wl.rho), T(wl.phi), T(wl.w)]
    img = pj.forward(*args).cpu().numpy()
    assert pj.status() == 0
    ref = O.render(dict(mu0=wl.mu0, scale=wl.scale, quat=wl.quat, rho=wl.rho), wl.lattice, wl.phi, wl.w, wl.views)
    assert np.linalg.norm(img - ref) <= 1e-5 * np.linalg.norm(ref)
    meas = T(0.9 * ref + 0.01)
    out = torch.empty_like(meas)
    loss = float(pj.loss(*args, meas, proj=out).item())
    want = O.mse_loss(ref, 0.9 * ref + 0.01)
    assert np.linalg.norm(out.cpu().numpy() - ref) <= 1e-5 * np.linalg.norm(ref) and abs(loss - want) <= 1e-5 * want
