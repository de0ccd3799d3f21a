"""The backward raster's launch shapes (one warp or several per group of 32 records, 16 and 32 lanes per record) at
group remainders and on both sides of the line between them, against the FP64 oracle.  Bound: the gradients'
1e-4, on the Gaussians whose every pixel decision is outside FP32 rounding."""
import numpy as np
import pytest
import torch

import synth
from conftest import unambiguous
from oracle import digs_oracle as O

pytestmark = pytest.mark.gpu


def T(a):
    return torch.as_tensor(np.asarray(a), dtype=torch.float32, device="cuda").contiguous()


@pytest.mark.parametrize("lanes", [16, 32])
@pytest.mark.parametrize("n,views", [(1, 2), (33, 3), (70, 2), (2200, 128)])
def test_backward_launch_shapes(n, views, lanes):
    import paper_2506_22280_gb300 as pkg
    wl = synth.tiny(seed=n + 1, n=n, n_proj=views, nu=24, nv=19, du=4.3, dv=5.1)
    wl = wl.subset(unambiguous(wl, wl.w, wl.views))
    pj = pkg.Projector(wl.lattice, wl.views, bwd_lanes=lanes)
    gp = synth.random_grad_proj(views, 19, 24, seed=n)
    g = pj.backward(T(wl.mu0), T(wl.scale), T(wl.quat), T(wl.rho), T(wl.phi), T(wl.w), T(gp))
    ref = O.project_vjp(dict(mu0=wl.mu0, scale=wl.scale, quat=wl.quat, rho=wl.rho), wl.lattice, wl.phi, wl.w,
                        wl.views, gp)
    for k in ("mu0", "scale", "quat", "rho", "phi", "w"):
        a, b = g[k].cpu().numpy(), ref[k]
        assert np.linalg.norm(a - b) <= 1e-4 * np.linalg.norm(b), k
