"""The backward raster ranks the live records of each group of 32 and sweeps them in pairs: groups with an odd number
of records that do not exist (past the cloud) or were culled (off the detector), against the FP64 oracle with the
gradients' bound of 1e-4.  Culled Gaussians get zeros."""
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
@pytest.mark.parametrize("n,culled", [(31, 0), (63, 0), (64, 3), (95, 30), (33, 33)])
def test_groups_with_missing_records(n, culled, lanes):
    import paper_2506_22280_gb300 as pkg
    wl = synth.tiny(seed=n + culled, n=n + 20, n_proj=3, nu=24, nv=19, du=4.3, dv=5.1)
    wl = wl.subset(unambiguous(wl, wl.w, wl.views)[:n])
    assert wl.n == n
    off = np.random.default_rng(n).permutation(n)[:culled]
    wl.mu0[off, 2] += 500.0
    pj = pkg.Projector(wl.lattice, wl.views, bwd_lanes=lanes)
    gp = synth.random_grad_proj(3, 19, 24, seed=n)
    g = pj.backward(T(wl.mu0), T(wl.scale), T(wl.quat), T(wl.rho), T(wl.phi), T(wl.w), T(gp))
    names = ("mu0", "scale", "quat", "rho", "phi", "w")
    if culled == n:  # the oracle's sums over no Gaussian: zero
        assert not any(g[k].any() for k in names)
        return
    ref = O.project_vjp(dict(mu0=wl.mu0, scale=wl.scale, quat=wl.quat, rho=wl.rho), wl.lattice, wl.phi, wl.w,
                        wl.views, gp)
    for k in names:
        a, b = g[k].cpu().numpy(), ref[k]
        assert np.linalg.norm(a - b) <= 1e-4 * np.linalg.norm(b), k
        if a.shape[0] == n and k != "phi":
            assert not a[off].any(), k
