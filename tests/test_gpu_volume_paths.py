"""Voxeliser and displacement field at the sizes where their launch shapes change, against the FP64 oracle.

The cutoff is 12 here: a voxel whose distance lies within rounding of it then carries e^-72 of a peak, so the
bound is rounding alone (the 1e-5 of the projections: about 20 FP32 roundings of a few 1e-7)."""
import numpy as np
import pytest
import torch

import synth
from oracle import digs_oracle as O

pytestmark = pytest.mark.gpu


def T(a):
    return torch.as_tensor(np.asarray(a), dtype=torch.float32, device="cuda").contiguous()


def scene(R, dims, spacing):
    wl = synth.tiny(seed=3, n=37)
    rng = np.random.default_rng(7)
    grid = dict(nx=dims[0], ny=dims[1], nz=dims[2], spacing=list(spacing),
                origin=[-0.5 * (dims[a] - 1) * spacing[a] + 0.3 for a in range(3)])
    return wl, dict(wl.lattice, R=R), rng.normal(size=(R, 8, 8, 8, 3)), rng.normal(size=R), grid


@pytest.mark.parametrize("R,dims,spacing", [
    (2, (1, 1, 1), (3.0, 3.0, 3.0)),           # one voxel
    (1, (129, 17, 5), (0.5, 2.0, 7.0)),        # boxes of many columns, one layer deep
    (3, (70, 9, 6), (0.25, 4.0, 5.0)),         # boxes wider than a warp
])
def test_voxelize_launch_shapes(R, dims, spacing):
    from paper_2506_22280_gb300 import digs as D
    wl, lat, phi, w, grid = scene(R, dims, spacing)
    vol = D.voxelize(T(wl.mu0), T(wl.scale), T(wl.quat), T(wl.rho), T(phi), T(w), lat, grid, cutoff=12.0)
    ref = O.voxelize(dict(mu0=wl.mu0, scale=wl.scale, quat=wl.quat, rho=wl.rho), lat, phi, w, grid, cutoff=12.0)
    assert np.linalg.norm(vol.cpu().numpy() - ref) <= 1e-5 * np.linalg.norm(ref)


@pytest.mark.parametrize("R,dims,spacing", [
    (2, (1, 1, 1), (3.0, 3.0, 3.0)),           # one voxel
    (1, (129, 17, 5), (0.5, 2.0, 7.0)),        # one past a 128-voxel row slice and a 16-row group
    (4, (20, 21, 3), (40.0, 3.0, 20.0)),       # voxels so coarse that each is evaluated by itself
    (2, (40, 19, 4), (20.0, 30.0, 9.0)),       # fewer voxels and rows per block than its threads allow
])
def test_dvf_launch_shapes(R, dims, spacing):
    from paper_2506_22280_gb300 import digs as D
    _, lat, phi, w, grid = scene(R, dims, spacing)
    d, dref = D.dvf(T(phi), T(w), lat, grid).cpu().numpy(), O.dvf(lat, phi, w, grid)
    assert np.linalg.norm(d - dref) <= 1e-5 * np.linalg.norm(dref)
