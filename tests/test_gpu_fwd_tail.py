"""The last batch of a tile's list is rarely full.  A Gaussian without density, appended to a cloud, makes a batch of one
record after full ones and must not change a bit of any projection: needles, whose quadratic form's FP32 value can
round below zero where its terms cancel, were counted twice by lanes that still held a record of the batch before."""
import math

import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


def T(a):
    return torch.as_tensor(np.asarray(a), dtype=torch.float32, device="cuda").contiguous()


@pytest.mark.parametrize("tile", [8, 16, 32])
@pytest.mark.parametrize("thin", [3e-3, 1e-3, 3e-4])
def test_appended_empty_gaussian_changes_nothing(tile, thin):
    import paper_2506_22280_gb300 as pkg
    rng = np.random.default_rng(5)
    n = 256  # whole batches of 32 for any split of the list over warps
    mu0 = np.zeros((n + 1, 3))
    mu0[:n, 1:] = rng.integers(-3, 3, size=(n, 1)) + 0.5  # on a diagonal of pixel centres, along it
    scale = np.tile([1.0, 6.0, thin], (n + 1, 1))
    scale[:n, 2] *= rng.uniform(0.7, 1.4, size=n)
    scale[n] = 8.0
    half = np.full(n + 1, math.pi / 8)
    quat = np.stack([np.cos(half), np.sin(half), 0 * half, 0 * half], 1)
    rho = np.ones(n + 1)
    rho[n] = 0.0
    lat = {"nx": 8, "ny": 8, "nz": 8, "R": 1, "origin": (-112.0,) * 3, "spacing": (32.0,) * 3}
    phi, w = T(np.zeros((1, 8, 8, 8, 3))), T(np.zeros((1, 1)))
    view = dict(src=(1024.0, 0.0, 0.0), det_c=(-512.0, 0.0, 0.0), e_u=(0.0, 1.0, 0.0), e_v=(0.0, 0.0, 1.0), du=1.0, dv=1.0,
                off_u=0.0, off_v=0.0, nu=48, nv=48, parallel=True)
    img = [pkg.Projector(lat, [view], tile=tile).forward(*(T(a[:k]) for a in (mu0, scale, quat, rho)), phi, w)
           for k in (n, n + 1)]
    assert int((img[0] != 0).sum()) > 0
    assert torch.equal(img[0], img[1])
