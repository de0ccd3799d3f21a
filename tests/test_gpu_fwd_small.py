"""Gaussians from a tenth of a pixel to a pixel wide: the forward raster against the FP64 oracle where the set-up's own
rounding cannot hide the raster's.  Parallel beams along an axis, no motion, one-millimetre pixels, means on 1/64 of a
pixel and power-of-two scales: every record is exact in FP32 up to a few units in the last place of the quadratic form.

Bound: E takes about five FP32 roundings of terms that do not cancel (3e-7 E; E e^-E/2 weighs E at about 2: 3e-7 of the
value), the exponential, reciprocal square root and amplitude 4e-7, the record 3e-7 and the pixel's sum 1e-7: 1.1e-6
at the worst of each, 2e-6 is allowed.  The cutoff of 3.3 lies 1e-5 off any E that these means and scales can give."""
import numpy as np
import pytest
import torch

from oracle import digs_oracle as O

pytestmark = pytest.mark.gpu


def T(a):
    return torch.as_tensor(np.asarray(a), dtype=torch.float32, device="cuda").contiguous()


@pytest.mark.parametrize("tile", [8, 16, 32])
@pytest.mark.parametrize("sigma", [0.0625, 0.125, 0.25, 0.5, 1.0])
def test_small_gaussians(sigma, tile):
    import paper_2506_22280_gb300 as pkg
    rng = np.random.default_rng(int(1000 * sigma))
    n, nu, nv = 3000, 61, 54
    mu0 = np.zeros((n, 3))
    mu0[:, 1:] = rng.integers(-28 * 64, 28 * 64, size=(n, 2)) / 64.0
    scale = np.full((n, 3), sigma)
    quat = np.tile([1.0, 0.0, 0.0, 0.0], (n, 1))
    rho = (0.5 + rng.uniform(size=n)).astype(np.float32).astype(np.float64)
    lat = {"nx": 8, "ny": 8, "nz": 8, "R": 1, "origin": np.full(3, -112.0), "spacing": np.full(3, 32.0)}
    phi, w = np.zeros((1, 8, 8, 8, 3)), np.zeros((1, 1))
    view = dict(src=np.array([1024.0, 0.0, 0.0]), det_c=np.array([-512.0, 0.0, 0.0]), e_u=np.array([0.0, 1.0, 0.0]),
                e_v=np.array([0.0, 0.0, 1.0]), du=1.0, dv=1.0, off_u=0.0, off_v=0.0, nu=nu, nv=nv, parallel=True)
    img = pkg.Projector(lat, [view], tile=tile, cutoff=3.3).forward(T(mu0), T(scale), T(quat), T(rho), T(phi), T(w))
    ref = O.render(dict(mu0=mu0, scale=scale, quat=quat, rho=rho), lat, phi, w, [view], cutoff=3.3)
    assert np.count_nonzero(ref) > 100
    assert np.linalg.norm(img.cpu().numpy() - ref) <= 2e-6 * np.linalg.norm(ref)
