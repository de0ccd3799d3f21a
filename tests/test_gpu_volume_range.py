"""The voxeliser at the ends of its range: values below the smallest normal FP32 number, more layers than FP32 counts
and a Gaussian over more columns than 32 bits count."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

LAT = {"nx": 8, "ny": 8, "nz": 8, "R": 1, "origin": (-112.0,) * 3, "spacing": (32.0,) * 3}


def _volume(scale, rho, grid, cutoff):
    from paper_2506_22280_gb300 import digs as D
    f = lambda a: torch.tensor(a, dtype=torch.float32, device="cuda")  # noqa: E731
    return D.voxelize(f([[0.0, 0.0, 0.0]]), f([[scale] * 3]), f([[1.0, 0.0, 0.0, 0.0]]), f([rho]),
                      f(np.zeros((1, 8, 8, 8, 3))), f([0.0]), LAT, grid, cutoff=cutoff)


def test_values_below_the_smallest_normal():
    # E up to 196: e^(-E/2) down to 2e-43, in steps of 2^-149.  The exponent's argument, up to 141, carries E's and its
    # own FP32 rounding: 3e-5 of the value at most, 1e-4 allowed.
    n, x0, h, rho = 23, 12.93, 0.05, 1e10
    vol = _volume(1.0, rho, dict(nx=n, ny=1, nz=1, origin=[x0, 0.0, 0.0], spacing=[h, 1.0, 1.0]), 14.0)
    x = np.float32(x0) + np.arange(n) * np.float64(np.float32(h))
    ref = np.where(x * x <= 196.0, rho * np.exp(-0.5 * x * x), 0.0)
    got = vol.cpu().numpy().astype(np.float64).ravel()
    assert np.all(np.abs(got - ref) <= 1e-4 * ref + rho * 2.0 ** -149)


def test_more_layers_than_fp32_counts():
    # 20 layers a sigma around layer 2^24; beyond it FP32 rounds a layer's number to the next even one, a twentieth of a
    # sigma: at most 0.607 / 20 of the peak
    top, sig, h = 1 << 24, 20.0, 2.0 ** -20
    vol = _volume(sig * h, 1.0, dict(nx=1, ny=1, nz=top + 64, origin=[0.0, 0.0, -16.0], spacing=[1.0, 1.0, h]), 3.5)
    k = np.arange(top - 69, top + 64)
    ref = np.exp(-0.5 * ((k - top) / sig) ** 2)
    got = vol[k[0]:].cpu().numpy().astype(np.float64).ravel()
    assert np.all(np.abs(got - ref) <= np.where(k <= top, 1e-5, 0.031))
    assert not vol[:k[0] - 1].any()


def test_more_columns_than_32_bits_count():
    # 46342^2 > 2^31 columns of one layer, all within the Gaussian's cutoff
    n, h = 46342, 1.0
    c = 0.5 * (n - 1)
    vol = _volume(30000.0, 1.0, dict(nx=n, ny=n, nz=1, origin=[-c, -c, 0.0], spacing=[h, h, 1.0]), 3.5)
    for j, i in ((0, 0), (0, n - 1), (n - 1, 0), (n - 1, n - 1), (23171, 23171), (46341, 17), (12345, 45678)):
        want = np.exp(-0.5 * ((i - c) ** 2 + (j - c) ** 2) / 9e8)
        assert abs(float(vol[0, j, i]) - want) <= 1e-5
