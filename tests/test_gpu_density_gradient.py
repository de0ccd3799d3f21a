"""Projections are linear in the densities, so for any upstream gradient g, sum_n rho_n dL/drho_n = sum_pixels g I.  The
forward and the backward raster evaluate every pair's value by themselves, each with its own rounding: random, a few
1e-7 of a pair at most, so that over the 10^5 pairs here (and 2,000 records, 65,000 pixels rounded once) it averages to
some 1e-8 of the sum; 2e-8 is allowed.  A systematic error of either side does not average out: a density gradient
formed from 1 / D and multiplied by D again, with the reciprocal square root's own error in between, was off by 4e-8."""
import numpy as np
import pytest
import torch

import synth

pytestmark = pytest.mark.gpu


def T(a):
    return torch.as_tensor(np.asarray(a), dtype=torch.float32, device="cuda").contiguous()


@pytest.mark.parametrize("lanes", [16, 32])
@pytest.mark.parametrize("ewa", [False, True])
def test_density_gradient_has_no_bias(ewa, lanes):
    import paper_2506_22280_gb300 as pkg
    wl = synth.tiny(seed=5, n=2000, n_proj=16)
    args = [T(wl.mu0), T(wl.scale), T(wl.quat), T(wl.rho), T(wl.phi), T(wl.w)]
    pj = pkg.Projector(wl.lattice, wl.views, bwd_lanes=lanes, ewa=ewa)
    img = pj.forward(*args)
    g = pj.backward(*args, torch.ones_like(img))
    left, right = float((args[3].double() * g["rho"].double()).sum()), float(img.double().sum())
    assert abs(left - right) <= 2e-8 * right
