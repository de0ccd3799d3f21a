"""The CNN's FP32 and tensor-core modes on one workspace: each mode's backward reads what its own forward kept, and
writes only buffers of its own size.  The FP32 gradient against the FP64 oracle at batches on both sides of 96 (a
gradient buffer of the first convolution is twice that of the second) with the bound of the other FP32 comparisons."""
import numpy as np
import pytest
import torch

from oracle import cnn_oracle as C
from test_gpu_cnn import P, R, _inputs, _stable_masks, relL2  # noqa: F401

pytestmark = pytest.mark.gpu


def _batch(B, seed):
    img, cs = _inputs(B, seed=seed)
    gw = np.random.default_rng(seed + 1).normal(size=(B, R)).astype(np.float32)
    return img, cs, gw, [torch.as_tensor(a, device="cuda") for a in (img, cs, gw)]


@pytest.mark.parametrize("B", [37, 77, 97, 130])
def test_fp32_forward_and_gradient(P, B):  # noqa: F811
    net = P.WeightPredictor(R, seed=6)
    _stable_masks(net, seed=60 + B)
    img, cs, gw, (I, Cs, G) = _batch(B, 13)
    flat = net.params.cpu().numpy().astype(np.float64)
    assert relL2(net.forward(I, Cs).cpu().numpy(), C.forward(flat, R, img, cs)) < 1e-5
    g, gref = net.backward(G).cpu().numpy(), C.vjp(flat, R, img, cs, gw)
    off = 0
    for name, shape in C.param_shapes(R):
        k = int(np.prod(shape))
        assert relL2(g[off:off + k], gref[off:off + k]) < 1e-4, name
        off += k


@pytest.mark.parametrize("B", [6, 130])
def test_fp32_backward_leaves_the_tensor_core_mode_alone(P, B):  # noqa: F811
    _, _, _, (I, Cs, G) = _batch(B, 17)
    grads = []
    for fp32 in (False, True):
        net = P.WeightPredictor(R, seed=6)
        _stable_masks(net, seed=70)
        if fp32:
            net.forward(I, Cs)
        net.forward(I, Cs, tensor_cores=True)
        if fp32:
            net.backward(G)
        grads.append(net.backward(G, tensor_cores=True))
    assert torch.equal(grads[0], grads[1])
