"""The tensor-core convolutions at batches where their tiles end: one image, an odd batch (the last
convolution's tiles hold two images) and more tiles than SMs, against the FP64 oracle with the operands
rounded alike.  Tolerances and parameters are those of the other tensor-core comparisons: ReLU decisions
fixed by construction, so that FP32 summation and activations on a rounding boundary remain."""
import numpy as np
import pytest
import torch

from oracle import cnn_oracle as C
from test_gpu_cnn import P, R, _inputs, _stable_masks, relL2  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B", [1, 3, 37])
def test_forward_and_gradient_at_tile_edges(P, B):  # noqa: F811
    net = P.WeightPredictor(R, seed=6)
    _stable_masks(net, seed=40 + B)
    img, cs = _inputs(B, seed=9)
    out = net.forward(torch.as_tensor(img, device="cuda"), torch.as_tensor(cs, device="cuda"), tensor_cores=True)
    flat = net.params.cpu().numpy().astype(np.float64)
    assert relL2(out.cpu().numpy(), C.forward(flat, R, img, cs, bf16=True)) < 1e-3
    gw = np.random.default_rng(10).normal(size=(B, R)).astype(np.float32)
    g = net.backward(torch.as_tensor(gw, device="cuda"), tensor_cores=True).cpu().numpy()
    gref = C.vjp(flat, R, img, cs, gw, bf16=True)
    off = 0
    for name, shape in C.param_shapes(R):
        k = int(np.prod(shape))
        assert relL2(g[off:off + k], gref[off:off + k]) < 3e-3, name
        off += k


def test_images_need_only_element_alignment(P):  # noqa: F811
    net = P.WeightPredictor(R, seed=6)
    img, cs = _inputs(3, seed=12)
    I, Cs = torch.as_tensor(img, device="cuda"), torch.as_tensor(cs, device="cuda")
    flat = torch.empty(I.numel() + 1, device="cuda")
    shifted = flat[1:].view(I.shape)
    shifted.copy_(I)
    assert shifted.data_ptr() % 16 == 4
    assert torch.equal(net.forward(shifted, Cs, tensor_cores=True), net.forward(I, Cs, tensor_cores=True))
