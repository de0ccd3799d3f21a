"""The CNN at batches where the tensor-core convolutions' persistent thread blocks take several tiles (three or more each,
two in convolution 3's forward: accumulators, staging and activation buffers are used again) and where the FP32 mode's
last convolution takes its larger tiles, against the FP64 oracle.  Parameters and bounds as in the other comparisons."""
import numpy as np
import pytest
import torch

from oracle import cnn_oracle as C
from test_gpu_cnn import P, R, _inputs, _stable_masks, relL2  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B,tc,bounds", [(513, True, (1e-3, 3e-3)), (305, False, (1e-5, 1e-4))])
def test_forward_and_gradient_of_large_batches(P, B, tc, bounds):  # noqa: F811
    net = P.WeightPredictor(R, seed=6)
    _stable_masks(net, seed=40 + B)
    img, cs = _inputs(B, seed=9)
    out = net.forward(torch.as_tensor(img, device="cuda"), torch.as_tensor(cs, device="cuda"), tensor_cores=tc)
    flat = net.params.cpu().numpy().astype(np.float64)
    assert relL2(out.cpu().numpy(), C.forward(flat, R, img, cs, bf16=tc)) < bounds[0]
    gw = np.random.default_rng(10).normal(size=(B, R)).astype(np.float32)
    g = net.backward(torch.as_tensor(gw, device="cuda"), tensor_cores=tc).cpu().numpy()
    gref = C.vjp(flat, R, img, cs, gw, bf16=tc)
    off = 0
    for name, shape in C.param_shapes(R):
        k = int(np.prod(shape))
        assert relL2(g[off:off + k], gref[off:off + k]) < bounds[1], name
        off += k
