"""A tensor-core kernel of the weight predictor that gives up a wait (here: every wait, at once) leaves no finite number
where its result is missing: the weights of a forward, the gradients of a backward from that layer down and a training
step's loss and gradients are NaN.  The passes after it, with the default limit, are bitwise those from before.

At a batch of 3 the dense layer's products have no K loop to wait in, so that its gradients (and the last
convolution's bias, summed from one of them) are as usual; at 257 they give up too."""
import numpy as np
import pytest
import torch

from oracle import cnn_oracle as C
from test_gpu_cnn import P, R, _inputs  # noqa: F401

pytestmark = pytest.mark.gpu


def _groups(g):
    out, off = {}, 0
    for name, shape in C.param_shapes(R):
        k = int(np.prod(shape))
        out[name] = g[off:off + k]
        off += k
    return out


@pytest.mark.parametrize("B", [3, 257])
def test_give_up_makes_outputs_nan(P, B):  # noqa: F811
    from paper_2506_22280_gb300 import digs as D
    img, cs = _inputs(B, seed=3)
    I, Cs = torch.as_tensor(img, device="cuda"), torch.as_tensor(cs, device="cuda")
    G = torch.as_tensor(np.random.default_rng(4).normal(size=(B, R)).astype(np.float32), device="cuda")
    net = P.WeightPredictor(R, seed=6)
    out = net.forward(I, Cs, tensor_cores=True)
    grad = net.backward(G, tensor_cores=True)
    try:
        D.set_wait_limit(0)
        lost = net.backward(G, tensor_cores=True)  # of a forward that was whole
        lost_out = [net.forward(I, Cs, tensor_cores=True), net.predict(I, Cs)]
        probe = P.WeightPredictor(R, seed=6)
        loss = probe.train_step(I, Cs, G, 1e-3, tensor_cores=True)
        torch.cuda.synchronize()
    finally:
        D.set_wait_limit(-1)
    whole = ("w_fc2", "b_fc2", "b_fc1") + (("w_fc1", "b3") if B == 3 else ())
    for name, g in _groups(lost).items():
        if name in whole:
            assert torch.equal(g, _groups(grad)[name]), name
        else:
            assert bool(g.isnan().all()), name
    assert all(bool(o.isnan().all()) for o in lost_out)
    assert bool(loss.isnan().all()) and bool(probe.grad.isnan().all())
    assert torch.equal(net.forward(I, Cs, tensor_cores=True), out)
    assert torch.equal(net.backward(G, tensor_cores=True), grad)
