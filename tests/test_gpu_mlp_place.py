"""The one-kernel forward pass of the warm-start network (``-m gpu``).

Compared with the layer-by-layer path, which the C entry point takes for an
output that is not 8-byte aligned, at the edges of its tiles (256 rows, 128 per
CTA; hidden chunks of 256 columns; 64-column slabs and their remainders) and
over several chunks.  Both round the activations to BF16 at the same places, so
they differ by FP32 summation orders and the BF16 roundings these tip over:
2.4e-4 of the outputs' norm against sums in 64 bits over random networks; the
bar is four times that.  The intermediates of the last chunk must be those of
the layer-by-layer path, also when the weights have changed since.
"""
import ctypes

import numpy as np
import pytest
import torch

from paper_2303_05455_gb300 import ivhd

pytestmark = pytest.mark.gpu


def network(n_in, hidden, max_batch, seed):
    net = ivhd.MLP(n_in, hidden, max_batch=max_batch)
    rng = np.random.default_rng(seed)
    net.set_params((rng.standard_normal(net.n_params) / np.sqrt(max(n_in, hidden))).astype(np.float32))
    return net


def layer_by_layer(net, x):
    buf = torch.empty(2 * x.shape[0] + 1, device="cuda")
    y = buf[1:]
    code = {torch.bfloat16: 0, torch.uint8: 1, torch.float32: 2}[x.dtype]
    assert y.data_ptr() % 8 == 4
    assert net._L.ivhd_mlp_forward(net._h, x.data_ptr(), code, ctypes.c_float(1.0), x.shape[0],
                                   y.data_ptr()) == 0
    return y.reshape(-1, 2).clone()


@pytest.mark.parametrize("n_in,hidden,max_batch", [(8, 16, 64), (72, 48, 4096), (64, 256, 512),
                                                   (200, 272, 1024), (784, 512, 1000), (40, 320, 8),
                                                   (784, 496, 4096)])
@pytest.mark.parametrize("rows", [1, 127, 129, 256, 257, 2600])
def test_equals_layer_by_layer(n_in, hidden, max_batch, rows):
    net = network(n_in, hidden, max_batch, rows)
    x = torch.randn((rows, n_in), device="cuda")
    ref = layer_by_layer(net, x)
    last = [net.activations(a) for a in ("x", "h1", "h2", "y")]
    got = net.forward(x)
    err = float((got - ref).norm() / ref.norm())
    assert err < 1e-3, err
    assert torch.equal(got, net.forward(x))
    net.set_params(net.get_params() * 0 + 1)  # the last chunk's activations are the old weights'
    for a, b in zip([net.activations(a) for a in ("x", "h1", "h2")], last):
        assert np.array_equal(a, b)
    assert np.array_equal(net.activations("y").shape, last[3].shape)


@pytest.mark.parametrize("dtype", [torch.uint8, torch.bfloat16])
def test_rows_do_not_depend_on_their_place(dtype):
    net = network(104, 512, 512, 5)
    x = (torch.randint(0, 256, (1500, 104), device="cuda") if dtype == torch.uint8
         else torch.randn((1500, 104), device="cuda")).to(dtype)
    y = net.forward(x, x_scale=0.25)
    for lo, hi in ((0, 1), (130, 131), (400, 1111), (1499, 1500)):
        assert torch.equal(y[lo:hi], net.forward(x[lo:hi].contiguous(), x_scale=0.25))
