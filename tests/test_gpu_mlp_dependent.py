"""The training step's dependent launches (``-m gpu``): each kernel is set up while
the one before it runs and must not read before that one is complete.  Steps on
changing batches give the same weights bit for bit whether they follow each other at
once or each is waited for, or the same products run outside the graph in
between; widths and batches reach all tile widths of the GEMM (64, 128, 256).
"""
import numpy as np
import pytest
import torch

from paper_2303_05455_gb300 import ivhd

pytestmark = pytest.mark.gpu


def run(n_in, H, B, x, t, wait, between=False):
    net = ivhd.MLP(n_in, H, max_batch=B)
    net.init_params(3)
    for i in range(x.shape[0]):
        if between:  # the same products outside the graph, on the same weights
            net.loss_grad(x[i], t[i])
        net.train_step(x[i], t[i], lr=1e-3)
        if wait:
            torch.cuda.synchronize()
    return net.get_params()


@pytest.mark.parametrize("n_in,H,B", [(8, 16, 8), (40, 64, 136), (784, 512, 4096), (256, 512, 12288),
                                      (64, 1024, 40960)])
def test_steps_in_a_row_equal_steps_waited_for(n_in, H, B):
    g = torch.Generator("cuda").manual_seed(B)
    x = torch.rand(6, B, n_in, device="cuda", generator=g)
    t = torch.rand(6, B, 2, device="cuda", generator=g)
    torch.cuda.synchronize()
    a = run(n_in, H, B, x, t, wait=True)
    assert np.isfinite(a).all()
    assert np.array_equal(a, run(n_in, H, B, x, t, wait=False))
    assert np.array_equal(a, run(n_in, H, B, x, t, wait=False, between=True))
