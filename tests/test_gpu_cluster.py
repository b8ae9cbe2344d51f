"""The cluster form with rows held in registers vs one launch per step (``-m gpu``).

Positions and optimiser state must agree bit for bit at sizes where the split
of items over the eight blocks can go wrong: fewer items than blocks, one item
more than a multiple of eight, ragged last slices, hub rows sharing a warp,
rows of 256 entries and more (a whole warp each, four int4 groups per lane),
odd and even step counts (both ping-pong buffers), and a layout shape that the
register form does not take (hub threshold above 16).
"""
import numpy as np
import pytest

from paper_2303_05455_gb300 import ivhd, synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("M,k,hubs,shape", [(2, 1, 0, {}), (31, 2, 0, {}), (33, 2, 0, {}),
                                            (225, 3, 0, {}), (257, 1, 0, {}), (1001, 5, 8, {}),
                                            (3003, 3, 30, {}), (3003, 3, 30, {"hub_threshold": 64}),
                                            (3003, 3, 30, {"vertices_per_warp": 8})])
@pytest.mark.parametrize("opt,metric", [("momentum", "l2"), ("nesterov", "l2"), ("adadelta", "l2"),
                                        ("momentum", "l1")])
def test_cluster_form_equals_one_launch_per_step(M, k, hubs, shape, opt, metric):
    knn = synth.random_knn_graph(M, k, M + k, hub_frac=0.4 if hubs else 0.0, n_hubs=hubs)
    got = []
    for resident in ("cluster", False):
        e = ivhd.Embedding(knn, r=1, c=0.05, opt=opt, b=0.002, seed=3, resident=resident, **shape)
        e.set_metric(metric)
        for n in (1, 2, 5):
            e.step(n)
        got.append((e.positions(host=True), e.get_state(), e.info()["kernel_launches"]))
        e.close()
    assert got[0][2] == 3 and got[1][2] == 8
    assert np.isfinite(got[0][0]).all()
    assert np.array_equal(got[0][0], got[1][0]) and got[0][1] == got[1][1]
