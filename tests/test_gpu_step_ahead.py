"""The step kernel that reads its ids ahead of the dependency wait (``-m gpu``).

Small graphs run it in the multi-launch form; the persistent grid runs the
plain traversal, so the two must agree bit for bit where the held id groups (four per lane) can go wrong:
rows with fewer and more groups than a lane holds (slices of up to 32 groups,
hub rows of 300 entries, rows of 512 entries and more on four warps), ragged
last slices, all block sizes, and a layout rebuilt between single steps.
"""
import numpy as np
import pytest

from paper_2303_05455_gb300 import ivhd, synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("M,k,hubs,frac", [(37, 3, 0, 0.0), (3001, 5, 20, 0.6), (9001, 4, 30, 0.4)])
@pytest.mark.parametrize("shape", [{}, {"hub_threshold": 128}, {"hub_threshold": 32, "block_size": 512},
                                   {"block_size": 256, "vertices_per_warp": 8}])
@pytest.mark.parametrize("opt", ["momentum", "nesterov", "adadelta"])
def test_ahead_equals_plain_traversal(M, k, hubs, frac, shape, opt):
    knn = synth.random_knn_graph(M, k, M + k, hub_frac=frac, n_hubs=hubs)
    got = []
    for resident in ("grid", False):
        e = ivhd.Embedding(knn, r=1, c=0.05, opt=opt, b=5e-4, seed=3, resident=resident, **shape)
        e.step(1)
        e.step(66)
        e.resample_random_neighbors(7)
        e.step(1)
        e.step(2)
        got.append((e.positions(host=True), e.get_state(), e.info()["max_degree"]))
        e.close()
    assert hubs == 0 or got[0][2] > 300
    assert np.isfinite(got[0][0]).all()
    assert np.array_equal(got[0][0], got[1][0]) and got[0][1] == got[1][1]
