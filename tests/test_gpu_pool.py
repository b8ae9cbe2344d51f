"""The library's own memory pool (``-m gpu``): bounded, given back, any thread and stream."""
import threading

import numpy as np
import pytest
import torch

from paper_2303_05455_gb300 import ivhd, synth

pytestmark = pytest.mark.gpu


def test_keeps_little_and_gives_it_back():
    X = torch.randn((200_000, 64), device="cuda")   # some hundred MB of scratch
    ivhd.knn_build(X, 5)
    torch.cuda.synchronize()
    ivhd.set_allocator()                             # nothing of the library's is in use
    free0 = torch.cuda.mem_get_info()[0]
    ivhd.knn_build(X, 5)
    torch.cuda.synchronize()
    held = free0 - torch.cuda.mem_get_info()[0]
    # the bound, and a granule of the driver at its edge
    assert 0 <= held <= (256 + 64) << 20
    ivhd.set_allocator()
    assert free0 - torch.cuda.mem_get_info()[0] <= 4 << 20


def test_threads_and_streams_get_their_own_memory():
    knn = synth.random_knn_graph(3000, 4, 5)
    want = {}
    for seed in range(6):
        with ivhd.Embedding(knn, r=1, c=0.05, seed=seed) as e:
            e.step(30)
            want[seed] = e.positions(host=True)
    got = {}

    def work(seed):
        s = torch.cuda.Stream()
        with torch.cuda.stream(s):
            for _ in range(10):
                with ivhd.Embedding(knn, r=1, c=0.05, seed=seed, stream=s) as e:
                    e.step(30)
                    got.setdefault(seed, []).append(e.positions(host=True))

    threads = [threading.Thread(target=work, args=(s,)) for s in range(6)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    for seed in range(6):
        assert len(got[seed]) == 10
        assert all(np.array_equal(y, want[seed]) for y in got[seed])
