"""Operand preparation and list merge of the tensor-core kNN (``-m gpu``): a warp
per row, wide loads where the rows are aligned and single ones elsewhere.  The
graph is the oracle's bit for bit at widths around the eight- and four-feature
steps and the 256-column pass, for rows that start off alignment, and with many
column segments, with both list lengths.
"""
import numpy as np
import pytest
import torch

import oracle
from paper_2303_05455_gb300 import ivhd

pytestmark = pytest.mark.gpu


def rows(dtype, M, N, seed):
    X = np.random.default_rng(seed).integers(0, 256, size=(M, N))
    return X.astype(np.uint8) if dtype == "u8" else ((X - 90) / 64).astype(np.float32)


def exact(dtype, X, k):
    return oracle.knn_u8(X, k) if dtype == "u8" else oracle.knn_f32(X, k)


@pytest.mark.parametrize("off", [0, 1])
@pytest.mark.parametrize("N", [1, 3, 4, 7, 8, 21, 22, 64, 129, 256, 264, 1024])
@pytest.mark.parametrize("dtype", ["f32", "u8"])
def test_widths_and_alignment(dtype, N, off):
    X = rows(dtype, 301, N, N)
    room = torch.empty(301 * N + off, dtype=torch.float32 if dtype == "f32" else torch.uint8,
                       device="cuda")
    Xd = room[off:].view(301, N)
    Xd.copy_(torch.from_numpy(X))
    got = ivhd.knn_build(Xd, 5, method="tensor_cores")
    assert np.array_equal(got.cpu().numpy(), exact(dtype, X, 5))


@pytest.mark.parametrize("k", [1, 8, 9, 32])
@pytest.mark.parametrize("M", [300, 5000])
def test_merge_of_few_and_many_lists(M, k):
    X = rows("u8", M, 6, k)
    X[M // 2:M // 2 + 20] = X[:20]  # equal rows: ties go to the lower index
    got = ivhd.knn_build(torch.from_numpy(X).cuda(), k, method="tensor_cores")
    assert np.array_equal(got.cpu().numpy(), oracle.knn_u8(X, k))
