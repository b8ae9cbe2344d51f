"""The spatial index behind Q_NX and cf_nn vs the oracle's full scan (``-m gpu``).

Neighbour lists, and with them both criteria, must equal the oracle's exactly:
at the edges of leaves (32 points) and nodes (1,024 points), for list lengths
at the edges of the kernel's registers (32, 64, 128), and for positions that
stress the pruning: many exact ties, points that all coincide, tight clusters,
extents whose squared distances overflow to infinity, and positions that are
not finite (which the full scan answers).
"""
import numpy as np
import pytest
import torch

import oracle
from paper_2303_05455_gb300 import ivhd, synth

pytestmark = pytest.mark.gpu


def positions(kind, M):
    rng = np.random.default_rng(M)
    Y = rng.random((M, 2)).astype(np.float32)
    if kind == "ties":
        return np.round(Y * 9).astype(np.float32)
    if kind == "same":
        return np.full_like(Y, 0.25)
    if kind == "clumps":
        return (rng.integers(0, 4, (M, 2)) + 1e-5 * rng.standard_normal((M, 2))).astype(np.float32)
    if kind == "line":
        Y[:, 1] = -3.0
        return Y
    if kind == "wide":
        return (np.sign(Y - 0.5) * np.float32(10.0) ** (60 * Y - 30)).astype(np.float32)
    if kind == "infinite":
        Y[::97] = np.inf
        Y[1::97, 0] = -np.inf
    return Y


@pytest.mark.parametrize("kind", ["even", "ties", "same", "clumps", "line", "wide", "infinite"])
@pytest.mark.parametrize("M,kk", [(2, 1), (33, 32), (1023, 5), (1024, 33), (1025, 64), (2500, 65),
                                  (2500, 128), (5000, 10)])
def test_lists_equal_the_full_scan(kind, M, kk):
    Y = positions(kind, M)
    rows = synth.sample_rows(M, 300, 3)
    if kind == "infinite":
        rows = rows[np.isfinite(Y[rows]).all(1)]
        kk = min(kk, int(np.isfinite(Y).all(1).sum()) - 1)
        if rows.size == 0 or kk < 1:
            pytest.skip("no finite positions")
    knn = synth.random_knn_graph(M, kk, M + kk) if kk < M // 4 else \
        np.stack([np.delete(np.arange(M), i)[:kk] for i in range(M)]).astype(np.int32)
    Yd, kd, rd = (torch.from_numpy(a).cuda() for a in (Y, knn, rows))
    q, low = ivhd.eval_qnx(Yd, kd, rd, return_lowd=True)
    q_ref, low_ref = oracle.qnx(Y, knn, rows, return_lowd=True)
    assert np.array_equal(low.cpu().numpy(), low_ref)
    assert q == q_ref
    lab = (np.arange(M) % 7).astype(np.int32)
    assert ivhd.eval_cf(Yd, lab, kk, rd) == oracle.cf(Y, lab, kk, rows)
