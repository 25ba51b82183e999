"""pm_predict_topk where its kernels meet: model counts around the row-per-lane kernel's
four and eight, feature counts with and without the staged copy, unaligned rows, row lists,
groups around the 128-row tile and the units, and ties (equal rows) by row.  Bit for bit
against the (time, row) order of pm_predict's own times, which test_gpu_exact_tc pins."""
import numpy as np
import pytest

from paper_1604_04997_gb300 import binding as B

pytestmark = pytest.mark.gpu

SIZES = [0, 1, 127, 128, 129, 16, 2047, 2049, 0, 5000]
LARGE = [4096, 12289, 8192]          # 512 rows a group and more: the tensor cores from five models


@pytest.fixture(scope="module")
def env():
    import torch
    import __graft_entry__
    __graft_entry__.build()
    ctx = B.Context(0, 64 << 20)
    yield ctx, torch.device("cuda:0")
    ctx.close()


@pytest.mark.parametrize("sizes", [SIZES, LARGE], ids=["ragged", "large"])
@pytest.mark.parametrize("listed", [False, True], ids=["rows", "list"])
@pytest.mark.parametrize("k,M,topk", [(32, 1, 16), (12, 3, 5), (24, 4, 1), (31, 4, 16), (32, 5, 16), (16, 8, 7), (17, 8, 16),
                                      (32, 8, 16), (13, 9, 16), (32, 33, 3), (28, 64, 16), (33, 8, 16), (40, 9, 2)])
def test_order_is_that_of_the_predicted_times(env, k, M, topk, listed, sizes):
    import torch
    ctx, dev = env
    rng = np.random.default_rng(1000 * k + 10 * M + listed)
    n, R = sum(sizes), 3000 if listed else sum(sizes)
    F = rng.integers(0, 1 << rng.integers(1, 41), size=(R, k))
    F[rng.integers(0, R, size=R // 2)] = F[rng.integers(0, R, size=R // 2)]       # equal rows
    Wm = rng.random((M, k)) * 10.0 ** rng.integers(-13, -8, size=(M, k))
    rows = rng.integers(0, R, size=n) if listed else np.arange(n)
    off = np.concatenate([[0], np.cumsum(sizes)]).astype(np.int64)
    base = torch.empty(R * k + 1, dtype=torch.int64, device=dev)
    dF = base[listed:listed + R * k].view(R, k)                                   # a list: 8-byte aligned only
    dF.copy_(torch.from_numpy(F))
    dW = torch.from_numpy(Wm).to(dev)
    idx = torch.full((len(sizes), M, topk), -5, dtype=torch.int64, device=dev)
    tt = torch.full((len(sizes), M, topk), np.nan, dtype=torch.float64, device=dev)
    ctx.predict_topk(dF, dW, off, topk, idx, tt, rows=torch.from_numpy(rows).to(dev) if listed else None)
    T = torch.empty((R, M), dtype=torch.float64, device=dev)
    ctx.predict(dF, dW, T)
    ctx.sync_status()
    idx, tt, T = idx.cpu().numpy(), tt.cpu().numpy(), T.cpu().numpy()
    for g in range(len(sizes)):
        mem = rows[off[g]:off[g + 1]]
        real = min(topk, len(mem))
        for m in range(M):
            order = np.lexsort((mem, T[mem, m]))[:real]
            assert np.array_equal(idx[g, m, :real], mem[order]), (g, m)
            assert np.array_equal(tt[g, m, :real], T[mem[order], m]), (g, m)
            assert (idx[g, m, real:] == -1).all() and np.isinf(tt[g, m, real:]).all()
