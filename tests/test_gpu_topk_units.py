"""pm_predict_topk with far more groups than SMs: every CTA takes several units, direct ones
(a group of one unit) and partial ones in turn, empty and one-row groups among them, with and
without a row list whose bad rows are skipped and reported; group lengths on both sides of the
line between the tensor cores and the integer tile.  Bit for bit against the (time, row) order
of pm_predict's own times, which test_gpu_exact_tc pins."""
import numpy as np
import pytest

from paper_1604_04997_gb300 import binding as B

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def env():
    import torch
    import __graft_entry__
    __graft_entry__.build()
    ctx = B.Context(0, 64 << 20)
    yield ctx, torch.device("cuda:0")
    ctx.close()


@pytest.mark.parametrize("longest,groups", [(400, 700), (60, 900)], ids=["long", "short"])
@pytest.mark.parametrize("listed", [False, True], ids=["rows", "list"])
@pytest.mark.parametrize("k,M,topk", [(12, 9, 16), (31, 64, 5), (32, 33, 16), (32, 64, 16), (12, 64, 1), (8, 9, 3), (32, 6, 4),
                                      (32, 7, 16), (32, 2, 16)])
def test_many_units_per_block(env, k, M, topk, listed, longest, groups):
    import torch
    ctx, dev = env
    rng = np.random.default_rng(100 * k + M)
    sizes = rng.integers(0, longest, size=groups)
    sizes[rng.integers(0, groups, size=40)] = 0
    sizes[rng.integers(0, groups, size=40)] = 1
    sizes[rng.integers(0, groups, size=3)] = 5000          # cut into several units
    n = int(sizes.sum())
    R = 20000 if listed else n
    F = rng.integers(0, 1 << rng.integers(1, 41), size=(R, k))
    F[rng.integers(0, R, size=R // 2)] = F[rng.integers(0, R, size=R // 2)]       # equal rows
    Wm = rng.random((M, k)) * 10.0 ** rng.integers(-13, -8, size=(M, k))
    rows = rng.integers(0, R, size=n) if listed else np.arange(n)
    if listed:
        bad = rng.random(n) < 0.01
        rows[bad] = rng.choice([-1, R, R + 7, -(1 << 40), 1 << 40], size=int(bad.sum()))
    off = np.concatenate([[0], np.cumsum(sizes)]).astype(np.int64)
    dF, dW = torch.from_numpy(F).to(dev), torch.from_numpy(Wm).to(dev)
    idx = torch.full((groups, M, topk), -5, dtype=torch.int64, device=dev)
    tt = torch.full((groups, M, topk), np.nan, dtype=torch.float64, device=dev)
    ctx.predict_topk(dF, dW, off, topk, idx, tt, rows=torch.from_numpy(rows).to(dev) if listed else None)
    if listed:
        with pytest.raises(B.PMError):
            ctx.sync_status()
    T = torch.empty((R, M), dtype=torch.float64, device=dev)
    ctx.predict(dF, dW, T)
    ctx.sync_status()
    idx, tt, T = idx.cpu().numpy(), tt.cpu().numpy(), T.cpu().numpy()
    models = sorted({0, 1, M // 2, M - 2, M - 1})
    for g in range(groups):
        mem = rows[off[g]:off[g + 1]]
        mem = mem[(mem >= 0) & (mem < R)]
        real = min(topk, len(mem))
        assert (idx[g, :, real:] == -1).all() and np.isinf(tt[g, :, real:]).all(), g
        for m in models:
            order = np.lexsort((mem, T[mem, m]))[:real]
            assert np.array_equal(idx[g, m, :real], mem[order]), (g, m)
            assert np.array_equal(tt[g, m, :real], T[mem[order], m]), (g, m)


@pytest.mark.parametrize("R", [130001, 131072, 140003])
@pytest.mark.parametrize("M", [5, 6, 7, 8])
def test_one_group_around_the_line_of_five_to_eight_models(env, M, R):
    import torch
    ctx, dev = env
    rng = np.random.default_rng(R + M)
    F = rng.integers(0, 1 << 30, size=(R, 32))
    F[rng.integers(0, R, size=R // 2)] = F[rng.integers(0, R, size=R // 2)]
    dF = torch.from_numpy(F).to(dev)
    dW = torch.from_numpy(rng.random((M, 32)) * 1e-9).to(dev)
    idx = torch.full((1, M, 16), -5, dtype=torch.int64, device=dev)
    tt = torch.full((1, M, 16), np.nan, dtype=torch.float64, device=dev)
    ctx.predict_topk(dF, dW, np.array([0, R], dtype=np.int64), 16, idx, tt)
    T = torch.empty((R, M), dtype=torch.float64, device=dev)
    ctx.predict(dF, dW, T)
    ctx.sync_status()
    idx, tt, T = idx.cpu().numpy(), tt.cpu().numpy(), T.cpu().numpy()
    for m in range(M):
        order = np.lexsort((np.arange(R), T[:, m]))[:16]
        assert np.array_equal(idx[0, m], order) and np.array_equal(tt[0, m], T[order, m]), m
