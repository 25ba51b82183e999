"""Served rankings bit for bit against pm_predict_topk over the materialised counts of the
same candidates: candidate counts around the ranking kernel's batches (32 keys a warp, 1,024
a pass, 4,096 in flight), many equal keys (repeated candidates) in index order."""
import numpy as np
import pytest

from paper_1604_04997_gb300 import binding as B
from paper_1604_04997_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("topk", [1, 5, 16])
def test_served_order_is_that_of_the_materialised_counts(topk):
    import torch
    import __graft_entry__
    __graft_entry__.build()
    dev = torch.device("cuda:0")
    ctx = B.Context(0, 64 << 20)
    vs = [v for v in W.all_variants() if v.template == "matmul"][::211]
    P = len(W.TEMPLATE_PARAMS["matmul"])
    ids = np.array([ctx.compile_counts(W.variant_ir(v), 32, [1] * P, [4096] * P)[0] for v in vs], dtype=np.int32)
    Wm = W.draw_weights(32, 3, 77)
    Wm[2, ::3] *= -1.0                                    # negative times too
    ctx.serve_set_weights(Wm)
    ctx.serve_start()
    rng = np.random.default_rng(topk)
    for n in (1, 15, 31, 33, 1023, 1025, 4095, 4097, 20000):
        distinct = rng.integers(1, 4097, size=(max(1, n // 4), P))
        pts = np.ascontiguousarray(distinct[rng.integers(0, len(distinct), size=n)])
        pts4 = np.ascontiguousarray(np.pad(pts, ((0, 0), (0, 4 - P))))
        tab = np.ascontiguousarray(ids[rng.integers(0, len(ids), size=n)])
        F = torch.empty((len(ids), n, 32), dtype=torch.int64, device=dev)
        ctx.eval_counts(ids.tolist(), torch.from_numpy(pts).to(dev), F)
        pick = torch.from_numpy(np.searchsorted(ids, tab)).to(dev)
        F = F[pick, torch.arange(n, device=dev)].contiguous()
        ref_i = torch.empty((1, 3, topk), dtype=torch.int64, device=dev)
        ref_t = torch.empty((1, 3, topk), dtype=torch.float64, device=dev)
        ctx.predict_topk(F, torch.from_numpy(Wm).to(dev), [0, n], topk, ref_i, ref_t)
        ctx.sync_status()
        for m in range(3):
            idx, t = np.empty(topk, dtype=np.int32), np.empty(topk)
            ticket = ctx.serve_submit(B.make_query(m, topk, tab, pts4, idx, t))
            while ctx.serve_poll(ticket, 1_000_000) == B.PM_PENDING:
                pass
            assert np.array_equal(idx, ref_i[0, m].cpu().numpy()), (n, m)
            assert np.array_equal(t, ref_t[0, m].cpu().numpy()), (n, m)
    ctx.close()
