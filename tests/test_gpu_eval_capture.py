"""pm_eval_counts of a table list that was seen allocates nothing more, whatever the number
of points: it runs under stream capture for every split of the list into work items (the
launch takes one to eight positions of a repeated table per item)."""
import numpy as np
import pytest

from paper_1604_04997_gb300 import binding as B
from paper_1604_04997_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("repeats", [1, 3, 11])
def test_a_seen_list_can_be_captured_for_any_point_count(repeats):
    import torch
    import __graft_entry__
    __graft_entry__.build()
    ctx, dev = B.Context(0), torch.device("cuda:0")
    vs = [v for v in W.all_variants() if v.template == "matmul"][::41][:9]
    P = len(W.TEMPLATE_PARAMS["matmul"])
    ids = [ctx.compile_counts(W.variant_ir(v), 12, [1] * P, [4096] * P)[0] for v in vs] * repeats
    ids = np.random.default_rng(1).permutation(ids + ids[:4] * 3).astype(np.int32)   # some more often than others
    n_tables = len(ids)
    pts = torch.from_numpy(W.draw_points(P, 40000, 3, 1, 4096)).to(dev)
    ref = torch.empty((n_tables, 40000, 12), dtype=torch.int64, device=dev)
    one = torch.empty((n_tables, 1, 12), dtype=torch.int64, device=dev)
    ctx.eval_counts(ids, pts[:1], one)                 # the list is seen
    ctx.sync_status()
    for n in (100, 5000, 12000, 21000, 40000):         # one to eight positions per item
        out = torch.zeros((n_tables, n, 12), dtype=torch.int64, device=dev)
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g):
            ctx.eval_counts(ids, pts[:n], out, stream=torch.cuda.current_stream())
        g.replay()
        torch.cuda.synchronize()
        ctx.eval_counts(ids, pts[:n], ref.view(-1)[:n_tables * n * 12].view(n_tables, n, 12))
        ctx.sync_status()
        assert torch.equal(out, ref.view(-1)[:n_tables * n * 12].view(n_tables, n, 12)), n
        for i in set(ids.tolist()):                    # every position has its table's rows
            at = torch.from_numpy(np.flatnonzero(ids == i)).to(dev)
            assert bool((out[at] == out[at[0]]).all())
            assert torch.equal(out[at[0], :1], one[at[0]])
    ctx.close()


def test_lists_of_equal_images_share_one_plan():
    """Tables compiled again and again (new ids, equal images) leave one work list behind."""
    import ctypes
    import torch
    import __graft_entry__
    __graft_entry__.build()
    ctx, dev = B.Context(0), torch.device("cuda:0")
    f = B.lib().pmx_eval_plans
    f.restype, f.argtypes = ctypes.c_int, [ctypes.c_void_p]
    vs = [v for v in W.all_variants() if v.template == "vecadd"][:3]
    P = len(W.TEMPLATE_PARAMS["vecadd"])
    pts = torch.from_numpy(W.draw_points(P, 40, 3)).to(dev)
    out = torch.empty((3, 40, 32), dtype=torch.int64, device=dev)
    first = None
    for _ in range(20):
        ids = [ctx.compile_counts(W.variant_ir(v), 32, [W.BOX_LO] * P, [W.BOX_HI] * P)[0] for v in vs]
        ctx.eval_counts(ids, pts, out)
        ctx.sync_status()
        first = out.clone() if first is None else first
        assert torch.equal(out, first)
    assert f(ctx.h) == 1
    with pytest.raises(B.PMError):
        ctx.eval_counts([ids[0], 10 ** 6], pts, out)
    with pytest.raises(B.PMError):
        ctx.eval_counts([-1], pts, out)
    ctx.close()
