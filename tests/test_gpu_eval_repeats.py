"""pm_eval_counts of table lists that name equal tables many times (by one id, and by several
ids of equal images): every position has its table's rows, for point counts around the
128-point block and outputs that are 16-byte aligned and not."""
import numpy as np
import pytest

import oracle
from paper_1604_04997_gb300 import binding as B
from paper_1604_04997_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("layout", [32, 12])
@pytest.mark.parametrize("n_points,n_tables", [(1, 5), (127, 40), (128, 9), (129, 700), (1500, 301), (20000, 33)])
def test_repeated_tables(layout, n_points, n_tables):
    import torch
    import __graft_entry__
    __graft_entry__.build()
    ctx, dev = B.Context(0), torch.device("cuda:0")
    vs = [v for v in W.all_variants() if v.template == "matmul"][::29][:12]
    irs = [W.variant_ir(v) for v in vs]
    irs += irs[:5]                                       # equal images under other ids
    P = len(W.TEMPLATE_PARAMS["matmul"])
    ids = [ctx.compile_counts(ir, layout, [1] * P, [4096] * P)[0] for ir in irs]
    assert len(set(ids)) == len(ids)
    rng = np.random.default_rng(n_points)
    pts = rng.integers(1, 4097, size=(n_points, P))
    pick = rng.integers(0, len(ids), size=n_tables)
    pick[: n_tables // 2] = pick[0]                      # one table in far more than one block's positions
    base = torch.full((n_tables * n_points * layout + 3,), -7, dtype=torch.int64, device=dev)
    ref = np.stack([oracle.Kernel(ir).features(pts[:200], layout, "struct") for ir in irs[:12]])
    for shift in (0, 1):
        out = base[shift:shift + n_tables * n_points * layout].view(n_tables, n_points, layout)
        ctx.eval_counts([ids[i] for i in pick], torch.from_numpy(pts).to(dev), out)
        ctx.sync_status()
        got = out[:, :200].cpu().numpy()
        for t, i in enumerate(pick):
            assert np.array_equal(got[t], ref[i % 12]), t
        # every later row too: equal to that of the first position of the same table
        for i in set(pick.tolist()):
            at = torch.from_numpy(np.flatnonzero(pick % 12 == i % 12)).to(dev)
            assert bool((out[at] == out[at[0]]).all())
        assert int(base[shift + n_tables * n_points * layout]) == -7
    ctx.close()
