"""The fused ranking of one template with more distinct tables than it ranks by counting
(32): 33 tables, 130, and 400, which is several groups for the larger programs; each table
once, or up to four variants of each.  Tables differ in the constants of their flop counts, so
weights that leave those out tie nearly all of them.  Bit for bit against exact sums in Python
integers, ties by variant."""
import math
import re

import numpy as np
import pytest

from paper_1604_04997_gb300 import binding as B
from paper_1604_04997_gb300 import workloads as W
from test_rank_programs import _key

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def env():
    import torch
    import __graft_entry__
    __graft_entry__.build()
    ctx = B.Context(0)
    yield ctx, torch.device("cuda:0"), {}
    ctx.close()


def _distinct(ctx, cache, template, n):
    """n tables of one template with different images: its IR with other flop constants."""
    if template not in cache:
        vs = [v for v in W.all_variants() if v.template == template]
        P = len(W.TEMPLATE_PARAMS[template])
        ids, seen = [], set()
        for i in range(20000):
            add = i // len(vs)
            ir = re.sub(r"(flop \w+ \w+) (\d+)", lambda m: f"{m.group(1)} {int(m.group(2)) + add}", W.variant_ir(vs[i % len(vs)]))
            tid = ctx.compile_counts(ir, 32, [W.BOX_LO] * P, [W.BOX_HI] * P)[0]
            image = ctx.table_image(tid).tobytes()
            if image not in seen:
                seen.add(image)
                ids.append(tid)
            if len(ids) == 400:
                break
        cache[template] = ids
    return cache[template][:n]


@pytest.mark.parametrize("tie", [False, True], ids=["weights", "ties"])
@pytest.mark.parametrize("repeat", [False, True], ids=["once", "repeats"])
@pytest.mark.parametrize("template,n,points,topk", [("vecadd", 33, 41, 16), ("matmul", 33, 32, 16), ("stencil", 40, 33, 5),
                                                    ("vecadd", 130, 70, 16), ("matmul", 130, 31, 1), ("stencil", 130, 40, 16),
                                                    ("matmul", 400, 37, 16), ("vecadd", 400, 33, 16), ("matmul", 17, 33, 16)])
def test_distinct_tables_rank_exactly(env, template, n, points, topk, repeat, tie):
    import torch
    ctx, dev, cache = env
    rng = np.random.default_rng(n + points)
    ids = np.array(_distinct(ctx, cache, template, n), dtype=np.int32)
    tables = ids if not repeat else np.repeat(ids, rng.integers(1, 5, size=n))
    tables = np.ascontiguousarray(rng.permutation(tables))
    P = len(W.TEMPLATE_PARAMS[template])
    pts = np.zeros((points, 4), dtype=np.int64)
    pts[:, :P] = W.draw_points(P, points, n)
    dp = torch.from_numpy(pts).to(dev)
    F = torch.empty((n, points, 32), dtype=torch.int64, device=dev)
    ctx.eval_counts(ids, dp[:, :P].contiguous(), F)
    ctx.sync_status()
    F = F.cpu().numpy()
    w = W.draw_weights(32, 1, n)[0]
    if tie:
        w[(F != F[:1]).any(axis=(0, 1))] = 0.0       # the columns in which any two tables differ
        w[int(np.argmax(F.sum(axis=(0, 1))))] = 1e-9   # but one: some tables tie, some do not
    idx = torch.full((points, topk), -7, dtype=torch.int32, device=dev)
    tt = torch.zeros((points, topk), dtype=torch.float64, device=dev)
    ctx.eval_predict_topk(tables, np.array([0, len(tables)], dtype=np.int32), dp, np.array([0, points], dtype=np.int64),
                          torch.from_numpy(w).to(dev), topk, idx, tt)
    ctx.sync_status()
    idx, tt = idx.cpu().numpy(), tt.cpu().numpy()
    s = 0.0
    for x in w:
        s += abs(float(x))
    E = 62 - math.frexp(s * (1.0 + 2.0 ** -40))[1]
    Wi = np.array([int(x) for x in np.rint(np.ldexp(w, E))], dtype=object)
    S = {int(t): F[i].astype(object) @ Wi for i, t in enumerate(ids)}
    ties = 0
    for p in range(points):
        want = sorted((_key(int(S[int(t)][p])), v) for v, t in enumerate(tables))[:topk]
        assert idx[p].tolist() == [v for _, v in want], p
        keys = [k for k, _ in want]
        ties += len(keys) - len(set(keys))
        for q, k in enumerate(keys):
            m, e = abs(k) & ((1 << 56) - 1), (abs(k) >> 56) - 1
            ref = math.ldexp((1 << 56) + m, e - 56 - E) if k else 0.0
            assert tt[p, q] == (ref if k >= 0 else -ref), (p, q)
    assert ties > 0 or topk < 16 or not (tie or repeat)   # the test covers ties where it means to
