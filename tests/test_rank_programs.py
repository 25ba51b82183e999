"""Ranking by program: variants that share a table share one evaluation, and the best
programs are expanded to the best variants.  The program table of a plan on the CPU, and
the fused ranking on the GPU against exact sums in Python integers: keys of 40 mantissa
bits, ties (equal tables, and different tables that are equal at a point) by variant."""
import numpy as np
import pytest

from paper_1604_04997_gb300 import binding as B
from paper_1604_04997_gb300 import tuning
from paper_1604_04997_gb300 import workloads as W
from test_rank_group import _u16, rank_plan


@pytest.mark.parametrize("slice_", [0, 64])
def test_program_table_lists_every_program_and_its_first_variants(slice_):
    import __graft_entry__
    __graft_entry__.build_library()
    ctx = B.Context(-1)
    b = tuning.build(ctx, n_variants=900, n_points=33, variant_seed=5, point_seed=6)
    images = {int(t): ctx.table_image(int(t)).tobytes() for t in set(b.tables.tolist())}
    pl = rank_plan(ctx, b, slice_)
    for g0, g1 in pl["groups"]:
        img = pl["img"][g0[0]:g0[0] + g0[1]]
        first = int(b.var_off[g1[0]] + g0[2])
        by_image, order = {}, []
        for v in range(int(g0[3])):
            im = images[int(b.tables[first + v])]
            if im not in by_image:
                by_image[im] = []
                order.append(im)
            by_image[im].append(v)
        n_progs, o_progs, o_span, o_pvid, staged = img[18:23]
        assert n_progs == len(order) and staged == g1[2] and staged % 4 == 0
        pos = 0
        for q in range(n_progs):
            root, pid = img[o_progs + q] & 0xFFFF, img[o_progs + q] >> 16
            vids = by_image[order[pid]]        # ids in the order of first variants
            off, n = img[o_span + pid] & 0xFFFF, img[o_span + pid] >> 16
            assert [_u16(img, o_pvid, off + i) for i in range(n)] == vids[:16]
            for v in vids:                     # the walk holds its variants side by side
                assert _u16(img, img[14], pos) == root and _u16(img, img[15], pos) == v
                pos += 1
        runs = [img[img[16] + 4 * r:img[16] + 4 * r + 4] for r in range(img[17])]
        assert [r[3] for r in runs] == sorted(r[3] for r in runs) and runs[0][3] == 0
    ctx.close()


def _key(S):
    """acc_key of an exact sum, cut to the entry's 48 bits."""
    if S == 0:
        return 0
    a, n = abs(S), abs(S).bit_length()
    m = (a >> (n - 57) if n > 57 else a << (57 - n)) & ((1 << 56) - 1)
    k = (n << 56) | m
    return (k if S > 0 else -k) >> 16 << 16


@pytest.mark.gpu
@pytest.mark.parametrize("seed,topk", [(1, 16), (2, 5), (3, 1), (4, 16)])
def test_fused_ranking_orders_variants_exactly(seed, topk):
    import math
    import torch
    import __graft_entry__
    __graft_entry__.build()
    ctx, dev = B.Context(0), torch.device("cuda:0")
    rng = np.random.default_rng(seed)
    b = tuning.build(ctx, n_variants=[700, 300, 40, 1200][seed - 1], n_points=41, variant_seed=60 + seed, point_seed=70 + seed)
    w = W.draw_weights(32, 1, seed)[0]
    if seed == 2:
        w = w * rng.choice([-1.0, 1.0], size=32)
    s = 0.0
    for x in w:
        s += abs(float(x))
    E = 62 - math.frexp(s * (1.0 + 2.0 ** -40))[1]
    Wi = np.array([int(x) for x in np.rint(np.ldexp(w, E))], dtype=object)
    pts = torch.from_numpy(b.points).to(dev)
    n = len(b.points)
    idx = torch.empty((n, topk), dtype=torch.int32, device=dev)
    tt = torch.empty((n, topk), dtype=torch.float64, device=dev)
    ctx.eval_predict_topk(b.tables, b.var_off, pts, b.pt_off, torch.from_numpy(w).to(dev), topk, idx, tt)
    ctx.sync_status()
    idx, tt = idx.cpu().numpy(), tt.cpu().numpy()
    ties = 0
    for t, name in enumerate(b.templates):
        ids = b.tables[b.var_off[t]:b.var_off[t + 1]].tolist()
        p0, p1, P = int(b.pt_off[t]), int(b.pt_off[t + 1]), len(W.TEMPLATE_PARAMS[name])
        if not ids:
            assert (idx[p0:p1] == -1).all()
            continue
        distinct = sorted(set(ids))
        F = torch.empty((len(distinct), p1 - p0, 32), dtype=torch.int64, device=dev)
        ctx.eval_counts(distinct, pts[p0:p1, :P].contiguous(), F)
        ctx.sync_status()
        S = {tid: F[i].cpu().numpy().astype(object) @ Wi for i, tid in enumerate(distinct)}
        for p in range(p0, p1):
            want = sorted((_key(int(S[tid][p - p0])), v) for v, tid in enumerate(ids))[:topk]
            got = [(int(i)) for i in idx[p] if i >= 0]
            assert got == [v for _, v in want], (name, p)
            keys = [k for k, _ in want]
            ties += len(keys) - len(set(keys))
            for q, k in enumerate(keys):
                m, e = abs(k) & ((1 << 56) - 1), (abs(k) >> 56) - 1
                ref = math.ldexp((1 << 56) + m, e - 56 - E) if k else 0.0
                assert tt[p, q] == (ref if k >= 0 else -ref), (name, p, q)
    assert ties > 0 or topk == 1
    ctx.close()
