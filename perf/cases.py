"""The work a user of this framework has it do, as cases for timing and comparison.

A case names one public entry point, its sizes and its options:

  counts   Context.eval_counts: exact counts of compiled kernels, [tables][points][layout]
  predict  Context.predict: predicted times of materialised feature rows, [rows][models]
  argmin   Context.predict_argmin: the fastest row per model
  topk     Context.predict_topk: the fastest rows per (group, model)
  points   eval_counts' rows ranked per point through a row list (Context.predict_topk)
  rank     Context.eval_predict_topk: count, predict and rank a tuning space in one call
  fit      Context.fit_weights: weights of device models from measured times
  serve    Context.serve_submit / serve_poll: a burst of autotuner queries

One context per process holds the compiled kernels, as a tuner's process does; a case's
seed draws the parameter points, features, weights and timings.
"""
import math

import numpy as np
import torch

from paper_1604_04997_gb300 import binding as B
from paper_1604_04997_gb300 import tuning
from paper_1604_04997_gb300 import workloads as W

DEV = "cuda"
PREC = {"fp64": B.PREC_FP64, "bf16x3": B.PREC_BF16X3}
MAX_ROWS = 1_000_000          # feature rows of the largest prediction problems
MAX_COUNT_ROWS = 2_720_000    # (table, point) pairs of the largest counts case
MAX_POINT_ROWS = 4_500_000    # ranked rows of the largest per-point ranking
FIT_COLS_12 = (0, 1, 2, 3, 4, 5, 6, 7, 13, 15, 17, 24)   # twelve columns the feature families use


def listed():
    return [
        # one kernel at the small workload's 32 points: a tuner asking about one launch
        dict(name="counts_one_kernel", kind="counts", template="matmul", tables=1, points=32, layout=32),
        # every matmul variant of the 10,000-variant tuning space, counts kept for later use
        dict(name="counts_space", kind="counts", template="matmul", tables=2656, points=1024, layout=32),
        # a calibration set in the aggregated layout, three devices, ragged sizes
        dict(name="predict_small_k12", kind="predict", prec="fp64", rows=4097, k=12, models=3),
        # cross-model prediction, a million rows for 64 devices, FP64-accurate
        dict(name="predict_fp64", kind="predict", prec="fp64", rows=MAX_ROWS, k=32, models=64),
        # the same problem where 1e-6 is enough
        dict(name="predict_bf16x3", kind="predict", prec="bf16x3", rows=MAX_ROWS, k=32, models=64),
        # the fastest configuration per device, reduced precision
        dict(name="argmin_bf16x3", kind="argmin", prec="bf16x3", rows=MAX_ROWS, k=32, models=64),
        # the sixteen fastest of a million configurations for each of 64 devices
        dict(name="topk_64_models", kind="topk", rows=MAX_ROWS, k=32, models=64, groups=1, topk=16),
        # one device: the sixteen fastest variants for each problem size, counts already in memory
        dict(name="points_one_model", kind="points", template="reduction", tables=1094, points=4096, models=1, topk=16),
        # the batched tuning space: 10,000 variants x 4,096 points of 8 templates, fused
        dict(name="rank_space", kind="rank", coupled=False, variants=10000, points=4096, topk=16),
        # triangles, bands and pair loops (counts with a denominator), odd point count
        dict(name="rank_coupled", kind="rank", coupled=True, variants=3000, points=1001, topk=5),
        # weights of 64 devices from 200,000 measurements each
        dict(name="fit_64_models", kind="fit", prec="bf16x3", objective="relative", rows=200_000, k=32, models=64),
        # a burst of 64 queries of up to 50,000 candidates
        dict(name="serve_burst", kind="serve", queries=64, max_cand=50_000, topk=16),
    ]


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(math.exp(rng.uniform(math.log(lo), math.log(hi + 1))))))


def draw(rng):
    kind = rng.choice(["counts", "predict", "predict", "argmin", "topk", "points", "rank", "rank", "fit", "fit", "serve"])
    if kind == "counts":
        tables = _log_int(rng, 1, 500)
        return dict(kind=kind, template=rng.choice(W.TEMPLATES), tables=tables,
                    points=_log_int(rng, 32, MAX_COUNT_ROWS // tables // 4), layout=rng.choice([12, 32]))
    if kind in ("predict", "argmin"):
        prec = rng.choice(["fp64", "fp64", "bf16x3"])
        return dict(kind=kind, prec=prec, rows=_log_int(rng, 64, MAX_ROWS), k=32 if prec == "bf16x3" else rng.choice([12, 32]),
                    models=rng.choice([1, 4, 17, 64, rng.randint(1, 64)]))
    if kind == "topk":
        rows = _log_int(rng, 256, MAX_ROWS)
        return dict(kind=kind, rows=rows, k=rng.choice([12, 32]), models=rng.choice([1, 3, 8, 16, rng.randint(1, 64)]),
                    groups=_log_int(rng, 1, max(1, rows // 64)), topk=rng.choice([1, 5, 16]))
    if kind == "points":
        tables = _log_int(rng, 32, 1000)
        return dict(kind=kind, template=rng.choice(W.TEMPLATES), tables=tables,
                    points=_log_int(rng, 32, MAX_POINT_ROWS // tables // 2), models=rng.choice([1, 1, 2, 5]), topk=rng.choice([1, 5, 16]))
    if kind == "rank":
        return dict(kind=kind, coupled=rng.random() < 0.3, variants=_log_int(rng, 64, 10000), points=_log_int(rng, 32, 4096),
                    topk=rng.choice([1, 5, 16]))
    if kind == "fit":
        prec = rng.choice(["bf16x3", "bf16x3", "fp64"])
        models = rng.choice([1, 5, 16, rng.randint(1, 64 if prec == "bf16x3" else 16)])
        return dict(kind=kind, prec=prec, objective=rng.choice(["relative", "relative", "absolute"]),
                    rows=_log_int(rng, 1000, 200_000 if prec == "bf16x3" else 60_000), k=rng.choice([12, 32]), models=models)
    return dict(kind=kind, queries=_log_int(rng, 1, 64), max_cand=_log_int(rng, 100, 50_000), topk=rng.choice([1, 16]))


# ---------------------------------------------------------------- what a user's process keeps

_ctx = None
_ids = {}      # (template variant key, layout) -> table id in _ctx
_spaces = {}   # tuning spaces compiled so far


def _context():
    global _ctx
    if _ctx is None:
        _ctx = B.Context(0)
    return _ctx


def _compile(variants, layout):
    return tuning.compile_variants(_context(), variants, W.BOX_LO, W.BOX_HI, layout, _ids.setdefault(layout, {}))


def _template_tables(template, n, layout):
    """The first n variants of one template, in the order of the batched tuning space."""
    pool = [v for v in W.draw_variants(10000, 2) if v.template == template]
    return _compile([pool[i % len(pool)] for i in range(n)], layout)


def _space(n_variants, coupled):
    """(tables, var_off, templates) of a tuning space of n_variants drawn variants."""
    key = (n_variants, coupled)
    if key not in _spaces:
        templates = ("trmv", "band", "pairs") if coupled else W.TEMPLATES
        drawn = W.draw_coupled_variants(n_variants, 12) if coupled else W.draw_variants(n_variants, 2)
        variants, var_off = [], [0]
        for t in templates:
            variants += [v for v in drawn if v.template == t]
            var_off.append(len(variants))
        _spaces[key] = (np.array(_compile(variants, 32), dtype=np.int32), np.array(var_off, dtype=np.int32), templates)
    return _spaces[key]


def _template_points(templates, n, seed):
    """Log-uniform points per template, padded to four parameters, and their offsets."""
    rows = []
    for i, t in enumerate(templates):
        p = np.zeros((n, 4), dtype=np.int64)
        P = len(W.TEMPLATE_PARAMS[t])
        p[:, :P] = W.draw_points(P, n, 1000 * seed + i)
        rows.append(p)
    return np.concatenate(rows), np.arange(0, n * len(templates) + 1, n, dtype=np.int64)


# ---------------------------------------------------------------- inputs

def _gen(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(seed)
    return g


def _weights(k, models, seed):
    """Per-device weights, seconds per operation."""
    return torch.from_numpy(W.draw_weights(k, models, 50_000 + seed)).to(DEV)


def _features(rows, k, seed):
    """Feature rows of the measurement-kernel families (sparse counts up to about 2^43),
    drawn from a pool of 16,384 with a repeat factor per row."""
    pool = W.fit_features(16384, 32, seed)
    pool = torch.from_numpy(pool if k == 32 else np.ascontiguousarray(pool[:, FIT_COLS_12])).to(DEV)
    g = _gen(seed)
    pick = torch.randint(len(pool), (rows,), generator=g, device=DEV)
    return pool[pick] * torch.randint(1, 512, (rows, 1), generator=g, device=DEV)


def _count_inputs(case, seed):
    P = len(W.TEMPLATE_PARAMS[case["template"]])
    return torch.from_numpy(W.draw_points(P, case["points"], 1000 * seed + 7)).to(DEV)


def _topk_inputs(case, seed):
    F, w = _features(case["rows"], case["k"], seed), _weights(case["k"], case["models"], seed)
    cuts = np.sort(np.random.default_rng(seed).integers(0, case["rows"] + 1, size=case["groups"] - 1))
    return F, w, np.concatenate([[0], cuts, [case["rows"]]]).astype(np.int64)


def _point_inputs(case, seed):
    """Counts of every (table, point) pair, the weights, and per point the list of its rows."""
    n, T = case["points"], case["tables"]
    ids = _template_tables(case["template"], T, 32)
    F = torch.empty((T, n, 32), dtype=torch.int64, device=DEV)
    _context().eval_counts(ids, _count_inputs(case, seed), F)
    rows = (torch.arange(T, device=DEV)[None, :] * n + torch.arange(n, device=DEV)[:, None]).reshape(-1).contiguous()
    return F.view(T * n, 32), _weights(32, case["models"], seed), rows, np.arange(0, T * n + 1, T, dtype=np.int64)


def _fit_inputs(case, seed):
    """Measured feature rows and their timings: the linear model times exp(0.05 N(0, 1))."""
    F = W.fit_features(case["rows"], 32, seed)
    F = torch.from_numpy(F if case["k"] == 32 else np.ascontiguousarray(F[:, FIT_COLS_12])).to(DEV)
    w = _weights(case["k"], case["models"], seed)
    e = torch.randn((case["rows"], case["models"]), generator=_gen(seed), dtype=torch.float64, device=DEV)
    return F, (F.double() @ w.T) * torch.exp(0.05 * e)


def prepare(case, seed):
    kind = case["kind"]
    st = dict(case=case)
    if kind == "counts":
        st["ids"] = np.array(_template_tables(case["template"], case["tables"], case["layout"]), dtype=np.int32)
        st["points"] = _count_inputs(case, seed)
        st["out"] = torch.empty((case["tables"], case["points"], case["layout"]), dtype=torch.int64, device=DEV)
    elif kind in ("predict", "argmin"):
        st["F"], st["w"] = _features(case["rows"], case["k"], seed), _weights(case["k"], case["models"], seed)
        if kind == "predict":
            st["T"] = torch.empty((case["rows"], case["models"]), dtype=torch.float64, device=DEV)
        else:
            st["arg"] = torch.empty(case["models"], dtype=torch.int64, device=DEV)
            st["min"] = torch.empty(case["models"], dtype=torch.float64, device=DEV)
    elif kind in ("topk", "points"):
        if kind == "topk":
            (st["F"], st["w"], st["seg"]), st["rows"] = _topk_inputs(case, seed), None
        else:
            st["F"], st["w"], st["rows"], st["seg"] = _point_inputs(case, seed)
        shape = (len(st["seg"]) - 1, case["models"], case["topk"])
        st["idx"] = torch.empty(shape, dtype=torch.int64, device=DEV)
        st["t"] = torch.empty(shape, dtype=torch.float64, device=DEV)
    elif kind == "rank":
        st["tables"], st["var_off"], templates = _space(case["variants"], case["coupled"])
        points, st["pt_off"] = _template_points(templates, case["points"], seed)
        st["points"] = torch.from_numpy(points).to(DEV)
        st["w"] = _weights(32, 1, seed)[0].contiguous()
        st["idx"] = torch.empty((len(points), case["topk"]), dtype=torch.int32, device=DEV)
        st["t"] = torch.empty((len(points), case["topk"]), dtype=torch.float64, device=DEV)
    elif kind == "fit":
        st["F"], st["T"] = _fit_inputs(case, seed)
        st["W"] = torch.empty((case["models"], case["k"]), dtype=torch.float64, device=DEV)
    else:
        # a serving process of its own: the tables of a 1,000-variant space loaded from their images
        tables, var_off, templates = _space(1000, False)
        sv = B.Context(0, 64 << 20)
        ids = {t: sv.table_load(_context().table_image(t)) for t in sorted(set(tables.tolist()))}
        tables = np.array([ids[t] for t in tables.tolist()], dtype=np.int32)
        points, pt_off = _template_points(templates, 512, seed)
        sv.serve_set_weights(W.draw_weights(32, 64, 50_000 + seed))
        sv.serve_start()
        # the burst's candidate counts are those of the query stream, the candidates the seed's
        sizes = [len(q.variant) for q in W.draw_queries(case["queries"], 2000.0, np.diff(var_off), 512, 64, 9, case["max_cand"])]
        rng = np.random.default_rng(seed)
        st["idx"] = np.empty((len(sizes), case["topk"]), dtype=np.int32)
        st["t"] = np.empty((len(sizes), case["topk"]), dtype=np.float64)
        st["sv"], st["keep"], st["queries"] = sv, [], []
        for i, n in enumerate(sizes):
            t = int(rng.integers(len(templates)))
            tab = np.ascontiguousarray(tables[rng.integers(var_off[t], var_off[t + 1], size=n)])
            pts = np.ascontiguousarray(points[rng.integers(pt_off[t], pt_off[t + 1], size=n)])
            st["keep"].append((tab, pts))
            st["queries"].append(B.make_query(int(rng.integers(64)), case["topk"], tab, pts, st["idx"][i], st["t"][i]))
    return st


def run(st):
    case = st["case"]
    kind = case["kind"]
    if kind == "serve":
        tickets = [st["sv"].serve_submit(q) for q in st["queries"]]
        for t in tickets:
            while st["sv"].serve_poll(t, 1_000_000) == B.PM_PENDING:
                pass
        return {"idx": st["idx"], "t": st["t"]}
    ctx = _context()
    if kind == "counts":
        ctx.eval_counts(st["ids"], st["points"], st["out"])
        return st["out"]
    if kind == "predict":
        ctx.predict(st["F"], st["w"], st["T"], PREC[case["prec"]])
        return st["T"]
    if kind == "argmin":
        ctx.predict_argmin(st["F"], st["w"], st["arg"], st["min"], PREC[case["prec"]])
        return {"arg": st["arg"], "min": st["min"]}
    if kind in ("topk", "points"):
        ctx.predict_topk(st["F"], st["w"], st["seg"], case["topk"], st["idx"], st["t"], rows=st["rows"])
        return {"idx": st["idx"], "t": st["t"]}
    if kind == "rank":
        ctx.eval_predict_topk(st["tables"], st["var_off"], st["points"], st["pt_off"], st["w"], case["topk"], st["idx"], st["t"])
        return {"idx": st["idx"], "t": st["t"]}
    _, reports = ctx.fit_weights(st["F"], st["T"], st["W"], B.FIT_RELATIVE if case["objective"] == "relative" else B.FIT_ABSOLUTE,
                                 PREC[case["prec"]], 3)
    return {"W": st["W"], "rank": np.array([r["rank"] for r in reports], dtype=np.int64)}


def work(case):
    """Each input read once and each output written once; a multiply and an add per
    feature and prediction (per entry of the normal equations for a fit)."""
    kind = case["kind"]
    if kind == "counts":
        P = len(W.TEMPLATE_PARAMS[case["template"]])
        return {"bytes": 8 * case["points"] * (P + case["tables"] * case["layout"]), "flops": 0}
    if kind in ("predict", "argmin", "topk"):
        R, k, M = case["rows"], case["k"], case["models"]
        out = {"predict": R * M * 8, "argmin": M * 16}.get(kind, case.get("groups", 0) * M * case.get("topk", 0) * 16)
        return {"bytes": R * k * 8 + M * k * 8 + out, "flops": 2 * R * k * M}
    if kind == "points":
        R, M = case["tables"] * case["points"], case["models"]
        return {"bytes": R * (32 * 8 + 8) + case["points"] * M * case["topk"] * 16, "flops": 2 * R * 32 * M}
    if kind == "rank":
        n = case["points"] * (3 if case["coupled"] else 8)
        return {"bytes": n * (32 + 12 * case["topk"]), "flops": 64 * case["variants"] * case["points"]}
    if kind == "fit":
        R, k, M = case["rows"], case["k"], case["models"]
        return {"bytes": 8 * (R * k + R * M + M * k), "flops": M * R * (k * (k + 1) + 4 * 3 * k)}
    n = case["queries"] * case["max_cand"] // max(1, int(math.log(case["max_cand"] + 1)))   # mean of the log-uniform sizes
    return {"bytes": n * 36 + case["queries"] * case["topk"] * 12, "flops": 64 * n}


def exact(case, seed):
    """Plain 64-bit torch.  Counts are whole numbers, which are compared as they are; the
    fused and the served rankings start from counts that only the compiled tables give."""
    kind = case["kind"]
    if kind == "predict":
        return _features(case["rows"], case["k"], seed).double() @ _weights(case["k"], case["models"], seed).T
    if kind == "argmin":
        T = _features(case["rows"], case["k"], seed).double() @ _weights(case["k"], case["models"], seed).T
        return {"arg": None, "min": T.min(dim=0).values}
    if kind in ("topk", "points"):
        if kind == "topk":
            F, w, seg = _topk_inputs(case, seed)
            T = F.double() @ w.T
        else:
            F, w, rows, seg = _point_inputs(case, seed)
            T = (F.double() @ w.T)[rows]
        if len(seg) - 1 > 5000:
            return None
        out = torch.full((len(seg) - 1, case["models"], case["topk"]), math.inf, dtype=torch.float64, device=DEV)
        for g in range(len(seg) - 1):
            n = min(case["topk"], int(seg[g + 1] - seg[g]))
            if n:
                out[g, :, :n] = T[seg[g]:seg[g + 1]].topk(n, dim=0, largest=False, sorted=True).values.T
        return {"idx": None, "t": out}
    if kind == "fit":
        F, T = _fit_inputs(case, seed)
        s = F.abs().max(dim=0).values.double().clamp(min=1)
        out = torch.empty((case["models"], case["k"]), dtype=torch.float64, device=DEV)
        for m in range(case["models"]):
            t = T[:, m:m + 1]
            A, b = (F.double() / s / t, torch.ones_like(t)) if case["objective"] == "relative" else (F.double() / s, t)
            c = A.abs().max(dim=0).values
            A = A / c
            L = torch.linalg.cholesky(A.T @ A)
            x = torch.cholesky_solve(A.T @ b, L)
            for _ in range(3):
                x = x + torch.cholesky_solve(A.T @ (b - A @ x), L)
            out[m] = x[:, 0] / c / s
        return {"W": out, "rank": None}
    return None
