"""pm_fit_weights at the edges of its kernels' tiles (columns, models, rows) against the
oracle's Householder QR: the weights to 1e-8 of the scaled problem, as the well-conditioned
problems of test_gpu_fit."""
import numpy as np
import pytest

import oracle
from paper_1604_04997_gb300 import binding as B
from test_gpu_fit import _fit, _scaled_err, env  # noqa: F401  (env: the context fixture)

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", [B.PREC_BF16X3, B.PREC_FP64], ids=["bf16x3", "fp64"])
@pytest.mark.parametrize("R,k,M", [(40, 1, 1), (65, 31, 17), (129, 13, 16), (4097, 32, 64), (9000, 2, 63), (20481, 17, 33)])
def test_fit_edges_match_qr(env, R, k, M, precision):  # noqa: F811
    ctx, dev = env
    rng = np.random.default_rng(R + k)
    F = rng.integers(0, 1 << 20, size=(R, k)) << rng.integers(0, 20, size=k)
    F[:, 0] += 1
    T = (F.astype(float) @ rng.uniform(0.1, 1.0, size=(k, M))) * np.exp(0.05 * rng.standard_normal((R, M))) * 1e-9
    rc, rep, Wg = _fit(ctx, dev, F, T, precision=precision)
    assert rc == 0
    for m in sorted({0, M // 2, M - 1}):
        wref, rank, cond, res = oracle.fit(F, T[:, m], "relative")
        assert rank == k and cond <= 1e6 and rep[m]["rank"] == k
        assert _scaled_err(F, T, m, Wg[m], wref, "relative") <= 1e-8
