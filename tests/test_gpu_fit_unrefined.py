"""pm_fit_weights without refinement (refine_steps = 0): the weights of a three-term Gram are
within cond(A)^2 2^-18 where that is well below one; where it is not (nearly collinear columns, the
absolute objective over counts that span many decades) the exact Gram is used, whose entries
are rounded at 2^-47.  Against the oracle's QR."""
import numpy as np
import pytest

import oracle
from paper_1604_04997_gb300 import binding as B
from paper_1604_04997_gb300 import workloads as W
from test_gpu_fit import _fit, _scaled_err, env  # noqa: F401  (env: the context fixture)

pytestmark = pytest.mark.gpu
COLS_12 = [0, 1, 2, 3, 4, 5, 6, 7, 13, 15, 17, 24]


@pytest.mark.parametrize("objective", ["relative", "absolute"])
@pytest.mark.parametrize("R,k,M,seed", [(1000, 32, 1, 1), (1000, 32, 1, 2), (1000, 32, 2, 3), (4000, 32, 3, 1), (4096, 32, 4, 2),
                                        (1000, 12, 3, 1), (20000, 12, 2, 1)])
def test_unrefined_weights(env, R, k, M, seed, objective):  # noqa: F811
    ctx, dev = env
    F = W.fit_features(R, 32, seed)
    F = F if k == 32 else np.ascontiguousarray(F[:, COLS_12])
    T = W.synth_timings(F, W.draw_weights(k, M, 50_000 + seed), seed)
    rc, rep, Wg = _fit(ctx, dev, F, T, B.FIT_RELATIVE if objective == "relative" else B.FIT_ABSOLUTE, steps=0)
    assert rc == 0
    for m in range(M):
        wref, rank, cond, res = oracle.fit(F, T[:, m], objective)
        c2 = cond * cond
        assert rank == k and rep[m]["rank"] == k
        # 4 k: the solve's k-term sums on both sides
        assert _scaled_err(F, T, m, Wg[m], wref, objective) <= (c2 * 2.0 ** -18 if c2 < 2.0 ** 14 else 4 * k * c2 * 2.0 ** -47)
        assert rep[m]["rel_resid"] <= 1.01 * res
