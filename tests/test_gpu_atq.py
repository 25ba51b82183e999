"""The fit's U^T q adds its warps' float-float sums no worse than FP64 does.  One row per warp
and U = 1, so every warp's sum is its q as it stands, exactly: the result may then differ from
the exact sum by two FP64 roundings of the result, and by the third FP32 sum's rounding (eight
steps of at most 2^-24 of 2^-44 of the largest part)."""
import ctypes
from fractions import Fraction

import numpy as np
import pytest

from paper_1604_04997_gb300 import binding as B

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("case", ["equal", "spread", "cancel", "zeros", "tiny", "huge"])
def test_sum_of_the_warps(case):
    import torch
    import __graft_entry__
    __graft_entry__.build()
    rng = np.random.default_rng(len(case))
    M = 16
    h = (rng.standard_normal((8, M)) * {"equal": 1.0, "spread": 1.0, "cancel": 1.0, "zeros": 0.0, "tiny": 2.0 ** -90, "huge": 2.0 ** 100}[case])
    if case == "spread":
        h *= 2.0 ** rng.integers(-40, 1, size=(8, M))
    if case == "cancel":
        h[4:] = -h[:4] * (1 + 2.0 ** -20 * rng.standard_normal((4, M)))
    h = h.astype(np.float32)
    l = (h.astype(float) * 2.0 ** -24 * rng.uniform(-1, 1, size=(8, M))).astype(np.float32)
    if case == "zeros":
        l = (rng.standard_normal((8, M)) * 2.0 ** -30).astype(np.float32)   # all that is left of a cancelled sum
    dev = "cuda:0"
    one = torch.ones((8, 32), dtype=torch.float32, device=dev)
    amax = torch.full((M, 32), int(np.float32(0.5).view(np.int32)), dtype=torch.int32, device=dev)   # exponent 0
    g = torch.zeros((M, 32), dtype=torch.float64, device=dev)
    qh, ql = torch.from_numpy(h).to(dev), torch.from_numpy(l).to(dev)
    zero = torch.zeros_like(one)
    f = B.lib().pmx_atq
    f.restype = ctypes.c_int
    p = [ctypes.c_void_p(x.data_ptr()) for x in (one, zero, qh, ql)]
    assert f(*p, ctypes.c_int64(8), 32, M, ctypes.c_void_p(amax.data_ptr()), ctypes.c_void_p(g.data_ptr()), None) == B.PM_OK
    torch.cuda.synchronize()
    got = g.cpu().numpy()
    for m in range(M):
        exact = sum(Fraction(float(x)) for x in h[:, m]) + sum(Fraction(float(x)) for x in l[:, m])
        largest = max(abs(float(x)) for x in np.concatenate([h[:, m], l[:, m]]))
        bound = 8 * largest * 2.0 ** -68 + abs(float(exact)) * 2.0 ** -52
        for c in (0, 17, 31):
            assert abs(float(Fraction(got[m, c]) - exact)) <= bound, (case, m, c)
