"""Waits that run out in the working warps of the exact tensor-core kernels (prediction, top-k,
the fit's Gram) after their issuing warp has left: the status names the timeout, the kernel
ends, and the context stays usable.  The hooks run the kernels with an issuing warp that leaves
early by design (in bounds, nothing broken) and waits of 2 ms."""
import ctypes
import time

import numpy as np
import pytest

from paper_1604_04997_gb300 import binding as B

pytestmark = pytest.mark.gpu
TIMEOUT = 4   # the status bit of a device wait that ran out


def _hook(name, *args):
    """One call: status word after it, and its seconds."""
    import torch
    f = getattr(B.lib(), name)
    f.restype = ctypes.c_int
    status = torch.zeros(1, dtype=torch.int32, device="cuda:0")
    torch.cuda.synchronize()
    t0 = time.perf_counter()
    c = [ctypes.c_void_p(a.data_ptr()) if hasattr(a, "data_ptr") else a for a in args]
    assert f(*c, ctypes.c_void_p(status.data_ptr()), None) == B.PM_OK
    torch.cuda.synchronize()
    return int(status[0]), time.perf_counter() - t0


@pytest.fixture(scope="module")
def env():
    import torch
    import __graft_entry__
    __graft_entry__.build()
    ctx = B.Context(0)
    g = torch.Generator(device="cuda:0")
    g.manual_seed(3)
    F = torch.randint(0, 1 << 20, (400, 12), generator=g, device="cuda:0")
    w = torch.rand((5, 12), generator=g, dtype=torch.float64, device="cuda:0") * 1e-9
    yield ctx, F, w
    T = torch.empty((400, 5), dtype=torch.float64, device="cuda:0")
    ctx.predict(F, w, T)   # the same kernels still run
    ctx.sync_status()
    ref = F.double() @ w.T
    assert bool(((T - ref).abs() <= 1e-12 * ref).all())
    ctx.close()


def test_predict_reports(env):
    import torch
    _, F, w = env
    T = torch.empty((400, 5), dtype=torch.float64, device="cuda:0")
    status, s = _hook("pmx_predict_held", F, ctypes.c_int64(400), 12, w, 5, T)
    assert status & TIMEOUT and s < 5
    ref = F.double() @ w.T
    assert bool(((T[:128] - ref[:128]).abs() <= 1e-12 * ref[:128]).all())   # the tile that was issued


def test_argmin_without_a_status_reports(env):
    """pm_predict_argmin_static has no status: a timeout gives row -1 and NaN."""
    import torch
    _, F, w = env
    part = torch.zeros((5, 2), dtype=torch.int64, device="cuda:0")
    arg = torch.zeros(5, dtype=torch.int64, device="cuda:0")
    mn = torch.zeros(5, dtype=torch.float64, device="cuda:0")
    status, s = _hook("pmx_argmin_held", F, ctypes.c_int64(400), 12, w, 5, part, arg, mn)
    assert status & TIMEOUT and s < 5
    assert (arg.cpu() == -1).all() and mn.cpu().isnan().all()


@pytest.mark.parametrize("hook", ["pmx_topk_held", "pmx_topk_unwritten"])
@pytest.mark.parametrize("cuts", [[0, 400], [0, 100, 100, 130, 400]], ids=["tiles", "units"])
def test_topk_reports(env, cuts, hook):
    import torch
    _, F, w = env
    G = len(cuts) - 1
    units = np.zeros((G, 3), dtype=np.int64)   # p0, p1, (g, part) as two 32-bit words
    units[:, 0], units[:, 1] = cuts[:-1], cuts[1:]
    units[:, 2] = np.arange(G) | (0xFFFFFFFF << 32) - (1 << 64)
    u = torch.from_numpy(units).to("cuda:0")
    idx = torch.zeros((G, 5, 4), dtype=torch.int64, device="cuda:0")
    tt = torch.zeros((G, 5, 4), dtype=torch.float64, device="cuda:0")
    status, s = _hook(hook, F, ctypes.c_int64(400), 12, w, 5, u, G, 4, idx, tt)
    assert status & TIMEOUT and s < 5


@pytest.mark.parametrize("rows", [16, 700, 1024])
def test_gram_reports(env, rows):
    import torch
    g = torch.Generator(device="cuda:0")
    g.manual_seed(rows)
    U, rfh = (torch.rand((rows, 32), generator=g, device="cuda:0") for _ in range(2))
    rfl = torch.zeros_like(rfh)
    one = np.float32(1.0).view(np.int32).item()
    amax = torch.full((5, 32), one, dtype=torch.int32, device="cuda:0")
    rmax = torch.full((5,), one, dtype=torch.int32, device="cuda:0")
    G = torch.zeros((5, 32, 32), dtype=torch.float64, device="cuda:0")
    status, s = _hook("pmx_gram_held", U, rfh, rfl, ctypes.c_int64(rows), 12, 5, amax, rmax, G)
    assert status & TIMEOUT and s < 5
    assert not bool(G.any())   # no sums were reported
