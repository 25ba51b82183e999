"""The FP64-accurate prediction on the tensor cores (exact digit products): bit for bit
against the fixed-point scheme in Python integers (weights rounded once, exact sums, the
57 leading bits rounded to FP64), for ragged row counts, feature and model counts around
the kernel's paddings, unaligned buffers, and counts over the whole int64 range."""
import math
from fractions import Fraction

import numpy as np
import pytest

from paper_1604_04997_gb300 import binding as B

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def env():
    import torch
    import __graft_entry__
    __graft_entry__.build()
    ctx = B.Context(0, 64 << 20)
    yield ctx, torch.device("cuda:0")
    ctx.close()


def scheme(F, Wm):
    """The times of pm_predict at PM_PREC_FP64, from Python integers."""
    Fo = F.astype(object)
    T = np.empty((F.shape[0], len(Wm)))
    for m, w in enumerate(Wm):
        s = 0.0
        for x in w:
            s += abs(float(x))
        s *= 1.0 + 2.0 ** -40
        E = 62 - (math.frexp(s)[1] if s > 0 else 0)
        Wi = np.array([round(Fraction(float(x)) * Fraction(2) ** E) for x in w], dtype=object)
        for r, S in enumerate(Fo @ Wi):
            a, n = abs(int(S)), abs(int(S)).bit_length()
            if not a:
                T[r, m] = 0.0
                continue
            y = a >> (n - 57) if n > 57 else a << (57 - n)
            t = math.ldexp((y + 7 + ((y >> 4) & 1)) >> 4, n - 53 - E)
            T[r, m] = -t if S < 0 else t
    return T


def counts(R, k, rng):
    """Counts of every magnitude and sign: digit boundaries, the ends of int64, sparse rows."""
    F = (rng.integers(-(1 << 63), (1 << 63) - 1, size=(R, k), dtype=np.int64) >> rng.integers(0, 64, size=(R, k)))
    edge = np.array([0, 1, -1, 127, 128, -128, -129, 0x7F7F, 0x8080, 1 << 46, (1 << 46) - 1, -(1 << 46), (1 << 62) - 1,
                     (1 << 63) - 1, -(1 << 63), 0x7F7F7F7F7F7F7F7F, 0x7F80808080808080,
                     -0x7F80808080808080], dtype=np.int64)
    pick = rng.random((R, k)) < 0.3
    F[pick] = rng.choice(edge, size=int(pick.sum()))
    F[rng.random(R) < 0.1] = 0
    return F


def weights(M, k, rng):
    """Signs mixed, magnitudes spread over ten decades, some zero."""
    w = rng.uniform(-1, 1, size=(M, k)) * 10.0 ** rng.uniform(-13, -3, size=(M, k))
    w[rng.random((M, k)) < 0.1] = 0.0
    if M > 2:
        w[2] = 0.0
    return w


@pytest.mark.parametrize("R,k,M,shift", [(1, 1, 1, 0), (7, 5, 2, 1), (127, 12, 3, 0), (128, 16, 16, 0), (129, 17, 17, 1),
                                         (300, 31, 33, 0), (300, 32, 48, 1), (257, 32, 63, 0), (400, 32, 64, 0), (40, 33, 5, 0)])
def test_predict_and_argmin_equal_the_integer_scheme(env, R, k, M, shift):
    import torch
    ctx, dev = env
    rng = np.random.default_rng(R * 1000 + k * 10 + M)
    F, w = counts(R, k, rng), weights(M, k, rng)
    flat = torch.empty(R * k + shift, dtype=torch.int64, device=dev)   # shift: 8 bytes off a 16-byte boundary
    dF = flat[shift:].view(R, k)
    dF.copy_(torch.from_numpy(F))
    dW = torch.from_numpy(w).to(dev)
    T = torch.full((R * M + shift + 8,), math.nan, dtype=torch.float64, device=dev)
    ctx.predict(dF, dW, T[shift:shift + R * M].view(R, M))
    ctx.sync_status()
    got = T.cpu().numpy()
    assert np.isnan(got[:shift]).all() and np.isnan(got[shift + R * M:]).all()   # nothing outside T
    ref = scheme(F, w)
    assert np.array_equal(got[shift:shift + R * M].reshape(R, M).view(np.int64), ref.view(np.int64))
    arg = torch.empty(M, dtype=torch.int64, device=dev)
    mn = torch.empty(M, dtype=torch.float64, device=dev)
    for static in (False, True):
        if static:
            B.predict_argmin_static(dF, dW, arg, mn)
        else:
            ctx.predict_argmin(dF, dW, arg, mn)
        ctx.sync_status()
        assert np.array_equal(arg.cpu().numpy(), ref.argmin(axis=0))
        assert np.array_equal(mn.cpu().numpy(), ref.min(axis=0))


@pytest.mark.parametrize("bits", [1, 6, 7, 14, 38, 39, 46, 47, 54, 62])
def test_tiles_of_every_digit_count(env, bits):
    """More tiles than SMs, each with counts of at most `bits` bits, with one larger tile
    in between: tiles that skip digits follow tiles that do not."""
    import torch
    ctx, dev = env
    rng = np.random.default_rng(bits)
    R, k, M = 128 * 400 + 5, 32, 4
    F = rng.integers(-(1 << bits), 1 << bits, size=(R, k), dtype=np.int64)
    F[128 * 160:128 * 161] = counts(128, k, rng)
    w = weights(M, k, rng)
    T = torch.empty((R, M), dtype=torch.float64, device=dev)
    ctx.predict(torch.from_numpy(F).to(dev), torch.from_numpy(w).to(dev), T)
    ctx.sync_status()
    rows = np.r_[0:40, 128 * 152 - 3:128 * 152 + 3, 128 * 160 - 2:128 * 161 + 2, 128 * 312 - 2:128 * 312 + 2, R - 8:R]
    assert np.array_equal(T.cpu().numpy()[rows].view(np.int64), scheme(F[rows], w).view(np.int64))
