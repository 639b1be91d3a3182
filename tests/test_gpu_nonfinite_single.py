"""NaN and infinity through the single-precision products, on both tensor-core paths: an operand is split into two TF32
numbers, and what is not finite in it has to be in the pair, whatever its bits (0x7fffffff is the NaN of GPU arithmetic).

A value that is not finite makes every output entry that is a sum over it NaN and leaves the bits of all others alone.
"""
import ctypes as C

import numpy as np
import pytest
import torch

from oracle import rrf_oracle as orc
from paper_2608_28941_b200 import rrf

pytestmark = pytest.mark.gpu

MMA, TC = 0, 1
BITS = [0x7fffffff, 0xffffffff, 0x7fc00000, 0x7f800001, 0x7f800000, 0xff800000]


@pytest.fixture(scope="module")
def h():
    handle = rrf.rrf_create(0)
    yield handle
    rrf.rrf_destroy(handle)


def basis(m, k, b, rng):
    V, T = np.zeros((m, k)), np.zeros((b, k))
    for r in range(0, k, b):
        V[r:, r:r + b], _, T[:, r:r + b], _ = orc.panel_qr(rng.standard_normal((m - r, b)))
    return dev(V), dev(T)


def dev(x):
    return torch.from_numpy(np.ascontiguousarray(x.astype(np.float32))).cuda()


def planted(x, i, j, bits):
    x = x.clone()
    x.view(torch.int32)[i, j] = int(np.uint32(bits).astype(np.int32))
    return x


def only(got, clean, where):
    """got is NaN where `where` says and has the bits of `clean` elsewhere."""
    assert torch.isnan(got[where]).all()
    assert torch.isfinite(clean).all()
    assert torch.equal(got[~where], clean[~where])


def mask(like, rows=slice(None), cols=slice(None)):
    w = torch.zeros(like.shape, dtype=torch.bool, device=like.device)
    w[rows, cols] = True
    return w


def sample(h, Cm, OmT):
    lib, (rows, n), b = rrf.load(), Cm.shape, OmT.shape[0]
    need = C.c_size_t()
    assert lib.rrf_sample_workspace_bytes(rrf.RRF_F32, rows, b, C.byref(need)) == rrf.RRF_OK
    ws = torch.empty(need.value, dtype=torch.uint8, device="cuda")
    Y = torch.empty((rows, b), dtype=torch.float32, device="cuda")
    assert lib.rrf_sample_panel(h, rrf.RRF_F32, rows, n, b, C.c_void_p(Cm.data_ptr()), Cm.stride(0), C.c_void_p(OmT.data_ptr()),
                                OmT.stride(0), C.c_void_p(Y.data_ptr()), C.c_void_p(ws.data_ptr()), ws.numel(), None) == rrf.RRF_OK
    torch.cuda.synchronize()
    return Y


@pytest.mark.parametrize("bits", BITS)
@pytest.mark.parametrize("rows,n,b", [(300, 200, 32), (515, 1004, 64), (260, 516, 128)])
def test_sample(h, rows, n, b, bits):
    rng = np.random.default_rng(rows)
    Cm, Om = dev(rng.standard_normal((rows, n))), dev(rng.standard_normal((b, n)))
    clean = sample(h, Cm, Om)
    only(sample(h, planted(Cm, rows - 7, n - 1, bits), Om), clean, mask(clean, rows - 7))
    only(sample(h, Cm, planted(Om, b - 3, 5, bits)), clean, mask(clean, slice(None), b - 3))


@pytest.mark.parametrize("bits", BITS)
@pytest.mark.parametrize("engine", [MMA, TC])
@pytest.mark.parametrize("m,n,b,k", [(200, 72, 32, 64), (517, 400, 64, 128), (400, 260, 128, 256)])
def test_apply(h, engine, m, n, b, k, bits):
    rng = np.random.default_rng(m)
    V, T = basis(m, k, b, rng)
    Cm = dev(rng.standard_normal((m, n)))
    rrf.rrf_set_single_engine(h, engine, 2)
    try:
        for fn in (rrf.rrf_apply_qt, rrf.rrf_apply_q):
            clean = fn(h, V, T, b, k, Cm.clone())
            # the first block's reflectors reach every row, so the whole column depends on the entry
            only(fn(h, V, T, b, k, planted(Cm, m - 2, n - 3, bits)), clean, mask(clean, slice(None), n - 3))
        # in V: every entry of the rows which that block touches, which is the last to be applied here
        clean = rrf.rrf_apply_qt(h, V, T, b, k, Cm.clone())
        only(rrf.rrf_apply_qt(h, planted(V, m - 2, k - 5, bits), T, b, k, Cm.clone()), clean, mask(clean, slice(k - b, None)))
    finally:
        rrf.rrf_set_single_engine(h, TC, 2)


@pytest.mark.parametrize("bits", BITS)
@pytest.mark.parametrize("engine", [MMA, TC])
@pytest.mark.parametrize("m,b,k_old,k_new,n", [
    (300, 32, 64, 32, 100),       # through the small product of the bases
    (700, 64, 192, 64, 400),
    (300, 32, 64, 32, 60),        # M itself through all reflectors
])
def test_transfer(h, engine, m, b, k_old, k_new, n, bits):
    rng = np.random.default_rng(m + n)
    Vo, To = basis(m, k_old, b, rng)
    Vn, Tn = basis(m, k_new, b, rng)
    M = dev(rng.standard_normal((k_old, n)))
    rrf.rrf_set_single_engine(h, engine, 2)
    try:
        clean = rrf.rrf_subspace_transfer(h, Vo, To, k_old, Vn, Tn, k_new, b, M)
        for row in (1, k_old - 1):
            got = rrf.rrf_subspace_transfer(h, Vo, To, k_old, Vn, Tn, k_new, b, planted(M, row, 9, bits))
            only(got, clean, mask(clean, slice(None), 9))
    finally:
        rrf.rrf_set_single_engine(h, TC, 2)


def test_the_split_rounds_to_nearest(h):
    """hi and lo against their definition, round to 11 significant bits, ties away from zero, in exact arithmetic."""
    rng = np.random.default_rng(0)
    bits = rng.integers(0, 1 << 32, 1 << 20, dtype=np.uint64).astype(np.uint32)
    edge = np.array([0, 0x1000, 0x0fff, 0x1001, 0x2000, 0x3000], dtype=np.uint32)        # ties and their neighbours
    expo = (np.arange(256, dtype=np.uint32) << 23)[:, None]
    bits = np.concatenate([bits, (expo + edge).ravel(), (expo + edge).ravel() | np.uint32(1 << 31),
                           np.array([0x7f7fefff, 0x7f7fe000], dtype=np.uint32)])          # the largest that does not overflow
    x = bits.view(np.float32)
    x = x[np.isfinite(x) & (np.abs(x) < np.float32(2.0) ** 127 * np.float32(2 - 2.0 ** -11))]
    hi, lo = (t.cpu().numpy() for t in rrf.rrf_selftest_arithmetic(h, 0, torch.from_numpy(x).cuda()))
    lo = (lo.view(np.uint32) & np.uint32(0xffffe000)).view(np.float32)         # what the tensor core reads of it

    def tf32(v):                                             # float32 values, in float64
        v = v.astype(np.float64)
        quantum = np.ldexp(1.0, np.maximum(np.frexp(v)[1] - 11, -126 - 10))
        return np.copysign(np.floor(np.abs(v) / quantum + 0.5) * quantum, v)

    assert np.array_equal(hi.astype(np.float64), tf32(x))
    assert np.array_equal(lo.astype(np.float64), tf32((x - hi).astype(np.float32)))      # the difference is exact
    assert (np.abs(x.astype(np.float64) - hi - lo) <= np.maximum(2.0 ** -22 * np.abs(x.astype(np.float64)), 2.0 ** -137)).all()
    bad = np.array([b for b in BITS], dtype=np.uint32).view(np.float32)
    hi, lo = rrf.rrf_selftest_arithmetic(h, 0, torch.from_numpy(bad).cuda())
    assert torch.isnan(lo).all()
