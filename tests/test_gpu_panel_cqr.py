"""Panels through the Cholesky QR with Householder reconstruction, and those it hands to the column loop.

The factors are held to the oracle's within c u cond, the first-order perturbation bound of a QR factorisation (u the
unit round-off, cond the condition number of the panel with its columns scaled to unit length, which is what both
factorisations see; c = 100 covers the sums over b columns).
"""
import ctypes as C

import numpy as np
import pytest
import torch

from oracle import rrf_oracle as orc
from paper_2608_28941_b200 import rrf

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def h():
    handle = rrf.rrf_create(0)
    yield handle
    rrf.rrf_destroy(handle)


def panel(kind, rows, b, rng):
    Y = rng.standard_normal((rows, b))
    if kind.startswith("cond"):                    # singular values from 1 down to 10^-x
        s = 10.0 ** (-float(kind[4:]) * np.arange(b) / (b - 1))
        Y = (np.linalg.qr(Y)[0] * s) @ rng.standard_normal((b, b))
    elif kind == "graded":                         # columns of very different lengths
        Y *= 10.0 ** (-12.0 * np.arange(b) / (b - 1))
    elif kind == "dependent":                      # column loop: two equal columns
        Y[:, b // 2] = Y[:, 1]
    elif kind == "zero":                           # column loop: a column of zeros
        Y[:, 3] = 0.0
    elif kind == "nothing-below":                  # column loop, on the orthonormal panel: tau = 0 in some columns
        Y[b:] = 0.0
        Y[:b] = np.triu(Y[:b]) + 3.0 * np.eye(b)
    elif kind == "near":                           # second factor by a factorisation: two columns 1e-5 apart
        Y[:, b // 2] = Y[:, 1] + 1e-5 * Y[:, b // 2]
    elif kind == "nearer":                         # column loop: 1e-7 apart, a pivot of 1e-14
        Y[:, b // 2] = Y[:, 1] + 1e-7 * Y[:, b // 2]
    elif kind == "huge":                           # column loop: squares overflow
        Y *= 1e160
    return Y


def check(h, Y, dtype, c=100.0):
    rows, b = Y.shape
    Y = Y.astype(np.float32).astype(np.float64) if dtype == "f32" else Y
    V, T = rrf.rrf_panel_qr(h, torch.from_numpy(Y.astype(np.float32) if dtype == "f32" else Y).cuda())
    assert rrf.rrf_last_status(h) == rrf.RRF_OK
    V, T = V.cpu().numpy().astype(np.float64), T.cpu().numpy().astype(np.float64)
    Vo, _, To, _ = orc.panel_qr(Y)
    norms = np.linalg.norm(Y, axis=0)
    s = np.linalg.svd(Y / np.where(norms > 0, norms, 1.0), compute_uv=False)
    cond = s[0] / s[-1] if s[-1] > 1e-12 * s[0] else None
    store = 2.0 ** -24 if dtype == "f32" else 0.0
    Q = np.eye(rows, b) - V @ (T @ V[:b].T)
    assert np.linalg.norm(Q.T @ Q - np.eye(b)) <= (5e-6 if dtype == "f32" else 1e-13) * b
    if cond is not None:
        tol = c * 1.1e-16 * cond + store
        assert np.max(np.abs(V - Vo)) <= tol * np.max(np.abs(Vo))
        assert np.max(np.abs(T - To)) <= 10 * tol * np.max(np.abs(To))
    return V, T


@pytest.mark.parametrize("b", [16, 32, 64])
@pytest.mark.parametrize("extra", [1, 7, 48, 65, 1023, 3072, 4097, 9000])
def test_heights(h, b, extra):
    """One row more than columns, strips of 16 and slabs that end in a remainder, one cluster and the whole grid."""
    rows = b + extra
    check(h, panel("gauss", rows, b, np.random.default_rng(rows)), "f64")


@pytest.mark.parametrize("b", [16, 32, 64])
@pytest.mark.parametrize("rows", [700, 6000])
@pytest.mark.parametrize("kind", ["cond3", "cond6", "cond7", "cond9", "graded", "dependent", "zero", "nothing-below"])
def test_conditioning(h, b, rows, kind):
    """First-order and full second factorisation, and every way into the column loop."""
    Y = panel(kind, rows, b, np.random.default_rng(rows + b))
    V, T = check(h, Y, "f64")
    if kind == "nothing-below":      # nothing to annihilate: H = I for every column, as in LAPACK
        assert not T.any()
        assert np.array_equal(V, np.eye(rows, b))


@pytest.mark.parametrize("b", [32, 64])
@pytest.mark.parametrize("rows", [100, 2049, 7001])
def test_single_precision(h, b, rows):
    check(h, panel("gauss", rows, b, np.random.default_rng(rows)), "f32")


@pytest.mark.parametrize("dtype", ["f64", "f32"])
@pytest.mark.parametrize("rows", [128, 129, 192, 200, 1000, 4097, 30000])
def test_two_halves(h, rows, dtype):
    """128 columns are two panels of 64 in double precision (in single the column loop does them): square, with a square
    second half, ragged ends, many slabs."""
    check(h, panel("gauss", rows, 128, np.random.default_rng(rows)), dtype)


@pytest.mark.parametrize("kind", ["cond6", "cond9", "dependent", "zero", "nothing-below"])
def test_two_halves_conditioning(h, kind):
    V, T = check(h, panel(kind, 1500, 128, np.random.default_rng(3)), "f64")
    if kind == "nothing-below":
        assert not T.any()
        assert np.array_equal(V, np.eye(1500, 128))


@pytest.mark.parametrize("zero", [0.0, -0.0])
@pytest.mark.parametrize("rows,b", [(500, 16), (9000, 64)])
def test_zero_first_pivot_keeps_its_sign(h, rows, b, zero):
    Y = panel("gauss", rows, b, np.random.default_rng(5))
    Y[0, 0] = zero
    check(h, Y, "f64")


def test_squares_that_overflow(h):
    """The column loop's sums of squares overflow too; all that is asked is that the call ends and the context lives."""
    rrf.rrf_panel_qr(h, torch.from_numpy(panel("huge", 900, 32, np.random.default_rng(1))).cuda())
    torch.cuda.synchronize()
    assert rrf.rrf_last_status(h) == rrf.RRF_OK and rrf.rrf_panel_path(h) == rrf.RRF_PATH_LOOP_Y
    check(h, panel("gauss", 900, 32, np.random.default_rng(2)), "f64")


@pytest.mark.parametrize("value", [1e160, np.inf, np.nan])
@pytest.mark.parametrize("rows,b", [(700, 16), (900, 32), (6000, 64)])
def test_last_column_overflows(h, rows, b, value):
    """Its sum of squares is not finite while its products with the others may be: the columns before it are what they are
    without it."""
    Y = panel("gauss", rows, b, np.random.default_rng(rows))
    if value == 1e160:
        Y[:, -1] *= value
    else:
        Y[rows - 2, -1] = value
    V, T = (t.cpu().numpy() for t in rrf.rrf_panel_qr(h, torch.from_numpy(Y).cuda()))
    assert rrf.rrf_last_status(h) == rrf.RRF_OK
    Vo, _, To, _ = orc.panel_qr(Y[:, :-1])
    cond = np.linalg.cond(Y[:, :-1])
    assert np.max(np.abs(V[:, :-1] - Vo)) <= 100.0 * 1.1e-16 * cond
    assert np.max(np.abs(T[:-1, :-1] - To)) <= 1000.0 * 1.1e-16 * cond * np.max(np.abs(To))


@pytest.mark.parametrize("b", [16, 32, 64])
@pytest.mark.parametrize("rows", [700, 6000])
@pytest.mark.parametrize("kind", ["gauss", "cond6"])
def test_repeats_itself(h, b, rows, kind):
    """Warps that factor a block in place, all lanes alike, keep their lanes apart: the same bits two hundred times."""
    Y = torch.from_numpy(panel(kind, rows, b, np.random.default_rng(rows))).cuda()
    V, T = rrf.rrf_panel_qr(h, Y)
    for _ in range(200):
        v, t = rrf.rrf_panel_qr(h, Y)
        assert torch.equal(v, V) and torch.equal(t, T)


def panel_at(h, Y, offset, fn="rrf_panel_qr"):
    """The call with a workspace that starts `offset` bytes past a 256-byte boundary: status, V, T."""
    lib, (rows, b) = rrf.load(), Y.shape
    dt = rrf.RRF_F64 if Y.dtype == torch.float64 else rrf.RRF_F32
    need = C.c_size_t()
    assert lib.rrf_panel_workspace_bytes(dt, rows, b, C.byref(need)) == rrf.RRF_OK
    ws = torch.empty(need.value + 256, dtype=torch.uint8, device="cuda")
    at = -ws.data_ptr() % 256 + offset
    V, T = torch.empty_like(Y), torch.empty((b, b), dtype=Y.dtype, device="cuda")
    s = getattr(lib, fn)(h, dt, rows, b, C.c_void_p(Y.data_ptr()), b, C.c_void_p(V.data_ptr()), b, C.c_void_p(T.data_ptr()), b,
                         C.c_void_p(ws.data_ptr() + at), need.value, None)
    torch.cuda.synchronize()
    assert rrf.rrf_last_status(h) == rrf.RRF_OK
    return s, V, T


@pytest.mark.parametrize("dtype", [torch.float64, torch.float32])
@pytest.mark.parametrize("rows,b", [(200, 32), (3000, 64), (9000, 64), (128, 128), (1500, 128), (30000, 128)])
def test_workspace_on_8_bytes(h, rows, b, dtype):
    """The same bits wherever the workspace starts, as long as a double can be stored there."""
    Y = torch.from_numpy(panel("gauss", rows, b, np.random.default_rng(rows))).cuda().to(dtype)
    want = panel_at(h, Y, 0)
    for offset in (8, 16, 120):
        got = panel_at(h, Y, offset)
        assert got[0] == want[0] == rrf.RRF_OK
        assert torch.equal(got[1], want[1]) and torch.equal(got[2], want[2])
    assert panel_at(h, Y, 4)[0] == rrf.RRF_ERR_WORKSPACE


def test_blocked_kernel_needs_a_workspace_on_16_bytes(h):
    """On 8 bytes the column loop takes its place; a panel too tall for that is refused."""
    Y = torch.from_numpy(panel("gauss", 2000, 64, np.random.default_rng(8))).cuda()
    for offset in (0, 8):
        s, V, T = panel_at(h, Y, offset, "rrf_panel_qr_blocked")
        assert s == rrf.RRF_OK
        Vo, _, To, _ = orc.panel_qr(Y.cpu().numpy())
        assert np.max(np.abs(V.cpu().numpy() - Vo)) <= 1e-12 and np.max(np.abs(T.cpu().numpy() - To)) <= 1e-12
    Y = torch.from_numpy(panel("gauss", 48000, 64, np.random.default_rng(9))).cuda()
    assert panel_at(h, Y, 0)[0] == rrf.RRF_OK
    assert panel_at(h, Y, 8)[0] == rrf.RRF_ERR_WORKSPACE


def test_reciprocals(h):
    """The factorisations' own 1/x and 1/sqrt(x) over the exponents that their pivots can have (a pivot is at least 1e-11 of
    a diagonal entry between 1e-280 and 1e280): the third-order step leaves the approximation's error cubed, 2^-60, and two
    roundings of its own, so 1/x is within one and 1/sqrt(x) within two units in the last place of the rounded quotient."""
    rng = np.random.default_rng(0)
    n = 1 << 20
    x = np.ldexp(1.0 + rng.random(n), rng.integers(-968, 931, n))
    edge = np.ldexp(1.0, np.arange(-968, 931)).astype(np.float64)
    x = np.concatenate([x, edge, np.nextafter(edge, 0.0), np.nextafter(edge, np.inf), 1.0 + np.arange(1, 4097) / 4096.0])
    rcp, rsq = (t.cpu().numpy() for t in rrf.rrf_selftest_arithmetic(h, 1, torch.from_numpy(x).cuda()))
    exact = np.longdouble(1.0) / x.astype(np.longdouble)
    ulp = np.spacing(exact.astype(np.float64)).astype(np.longdouble)
    assert np.max(np.abs(rcp - exact) / ulp) <= 1.0
    exact = np.longdouble(1.0) / np.sqrt(x.astype(np.longdouble))
    ulp = np.spacing(exact.astype(np.float64)).astype(np.longdouble)
    assert np.max(np.abs(rsq - exact) / ulp) <= 2.0


@pytest.mark.parametrize("b", [16, 32, 64, 128])
@pytest.mark.parametrize("rows", [700, 6000])      # one cluster, the whole grid; 128 columns: the second half of two
@pytest.mark.parametrize("kind,path", [
    ("gauss", rrf.RRF_PATH_FIRST_ORDER), ("graded", rrf.RRF_PATH_FIRST_ORDER), ("near", rrf.RRF_PATH_CHOLESKY),
    ("nearer", rrf.RRF_PATH_LOOP_Y), ("dependent", rrf.RRF_PATH_LOOP_Y), ("zero", rrf.RRF_PATH_LOOP_Y),
    ("huge", rrf.RRF_PATH_LOOP_Y), ("nothing-below", rrf.RRF_PATH_LOOP_Q1)])
def test_path_taken(h, b, rows, kind, path):
    """Which of its ways a panel goes."""
    if b == 128:                     # the columns that decide belong to the second half
        Y = np.concatenate([panel("gauss", rows, 64, np.random.default_rng(b)), panel(kind, rows, 64, np.random.default_rng(rows))], 1)
        if kind == "nothing-below":
            Y = panel(kind, rows, b, np.random.default_rng(rows))
    else:
        Y = panel(kind, rows, b, np.random.default_rng(rows + b))
    rrf.rrf_panel_qr(h, torch.from_numpy(Y).cuda())
    assert rrf.rrf_panel_path(h) == path


def test_panels_that_do_not_try(h):
    for rows, b, dtype in ((64, 64, torch.float64), (3000, 128, torch.float32), (30000, 128, torch.float32)):
        rrf.rrf_panel_qr(h, torch.randn((rows, b), dtype=dtype, device="cuda"))
        assert rrf.rrf_panel_path(h) == rrf.RRF_PATH_LOOP
