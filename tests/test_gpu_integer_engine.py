"""Double precision on the integer tensor cores (rrf_set_integer_engine) against the float64 oracle and against mma.sync."""
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


def _padded(x):
    rows, cols = x.shape
    t = torch.zeros((rows, cols + cols % 2), dtype=torch.float64, device="cuda")[:, :cols]
    t.copy_(torch.from_numpy(np.ascontiguousarray(x)))
    return t


def _problem(m, n, cap, scale, seed):
    rng = np.random.default_rng(seed)
    r = min(m, n, cap + 40)
    A = (rng.standard_normal((m, r)) * np.exp(-np.arange(r) / (0.4 * cap))) @ rng.standard_normal((r, n))
    if scale == "columns":           # every column its own power of two, forty apart at most
        A = A * np.exp2(rng.integers(-20, 21, n))
    elif scale == "rows":
        A = A * np.exp2(rng.integers(-6, 7, m))[:, None]
    elif scale == "huge":
        A = A * 2.0 ** 400
    elif scale == "tiny":
        A = A * 2.0 ** -400
    return A, rng.standard_normal((n, cap))


# tiles are 128 lines and 64 (32) indices, an update tile 128 x 32, a scale of V 1024 rows after the first b
@pytest.mark.parametrize("m,n,b,cap,scale", [
    (129, 65, 32, 64, "plain"), (160, 160, 32, 160, "plain"), (1057, 640, 32, 96, "plain"), (1089, 1025, 64, 192, "plain"),
    (2250, 333, 64, 256, "rows"), (700, 1301, 64, 192, "columns"), (515, 770, 64, 128, "huge"), (515, 770, 32, 96, "tiny"),
    (128, 200, 64, 128, "plain"), (300, 258, 128, 256, "plain"), (1281, 900, 128, 384, "columns"),
])
@pytest.mark.parametrize("sched", [rrf.RRF_FLAG_ONE_QUEUE, rrf.RRF_FLAG_TWO_QUEUES], ids=["one", "two"])
def test_run_matches_oracle(h, m, n, b, cap, scale, sched):
    A, Om = _problem(m, n, cap, scale, m + n)
    dA, dOm = _padded(A), _padded(Om.T)
    rrf.rrf_set_integer_engine(h, 1)
    try:
        g = [rrf.rrf_run(h, dA, b, 0.0, cap, omegaT=dOm, flags=sched | rrf.RRF_FLAG_FIXED_RANK) for _ in range(3)]
    finally:
        rrf.rrf_set_integer_engine(h, 2)
    o = orc.rrf(A, Om, b, 0.0, cap, fixed_rank=True)
    assert g[0].k == o.k == cap and g[0].fused_samples == 0
    for r in g[1:]:                                  # the call, its capture and its replay
        assert torch.equal(r.B[:cap], g[0].B[:cap]) and torch.equal(r.V[:, :cap], g[0].V[:, :cap])
    B = g[0].B[:cap].cpu().numpy()
    # The products of a block lose a few units of 2^-53 of the largest entry that shares a scale.  What becomes of that in the
    # blocks after it is the problem's condition, which the run on mma.sync shows: its rounding errors are of the same size
    # (columns forty powers of two apart make 3e-11 of them).
    rrf.rrf_set_integer_engine(h, 0)
    try:
        g0 = rrf.rrf_run(h, dA, b, 0.0, cap, omegaT=dOm, flags=sched | rrf.RRF_FLAG_FIXED_RANK)
    finally:
        rrf.rrf_set_integer_engine(h, 2)
    err, err0 = (np.linalg.norm(x - o.B, axis=0) / np.linalg.norm(o.B, axis=0) for x in (B, g0.B[:cap].cpu().numpy()))
    assert err.max() <= max(1e-12, 3.0 * err0.max()), (err.max(), err0.max())     # column by column, whatever its scale
    V0 = g[0].V[:, :b].cpu().numpy()
    assert np.linalg.norm(V0 - o.V[:, :b]) <= 1e-12 * np.linalg.norm(o.V[:, :b])
    assert abs(g[0].normA2 - np.sum(A * A)) <= 1e-12 * np.sum(A * A)


@pytest.mark.parametrize("m,n,b,cap", [(1100, 900, 64, 256), (700, 1000, 32, 128), (900, 1100, 128, 256)])
def test_variant_that_leaves_a_unchanged(h, m, n, b, cap):
    A, Om = _problem(m, n, cap, "plain", 5)
    dA, dOm = _padded(A), _padded(Om.T)
    out = []
    try:
        for engine in (0, 1):
            rrf.rrf_set_integer_engine(h, engine)
            out.append(rrf.rrf_run(h, dA, b, 1e-3, cap, omegaT=dOm, estimator=2, flags=rrf.RRF_FLAG_NO_UPDATE))
    finally:
        rrf.rrf_set_integer_engine(h, 2)
    a, c = out
    assert (a.k, a.status) == (c.k, c.status)
    assert float((a.V[:, :a.k] - c.V[:, :a.k]).norm()) <= 1e-11 * float(a.V[:, :a.k].norm())
    np.testing.assert_allclose(c.E_est_trace, a.E_est_trace, rtol=1e-11)


@pytest.mark.parametrize("m,n,b,k", [(128, 65, 32, 128), (1000, 770, 32, 96), (1153, 129, 64, 320), (900, 1090, 128, 384)])
@pytest.mark.parametrize("spike", [False, True])
def test_apply_qt_matches_oracle(h, m, n, b, k, spike):
    rng = np.random.default_rng(m)
    V, T = np.zeros((m, k)), np.zeros((b, k))
    for r in range(0, k, b):
        V[r:, r:r + b], _, T[:, r:r + b], _ = orc.panel_qr(rng.standard_normal((m - r, b)))
    C = rng.standard_normal((m, n)) * np.exp2(rng.integers(-30, 31, n))
    if spike:                                        # a column whose first rows dwarf the rest: gone from the scale after its block
        C[:b, ::3] *= 1e9
    ref = C.astype(np.longdouble)                    # in double the reference's own rounding is the larger part
    for r in range(0, k, b):
        v, t = V[r:, r:r + b].astype(np.longdouble), T[:, r:r + b].astype(np.longdouble)
        ref[r:] -= v @ (t.T @ (v.T @ ref[r:]))
    dV, dT = _padded(V), torch.from_numpy(T).cuda()
    out = []
    try:
        for engine in (0, 1):
            rrf.rrf_set_integer_engine(h, engine)
            out.append(rrf.rrf_apply_qt(h, dV, dT, b, k, _padded(C)).cpu().numpy())
    finally:
        rrf.rrf_set_integer_engine(h, 2)
    scale = np.linalg.norm(ref.astype(np.float64), axis=0)
    err = [np.linalg.norm((o - ref).astype(np.float64), axis=0) / scale for o in out]
    # an orthogonal transform in k / b <= 5 steps, each with a few 2^-53 of the column's norm; no worse than mma.sync as a whole
    assert err[1].max() <= 4e-15, (err[0].max(), err[1].max())
    assert np.sqrt(np.mean(err[1] ** 2)) <= 1.1 * np.sqrt(np.mean(err[0] ** 2))


def test_apply_qt_passes_on_what_is_not_finite(h):
    rng = np.random.default_rng(1)
    V, _, T, _ = orc.panel_qr(rng.standard_normal((500, 64)))
    C = rng.standard_normal((500, 300))
    C[400, 7], C[3, 200] = np.nan, np.inf
    rrf.rrf_set_integer_engine(h, 1)
    try:
        out = rrf.rrf_apply_qt(h, _padded(V), torch.from_numpy(T).cuda(), 64, 64, _padded(C)).cpu().numpy()
    finally:
        rrf.rrf_set_integer_engine(h, 2)
    assert not np.isfinite(out[:, [7, 200]]).any()
    assert np.isfinite(np.delete(out, [7, 200], axis=1)).all()


@pytest.mark.parametrize("bad", [np.nan, np.inf])
def test_non_finite_input_is_reported(h, bad):
    A, Om = _problem(700, 600, 128, "plain", 3)
    A[650, 599] = bad
    rrf.rrf_set_integer_engine(h, 1)
    try:
        g = rrf.rrf_run(h, _padded(A), 64, 0.0, 128, omegaT=_padded(Om.T), flags=rrf.RRF_FLAG_FIXED_RANK, check=False)
    finally:
        rrf.rrf_set_integer_engine(h, 2)
    assert g.status == rrf.RRF_ERR_NONFINITE


def test_workspace_without_the_digits_is_enough_for_the_other_path(h):
    m, n, b, cap = 1200, 1100, 64, 128
    A, Om = _problem(m, n, cap, "plain", 9)
    dA, dOm = _padded(A), _padded(Om.T)
    need = rrf.rrf_workspace_bytes(rrf.make_params(rrf.RRF_F64, m, n, b, 0.0, cap, flags=rrf.RRF_FLAG_FIXED_RANK))
    rrf.rrf_set_integer_engine(h, 1)
    try:
        ws = torch.empty(need - cap * n * 8 - 4096, dtype=torch.uint8, device="cuda")
        g = rrf.rrf_run(h, dA, b, 0.0, cap, omegaT=dOm, flags=rrf.RRF_FLAG_FIXED_RANK, workspace=ws)
    finally:
        rrf.rrf_set_integer_engine(h, 2)
    o = orc.rrf(A, Om, b, 0.0, cap, fixed_rank=True)
    assert np.linalg.norm(g.B[:cap].cpu().numpy() - o.B) <= 1e-12 * np.linalg.norm(o.B)


def test_engine_argument(h):
    with pytest.raises(rrf.RrfError):
        rrf.rrf_set_integer_engine(h, 3)
