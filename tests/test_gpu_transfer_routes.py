"""The two routes of the subspace transfer (through the small product of the bases, or M itself through all reflectors)
and form Q on the columns a block touches, against the oracle.

Tolerances: a transfer is a product of two matrices with orthonormal columns, so its error is a few units in the last
place of ||M|| per block applied: 1e-13 in double precision, 2e-5 in single (the plain bars of the apply tests).
"""
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


def basis(m, k, b, rng):
    V, T = np.zeros((m, k)), np.zeros((b, k))
    for r in range(0, k, b):
        V[r:, r:r + b], _, T[:, r:r + b], _ = orc.panel_qr(rng.standard_normal((m - r, b)))
    return V, T


def dev(x, dtype):
    return torch.from_numpy(np.ascontiguousarray(x.astype(dtype))).cuda()


@pytest.mark.parametrize("dtype", [np.float64, np.float32])
@pytest.mark.parametrize("m,b,k_old,k_new,n", [
    (300, 32, 64, 32, 64),        # 2 k_new columns: the general route
    (300, 32, 64, 32, 68),        # just beyond: the small product, column tiles with a remainder
    (517, 32, 32, 96, 400),       # more new blocks than old ones
    (700, 64, 192, 64, 1000),
    (260, 128, 128, 128, 516),
    (400, 32, 64, 32, 333),       # rows of M that do not start on 16 bytes: the general route
])
def test_transfer_routes(h, dtype, m, b, k_old, k_new, n):
    rng = np.random.default_rng(m + n)
    Vo, To = basis(m, k_old, b, rng)
    Vn, Tn = basis(m, k_new, b, rng)
    M = rng.standard_normal((k_old, n))
    got = rrf.rrf_subspace_transfer(h, dev(Vo, dtype), dev(To, dtype), k_old, dev(Vn, dtype), dev(Tn, dtype), k_new, b, dev(M, dtype))
    want = orc.subspace_transfer(Vo, To, Vn, Tn, b, M)
    tol = 1e-13 if dtype is np.float64 else 2e-5
    assert np.linalg.norm(got.double().cpu().numpy() - want) <= tol * np.linalg.norm(M)


@pytest.mark.parametrize("dtype", [np.float64, np.float32])
@pytest.mark.parametrize("m,b,k", [(200, 32, 32), (515, 32, 160), (900, 64, 256), (400, 128, 256)])
def test_form_q_on_the_columns_a_block_touches(h, dtype, m, b, k):
    V, T = basis(m, k, b, np.random.default_rng(m))
    q = rrf.rrf_form_q(h, dev(V, dtype), dev(T, dtype), b, k).double().cpu().numpy()
    tol = 1e-13 if dtype is np.float64 else 2e-5
    assert np.linalg.norm(q - orc.form_q(V, T, b)) <= tol * np.sqrt(k)
