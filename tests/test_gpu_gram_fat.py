"""S = Y_(n) Y_(n)^T of fat unfoldings (P_n > I_n) and the QRP of S inside hooi_iter, through tensors that
hold a matrix A entry for entry (identity factors in modes 2 and 3: Y_(1) = A)."""
import numpy as np
import pytest

import oracle
from tests.gpu_util import lib, torch

pytestmark = pytest.mark.gpu


def first_factor(A, a, b, k, scale=(1.0, 1.0)):
    """Y_(1), and U_1 after one sweep (scale: of the identities in modes 2 and 3)."""
    T = lib()
    m = A.shape[0]
    i, c = np.meshgrid(np.arange(m), np.arange(a * b), indexing="ij")
    coords = np.stack([i, c // b, c % b]).reshape(3, -1).astype(np.int32)
    U = [np.linalg.qr(np.random.default_rng(0).standard_normal((m, k)))[0], scale[0] * np.eye(a), scale[1] * np.eye(b)]
    ctx = T.tucker_init((m, a, b), torch.as_tensor(coords).cuda(), torch.as_tensor(A.reshape(-1)).cuda(), (k, a, b),
                        [torch.as_tensor(u).cuda() for u in U])
    Y = T.ttmc_mode(ctx, 0).cpu().numpy()
    T.hooi_iter(ctx)
    Q = T.tucker_get_factor(ctx, 0).cpu().numpy()
    T.tucker_free(ctx)
    return Y, Q


def fat(m, n, seed):
    """Rows of norms a few percent apart, in random order, with a common direction."""
    rng = np.random.default_rng(seed)
    scale = 1.03 ** -rng.permutation(m) if m <= 64 else rng.uniform(0.5, 2.0, m)
    return ((rng.standard_normal((m, n)) + 0.5 * rng.standard_normal((1, n))) * scale[:, None]).astype(np.float32)


@pytest.mark.parametrize("m,a,b", [(60, 10, 12), (1024, 33, 34), (1025, 33, 34)])
@pytest.mark.parametrize("row", [0, 37])
@pytest.mark.parametrize("what", ["inf", "nan"])
def test_overflowed_row_stays_visible(m, a, b, row, what):
    """A row of Y that overflows FP32 (from finite values and factors; a product of the last factor
    overflows to infinity, one of the factor before it also meets zeros of the last) makes the factor
    non-finite, on both sides of the sizes that the double-float kernel takes."""
    A = fat(m, a * b, m)
    A[row] = np.float32(3e38) * np.sign(A[row])
    Y, Q = first_factor(A, a, b, 8, scale=(1.0, 4.0) if what == "inf" else (4.0, 1.0))
    assert (np.isinf(Y[row]) if what == "inf" else np.isnan(Y[row])).all()
    assert np.isfinite(np.delete(Y, row, 0)).all()
    assert not np.isfinite(Q).all()


@pytest.mark.parametrize("m,a,b", [(1025, 33, 34), (1100, 33, 34)])
def test_above_1024_rows_in_fp64(m, a, b, monkeypatch):
    """More than 1,024 rows: S in FP64, as with TUCKER_CORE_TC=0, bit for bit."""
    A = fat(m, a * b, m)
    _, Q = first_factor(A, a, b, 8)
    monkeypatch.setenv("TUCKER_CORE_TC", "0")
    _, want = first_factor(A, a, b, 8)
    np.testing.assert_array_equal(Q, want)


@pytest.mark.parametrize("m,a,b,k", [(12, 3, 5, 6), (33, 6, 8, 16), (200, 16, 16, 16), (512, 20, 26, 16)])
def test_decided_pivots_run_the_gram_form(m, a, b, k, monkeypatch):
    """Where the pivots are decided Q is not the cluster form's (its roundings are others), and it is that
    of the FP64 reference: 2^-46 in S times its condition (below 1e4) times a few dozen."""
    A = fat(m, a * b, 5 * m + a)
    _, Q = first_factor(A, a, b, k)
    monkeypatch.setenv("TUCKER_QRP_FORM", "cluster")
    _, cluster = first_factor(A, a, b, k)
    assert not np.array_equal(Q, cluster)
    A = A.astype(np.float64)
    np.testing.assert_allclose(Q, oracle.qrp(A @ A.T, k).Q, atol=1e-8)
