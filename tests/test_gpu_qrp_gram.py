"""QRP of a tall FP32 unfolding from its Gram matrix (qrp_gram.cu) inside hooi_iter.

A tensor of sizes (m, a, b) that holds a matrix A (m x ab) entry for entry, with identity factors in
modes 2 and 3 at full ranks a and b, has Y_(1) = A exactly, so U_1 after one sweep is the Q of A.

- Against the oracle's Q of the same FP32 entries in FP64: 1e-10, for matrices of condition below 100
  whose pivots are separated (Q comes from A_p R^-1 in double-float, 2^-44 times the condition, and the
  orthogonality correction is carried to third order of an error below 4e-6: 1e-16).
- Orthonormal to 1e-12.
- Where the Gram matrix cannot decide (ties, rank deficiency, magnitudes outside its range) the cluster
  form runs in its place: the same Q, bit for bit, as when that form is asked for by name.
- A captured sweep replays the same kernels: bit for bit, whichever form ran."""
import numpy as np
import pytest

import oracle
from tests.gpu_util import lib, torch

pytestmark = pytest.mark.gpu


def context(A, a, b, k, **kw):
    T = lib()
    m = A.shape[0]
    i, c = np.meshgrid(np.arange(m), np.arange(a * b), indexing="ij")
    coords = np.stack([i, c // b, c % b]).reshape(3, -1).astype(np.int32)
    rng = np.random.default_rng(0)
    U = [np.linalg.qr(rng.standard_normal((m, k)))[0], np.eye(a), np.eye(b)]
    return T.tucker_init((m, a, b), torch.as_tensor(coords).cuda(), torch.as_tensor(A.reshape(-1)).cuda(), (k, a, b),
                         [torch.as_tensor(u).cuda() for u in U], **kw)


def first_factor(A, a, b, k):
    T = lib()
    ctx = context(A, a, b, k)
    Y = T.ttmc_mode(ctx, 0).cpu().numpy()
    T.hooi_iter(ctx)
    Q = T.tucker_get_factor(ctx, 0).cpu().numpy()
    T.tucker_sync_status(ctx)
    T.tucker_free(ctx)
    return Y, Q


def matrix(m, n, seed):
    """Columns of norms a few percent apart, in random order, with a common direction."""
    rng = np.random.default_rng(seed)
    scale = 1.03 ** -rng.permutation(n) if n <= 64 else rng.uniform(0.5, 2.0, n)
    return ((rng.standard_normal((m, n)) + 0.5 * rng.standard_normal((m, 1))) * scale).astype(np.float32)


@pytest.mark.parametrize("m,a,b,k", [
    (40, 3, 5, 6),  # the fewest reflectors
    (60, 5, 6, 16),
    (128, 8, 16, 6),  # exact tiles, square
    (143, 11, 13, 7),  # just past the tile in both directions
    (255, 8, 8, 8),
    (257, 10, 13, 12),  # a block of rows with a single row
    (1000, 16, 16, 16),
    (700, 16, 32, 16),  # the most columns
    (2003, 11, 35, 13),
    (10_000, 8, 8, 8),  # ranges of rows that start in the middle of a block
    (38_917, 5, 6, 10),
    (2000, 8, 16, 4),  # tall and narrow: four and five reflectors
    (5731, 5, 25, 5),
])
def test_q_matches_oracle(m, a, b, k):
    A = matrix(m, a * b, 7 * m + a)
    Y, Q = first_factor(A, a, b, k)
    np.testing.assert_array_equal(Y, A)
    np.testing.assert_allclose(Q.T @ Q, np.eye(k), atol=1e-12)
    np.testing.assert_allclose(Q, oracle.qrp(A.astype(np.float64), k).Q, atol=1e-10)


@pytest.mark.parametrize("m,a,b,k", [
    (12, 3, 5, 6),  # the smallest, a single tile and block
    (31, 6, 6, 7),
    (33, 6, 8, 16),  # one past a tile and two blocks
    (64, 9, 9, 8),
    (200, 16, 16, 16),
    (257, 17, 16, 13),
    (512, 20, 26, 16),  # the largest
])
def test_fat_branch(m, a, b, k, monkeypatch):
    """m < ab: the QR of S = A A^T in FP64 (qrp_gram64.cu), against the cluster form on the same S:
    both are backward stable, so 2^-53 times the condition of S (below 1e4) times a few dozen."""
    A = matrix(a * b, m, 5 * m + a).T.copy()
    _, Q = first_factor(A, a, b, k)
    monkeypatch.setenv("TUCKER_QRP_FORM", "cluster")
    _, want = first_factor(A, a, b, k)
    np.testing.assert_allclose(Q.T @ Q, np.eye(k), atol=1e-13)
    np.testing.assert_allclose(Q, want, atol=1e-10)


@pytest.mark.parametrize("name", ["copies", "rank-deficient", "tiny", "huge"])
def test_fat_branch_undecided_runs_the_cluster_form(name, monkeypatch):
    A = matrix(120, 60, 9).T.copy()
    if name == "copies":
        A[30:] = A[:30]
    elif name == "rank-deficient":
        rng = np.random.default_rng(6)
        A = (rng.integers(-8, 9, (60, 5)) @ rng.integers(-8, 9, (5, 120))).astype(np.float32)
    else:  # entries of S below 2^-60, above 2^60
        A *= np.float32(2.0 ** (-34 if name == "tiny" else 28))
    _, Q = first_factor(A, 10, 12, 8)
    monkeypatch.setenv("TUCKER_QRP_FORM", "cluster")
    _, want = first_factor(A, 10, 12, 8)
    np.testing.assert_array_equal(Q, want)


@pytest.mark.parametrize("power", [-60, 60])
def test_fat_branch_magnitudes(power, monkeypatch):
    """S of entries near the ends of FP32's range, where their products leave it: a power of two
    changes nothing but S's exponents."""
    A = matrix(120, 60, 9).T.copy()
    _, Q = first_factor(A * np.float32(2.0**power), 10, 12, 8)
    monkeypatch.setenv("TUCKER_QRP_FORM", "cluster")
    _, want = first_factor(A, 10, 12, 8)
    np.testing.assert_allclose(Q, want, atol=1e-10)


def hard(name):
    rng = np.random.default_rng(5)
    A = matrix(600, 48, 3)
    if name == "tie":  # the two largest columns have the same entries in another order
        A[:, 11] = 8 * np.abs(A[:, 11])
        A[:, 30] = A[::-1, 11]
    elif name == "copies":
        A[:, 24:] = A[:, :24]
    elif name == "rank-deficient":
        A = (rng.integers(-8, 9, (600, 5)) @ rng.integers(-8, 9, (5, 48))).astype(np.float32)
    elif name == "large":
        A[:, 7] *= np.float32(2.0**60)
    elif name == "small":
        A[:, 7] *= np.float32(2.0**-70)
    elif name == "near-dependent":  # a condition of 1e6 within the pivots
        A[:, 6:] = A[:, :6] @ rng.standard_normal((6, 42)).astype(np.float32) + 1e-6 * A[:, 6:]
    elif name == "zero-column":
        A[:, 7] = 0
    return A


@pytest.mark.parametrize("name", ["tie", "copies", "rank-deficient", "large", "small", "near-dependent"])
def test_undecided_runs_the_cluster_form(name, monkeypatch):
    A = hard(name)
    _, Q = first_factor(A, 6, 8, 8)
    monkeypatch.setenv("TUCKER_QRP_FORM", "cluster")
    _, want = first_factor(A, 6, 8, 8)
    np.testing.assert_array_equal(Q, want)


def test_zero_column():
    A = hard("zero-column")
    _, Q = first_factor(A, 6, 8, 8)
    np.testing.assert_allclose(Q, oracle.qrp(A.astype(np.float64), 8).Q, atol=1e-10)


@pytest.mark.parametrize("name", ["plain", "tie"])
def test_captured(name):
    T = lib()
    A = hard(name)
    stream = torch.cuda.Stream()
    with torch.cuda.stream(stream):
        x, y = (context(A, 6, 8, 8, stream=stream) for _ in range(2))
        fits = [T.hooi_iter(x, stream=stream) for _ in range(3)]
        fit = torch.zeros(1, dtype=torch.float64, device="cuda")
        for i in range(3):
            T.tucker_hooi_graph(y, 1, fit, stream=stream)
            stream.synchronize()
            assert float(fit.item()) == fits[i]
        for n in range(3):
            assert torch.equal(T.tucker_get_factor(x, n), T.tucker_get_factor(y, n))
        T.tucker_sync_status(y, stream=stream)
        T.tucker_free(x)
        T.tucker_free(y)
