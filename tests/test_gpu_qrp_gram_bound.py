"""The error bound by which the Gram form of tall FP32 unfoldings decides its pivots (qrp_gram.cu), against
matrices made for the largest error of S: a column with one large entry and 255 equal ones just above the
smallest that the slices hold exactly, all rounded the same way, beside a constant column.  After the
constant column, the pivot is one of two columns whose norms differ by less than that error."""
from fractions import Fraction

import numpy as np
import pytest

import oracle
from tests.test_gpu_qrp_gram import first_factor, matrix

pytestmark = pytest.mark.gpu


def near_tie(gap, sign):
    """A (512 x 8): column 0 constant in rows 0..255; column 1 in the same rows, 1 and 255 times x; column 2
    in the other rows, its squared norm (1 + gap) times what column 0 leaves of column 1's; the others
    small.  sign: x lies below (1) or above (-1) what it rounds to."""
    x = Fraction(2**23 - (3 if sign > 0 else 5), 2**32)  # halfway between multiples of 2^-31, to even
    A = np.zeros((512, 8))
    A[:256, 0] = 1.0
    A[0, 1], A[1:256, 1] = 1.0, float(x)
    d = 1 + 255 * x * x - (1 + 255 * x) ** 2 / 256
    want = d * (1 + Fraction(gap))
    rows = range(256, 512)
    left = want
    for r in rows:  # squares of FP32 numbers, each at most what is left
        v = np.float32(np.sqrt(float(left)))
        if Fraction(float(v)) ** 2 > left:
            v = np.nextafter(v, np.float32(0))
        A[r, 2] = v
        left -= Fraction(float(v)) ** 2
        if left < want / 2**50:
            break
    rng = np.random.default_rng(1)
    A[:, 3:] = rng.standard_normal((512, 5)) * np.array([0.3, 0.25, 0.2, 0.15, 0.1]) / np.sqrt(512)
    A = A.astype(np.float32)
    got = sum(Fraction(float(v)) ** 2 for v in A[:, 2])
    assert abs(got / d - 1 - Fraction(gap)) < Fraction(1, 2**46) and float(A[1, 1]) == float(x)
    return A


@pytest.mark.parametrize("sign", [1, -1])
@pytest.mark.parametrize("gap", [2.0**-34, -(2.0**-34), 2.0**-32, -(2.0**-32)])
def test_pivot_of_a_near_tie(gap, sign):
    A = near_tie(gap, sign)
    Y, Q = first_factor(A, 2, 4, 6)
    np.testing.assert_array_equal(Y, A)
    np.testing.assert_allclose(Q, oracle.qrp(A.astype(np.float64), 6).Q, atol=1e-6)


@pytest.mark.parametrize("m,a,b,k", [(40, 3, 5, 6), (1000, 16, 16, 16), (700, 16, 32, 16), (38_917, 5, 6, 10)])
def test_separated_pivots_are_decided(m, a, b, k, monkeypatch):
    """The bound is not so wide that ordinary matrices run the cluster form: Q is not that form's."""
    A = matrix(m, a * b, 7 * m + a)
    _, Q = first_factor(A, a, b, k)
    monkeypatch.setenv("TUCKER_QRP_FORM", "cluster")
    _, want = first_factor(A, a, b, k)
    assert not np.array_equal(Q, want)
    np.testing.assert_allclose(Q, want, atol=1e-5)


def test_given_up_before_s(monkeypatch):
    """Magnitudes outside the range: every block of S (three tiles, several ranges of rows) leaves as a whole,
    and the cluster form runs."""
    A = matrix(1000, 256, 2)
    A[500, 200] *= np.float32(2.0**60)
    _, Q = first_factor(A, 16, 16, 16)
    monkeypatch.setenv("TUCKER_QRP_FORM", "cluster")
    _, want = first_factor(A, 16, 16, 16)
    np.testing.assert_array_equal(Q, want)
