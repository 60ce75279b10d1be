"""The gauge-move QR of large matrices by panels (qr_panel.cu) against the
oracle's column rule, through the C ABI: ragged last panels (48 = 32 + 16, 65 =
2 x 32 + 1), graded columns, and matrices on which the panel path has to give
up and leave the result to the column loop: a dependent column in the first
and in a later panel, a column nearly (1e-7) inside the span of the others.
Tolerances: those of the column loop's tests for well-conditioned matrices
(1e-11 of max|A| for R, 1e-10 for Q); Q of the nearly dependent column is
determined to 2^-53 / 1e-7, and 1e-8 is allowed there."""
import numpy as np
import pytest

from oracle import linalg as OL

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def native():
    import __graft_entry__ as g
    g.build()
    from paper_2210_03763_gb300 import native as nat
    return nat


def _cmat(m, n, seed):
    rng = np.random.default_rng(seed)
    return rng.normal(size=(m, n)) + 1j * rng.normal(size=(m, n))


def _check(native, A, expect_dep):
    Q, R, nd, _ = native.selftest_qr(A)
    Qo, Ro = OL.qr_complete(A, None)
    scale = np.max(abs(A))
    assert nd == expect_dep
    assert np.max(abs(R - Ro)) <= 1e-11 * scale
    assert np.max(abs(Q - Qo)) <= 1e-10
    assert np.max(abs(Q.conj().T @ Q - np.eye(A.shape[1]))) < 1e-12
    assert np.max(abs(Q @ R - A)) <= 1e-12 * scale * np.sqrt(A.shape[1])


@pytest.mark.parametrize("M,D", [(2048, 48), (2049, 65), (3000, 96), (4096, 64)])
def test_panels_match_the_column_rule(native, M, D):
    _check(native, _cmat(M, D, M + D), 0)


def test_graded_columns(native):
    A = _cmat(2500, 70, 1)
    A *= 10.0 ** (-5.0 * np.random.default_rng(2).random(70))
    _check(native, A, 0)


@pytest.mark.parametrize("col", [7, 50])
def test_dependent_column_falls_back(native, col):
    A = _cmat(2304, 64, 3)
    A[:, col] = A[:, 0] - 2j * A[:, col - 1]
    _check(native, A, 1)


def test_nearly_dependent_column_keeps_q_orthonormal(native):
    # the column's direction outside the span is only determined to 2^-53 / 1e-7, so Q and R are checked by what
    # has to hold for either path: orthonormal columns and the product
    A = _cmat(2304, 64, 4)
    A[:, 40] = A[:, 3] + 1e-7 * A[:, 40]
    Q, R, nd, _ = native.selftest_qr(A)
    assert nd == 0
    assert np.max(abs(Q.conj().T @ Q - np.eye(64))) < 1e-12
    assert np.max(abs(Q @ R - A)) <= 1e-12 * np.max(abs(A)) * 8
