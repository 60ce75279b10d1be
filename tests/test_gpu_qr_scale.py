"""The gauge-move QR of well-conditioned matrices does not depend on the scale
of the matrix or of its columns (states lose norm under decay, tensors set by
the caller have any norm): every column is reproduced to a few 2^-53 of its own
norm.

Tolerance: R's entries are dot products with relative error below 2^-53 |q| |a|
each, so |Q R - a| takes sqrt(D) 2^-53 |a| from R, and as much again from the
rounding of Q's entries (sum over D columns of 2^-53 |R_kj|, |R_:j| = |a|); with
D <= 128, 2.5e-15 |a|.  The host's own product adds D 2^-53 at worst.  1e-14."""
import numpy as np
import pytest

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


def _check(native, A):
    Q, R, nd, _ = native.selftest_qr(A)
    assert nd == 0
    assert np.max(abs(Q.conj().T @ Q - np.eye(A.shape[1]))) < 1e-12
    assert np.all(np.tril(R, -1) == 0) and np.all(np.diag(R).imag == 0) and np.all(np.diag(R).real > 0)
    worst = np.max(np.linalg.norm(Q @ R - A, axis=0) / np.linalg.norm(A, axis=0))
    assert worst <= 1e-14, worst


@pytest.mark.parametrize("M,D", [(600, 96), (2049, 65), (4096, 128)])
@pytest.mark.parametrize("norm", [1.0, 1e-3, 1e-6, 1e-12, 1e8])
def test_scale_of_the_matrix(native, M, D, norm):
    A = _cmat(M, D, M + D)
    _check(native, A * (norm / np.linalg.norm(A)))


@pytest.mark.parametrize("order", ["random", "rising", "falling"])
def test_columns_on_their_own_scales(native, order):
    A = _cmat(1500, 96, 5)
    e = {"random": np.random.default_rng(6).random(96), "rising": np.linspace(1, 0, 96),
         "falling": np.linspace(0, 1, 96)}[order]
    _check(native, A * 10.0 ** (-6.0 * e))


@pytest.mark.parametrize("f", [1e-1, 1e-2, 1e-3])
@pytest.mark.parametrize("col,of", [(5, 3), (37, 36), (70, 3)])
def test_column_near_the_span_of_others(native, f, col, of):
    # the other columns have parts along the badly determined direction, and must not lose them
    A = _cmat(600, 96, 7)
    A[:, col] = A[:, of] + f * A[:, col]
    _check(native, A)
