"""FP64 contractions whose operands vary in size along K: small entries of one
operand that meet large ones of the other count in full, whatever else their
row holds.

Bound: that of an FP64 FMA chain, element by element.  The real part of a
complex dot product of K terms is a chain of 2 K real products, |error| <=
2 K 2^-53 sum |a_k||b_k| (and so is the imaginary one), so sqrt(2) 2 K 2^-53
sum |a_k||b_k| for the complex value."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def native():
    import __graft_entry__ as g
    g.build()
    from paper_2210_03763_gb300 import native as nat
    return nat


def _rand(M, N, K, seed):
    rng = np.random.default_rng(seed)
    return (rng.uniform(-1, 1, (M, K)) + 1j * rng.uniform(-1, 1, (M, K)),
            rng.uniform(-1, 1, (K, N)) + 1j * rng.uniform(-1, 1, (K, N)))


def _check(native, A, B, rows=37, cols=29):
    if np.finfo(np.longdouble).nmant < 60:
        pytest.skip("no extended precision on this host")
    C, _, _ = native.contract_host(A, B, native.FP64)
    m, n = slice(0, A.shape[0], max(1, A.shape[0] // rows)), slice(0, B.shape[1], max(1, B.shape[1] // cols))
    a, b, K = A[m], B[:, n], A.shape[1]
    ar, ai, br, bi = (np.asarray(x, dtype=np.longdouble) for x in (a.real, a.imag, b.real, b.imag))
    err = np.hypot(np.asarray(C[m, n].real - (ar @ br - ai @ bi), float),
                   np.asarray(C[m, n].imag - (ar @ bi + ai @ br), float))
    bound = np.sqrt(2) * 2 * K * 2.0 ** -53 * (abs(a) @ abs(b))
    assert np.all(err <= bound), float(np.max(err / np.where(bound > 0, bound, 1)))


SHAPES = [(600, 400, 64), (4097, 65, 65), (300, 300, 500), (64, 96, 4096), (97, 65, 9001)]


@pytest.mark.parametrize("M,N,K", SHAPES)
@pytest.mark.parametrize("bits", [32, 100])
def test_operands_graded_against_each_other(native, M, N, K, bits):
    A, B = _rand(M, N, K, 1)
    g = 2.0 ** (-bits * np.arange(K) / K)
    _check(native, A * g, B / g[:, None])


@pytest.mark.parametrize("M,N,K", SHAPES)
def test_each_row_and_column_graded_its_own_way(native, M, N, K):
    A, B = _rand(M, N, K, 2)
    rng = np.random.default_rng(3)
    _check(native, A * 2.0 ** (-60 * rng.random((M, K))), B * 2.0 ** (-60 * rng.random((K, N))))


def test_identity_with_noise_times_triangle(native):
    n = 300
    A, B = _rand(n, n, n, 4)
    _check(native, np.eye(n) + 1e-10 * A, np.triu(B))


@pytest.mark.parametrize("M,N,K", [(600, 400, 128), (97, 400, 9001)])
def test_sparse_operands_with_disjoint_supports(native, M, N, K):
    A, B = _rand(M, N, K, 5)
    A[:, ::2] = 0
    B[1::2] = 0
    B[1, 7::50] = 1e-30
    C, _, _ = native.contract_host(A, B, native.FP64)
    assert np.all(C[:, :7] == 0)
    _check(native, A, B)


def test_infinite_rows_next_to_graded_ones(native):
    A, B = _rand(600, 400, 64, 6)
    g = 2.0 ** (-np.arange(64.0))
    A, B = A * g, B / g[:, None]
    C0, _, _ = native.contract_host(A, B, native.FP64)
    A[70, 3] = np.inf
    B[5, 40] = np.nan
    C, _, _ = native.contract_host(A, B, native.FP64)
    mask = np.ones(C.shape, bool)
    mask[70], mask[:, 40] = False, False
    assert np.array_equal(C[mask], C0[mask])
    assert not np.any(np.isfinite(C[70].real)) and np.all(np.isnan(C[:, 40]))
