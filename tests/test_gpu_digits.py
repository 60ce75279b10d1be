"""FP64 contractions by digit products on the tensor cores (gemm_digits.cu)
against the host product, at shapes that the digit path takes.

* accuracy at the edges of tiles (128 rows, 32 complex columns), of K chunks
  (64 complex), ragged sizes, one-pass and two-pass packing (K <= 256), split K:
  1e-13 sqrt(K) of max|A B|, the bound of an FP64 dot product;
* the error against extended precision is no larger than an FP64 FMA chain's
  (0.3 x 2^-53 of |row||column|, derived below), for operands of one size and for rows and columns graded over 2^+-300;
* rows with an infinity or a NaN give what FP64 arithmetic gives, all other
  outputs are untouched by them; zero rows give exact zeros."""
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
    A = rng.uniform(-1, 1, (M, K)) + 1j * rng.uniform(-1, 1, (M, K))
    B = rng.uniform(-1, 1, (K, N)) + 1j * rng.uniform(-1, 1, (K, N))
    return A, B


SHAPES = [(4096, 64, 64), (4097, 65, 65), (300, 300, 300), (129, 1000, 257), (64, 64, 4096), (81, 81, 10368),
          (2048, 33, 127), (16384, 128, 128), (100, 90, 5003), (1000, 16, 700)]


@pytest.mark.parametrize("M,N,K", SHAPES)
def test_digit_contraction_vs_host_product(native, M, N, K):
    A, B = _rand(M, N, K, M + 7 * N + 13 * K)
    ref = A @ B
    C, _, _ = native.contract_host(A, B, native.FP64)
    assert np.max(abs(C - ref)) <= 1e-13 * np.sqrt(K) * np.max(abs(ref))


def _extended(A, B):
    """A @ B with the real products and sums in extended precision."""
    ar, ai, br, bi = (np.asarray(x, dtype=np.longdouble) for x in (A.real, A.imag, B.real, B.imag))
    return ar @ br - ai @ bi, ar @ bi + ai @ br


@pytest.mark.parametrize("K", [64, 500, 3000])
@pytest.mark.parametrize("graded", [False, True])
def test_digit_error_is_that_of_fp64_or_less(native, K, graded):
    if np.finfo(np.longdouble).nmant < 60:
        pytest.skip("no extended precision on this host")
    M, N = 600, 400
    A, B = _rand(M, N, K, 3)
    if graded:   # every row of A and column of B on its own scale
        rng = np.random.default_rng(4)
        A = A * 2.0 ** rng.integers(-300, 300, (M, 1))
        B = B * 2.0 ** rng.integers(-300, 300, (1, N))
    sub_m, sub_n = slice(0, 600, 29), slice(0, 400, 23)
    C, _, _ = native.contract_host(A, B, native.FP64)
    re, im = _extended(A[sub_m], B[:, sub_n])
    scale = np.sqrt(np.sum(abs(A[sub_m]) ** 2, 1))[:, None] * np.sqrt(np.sum(abs(B[:, sub_n]) ** 2, 0))[None]
    err = np.hypot(np.asarray((C[sub_m, sub_n].real - re) / scale, float), np.asarray((C[sub_m, sub_n].imag - im) / scale, float))
    # An FP64 FMA chain of 2 K real products of rms s: partial sums of rms sqrt(k) s, each rounded with rms
    # 0.3 x 2^-53 of its size, so 0.3 x 2^-53 s K sqrt(2) per part, 0.3 x 2^-53 of |a||b| for the complex value.
    assert np.sqrt(np.mean(err ** 2)) <= 0.3 * 2.0 ** -53


def test_infinities_nans_and_zero_rows(native):
    M, N, K = 2048, 96, 200
    A, B = _rand(M, N, K, 9)
    A[5] = 0
    B[:, 7] = 0
    C0, _, _ = native.contract_host(A, B, native.FP64)
    assert np.all(C0[5] == 0) and np.all(C0[:, 7] == 0)
    A1, B1 = A.copy(), B.copy()
    A1[1000, 3] = np.nan
    A1[70, 100] = np.inf
    B1[11, 40] = -np.inf
    C, _, _ = native.contract_host(A1, B1, native.FP64)
    mask = np.ones((M, N), bool)
    mask[[70, 1000]] = False
    mask[:, 40] = False
    assert np.array_equal(C[mask], C0[mask])
    assert np.all(np.isnan(C[1000].real) & np.isnan(C[1000].imag))
    # an infinity times ordinary numbers: infinite or NaN parts, never finite
    assert not np.any(np.isfinite(C[70].real)) and not np.any(np.isfinite(C[:, 40].imag))
