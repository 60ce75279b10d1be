"""Which kernels the shapes of the contraction and QR tests run on, so that those
tests cannot pass on another path: digit products on the tensor cores for large
FP64 contractions (and none of their outputs left to FMA chains where the
operands are of one size), the direct kernel for small ones; panels for
well-conditioned matrices from 48 x 24 on, the column loop with fine rows where
columns are dependent, with 128 rows where they are nearly so."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def native():
    import __graft_entry__ as g
    g.build()
    from paper_2210_03763_gb300 import native as nat
    return nat


def _rand(m, n, seed):
    rng = np.random.default_rng(seed)
    return rng.uniform(-1, 1, (m, n)) + 1j * rng.uniform(-1, 1, (m, n))


@pytest.mark.parametrize("M,N,K", [(4096, 64, 64), (4097, 65, 65), (300, 300, 300), (129, 1000, 257), (64, 64, 4096),
                                   (81, 81, 10368), (2048, 33, 127), (16384, 128, 128), (100, 90, 5003),
                                   (1000, 16, 700), (600, 400, 64), (600, 400, 3000), (2048, 96, 200)])
def test_large_fp64_contractions_run_as_digits(native, M, N, K):
    native.contract_host(_rand(M, K, 1), _rand(K, N, 2), native.FP64)
    assert native.selftest_last_path() == ("f64_digits", 0)


@pytest.mark.parametrize("M,N,K", [(1, 1, 700), (9, 9, 9), (12, 12, 145), (64, 64, 64), (257, 130, 17), (1000, 9, 3)])
def test_small_fp64_contractions_run_direct(native, M, N, K):
    native.contract_host(_rand(M, K, 1), _rand(K, N, 2), native.FP64)
    assert native.selftest_last_path()[0] == "f64_direct"


def test_graded_outputs_are_left_to_fma_chains(native):
    A, B = _rand(600, 64, 1), _rand(64, 400, 2)
    g = 2.0 ** (-np.arange(64.0))
    native.contract_host(A * g, B / g[:, None], native.FP64)
    assert native.selftest_last_path() == ("f64_digits", 600 * 400)
    B[:, 0] /= g                    # one column only
    native.contract_host(A * g, B, native.FP64)
    assert native.selftest_last_path() == ("f64_digits", 600)


@pytest.mark.parametrize("M,D,path", [(600, 96, "qr_panels"), (2049, 65, "qr_panels"), (81, 81, "qr_panels"),
                                      (48, 24, "qr_panels"), (47, 24, "qr_columns"), (48, 23, "qr_columns"),
                                      (300, 20, "qr_columns")])
def test_qr_path(native, M, D, path):
    A = _rand(M, D, 3)
    native.selftest_qr(A)
    assert native.selftest_last_path()[0] == path
    B = A.copy()
    B[:, 9] = B[:, 1] + 1e-7 * B[:, 9]
    native.selftest_qr(B)
    assert native.selftest_last_path()[0] == "qr_columns"
    B[:, 7] = B[:, 0]
    native.selftest_qr(B)
    assert native.selftest_last_path()[0] == "qr_columns_fine"
