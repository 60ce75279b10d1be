"""Outputs of split-precision contractions that are known exactly.

Entries are small integers times powers of two, so that every TF32 operand,
product and FP32 sum is exact and the result equals the host product bit for
bit: zeros, powers of two, both signs, sums with more than 24 bits between the
two float parts (the small columns), and scales whose results lie at the ends
of the FP32 exponent range, for both tile widths.  No tolerance.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def native():
    import __graft_entry__ as g
    g.build()
    from paper_2210_03763_gb300 import native as nat
    return nat


@pytest.mark.parametrize("M,N,K", [(64, 64, 16), (129, 70, 33), (300, 128, 512)])
@pytest.mark.parametrize("scale", [0, -80, -110, 100])
def test_exact_outputs(native, M, N, K, scale):
    rng = np.random.default_rng(M + K + 200 + scale)
    A = (rng.integers(-3, 4, (M, K)) + 1j * rng.integers(-3, 4, (M, K))) * 2.0 ** (scale // 2)
    B = (rng.integers(-3, 4, (K, N)) + 1j * rng.integers(-3, 4, (K, N))) * 2.0 ** (scale - scale // 2)
    B[:, 0] = 0.0
    A[:, 1:] *= rng.integers(0, 2, (M, 1))        # rows with one product: powers of two and zeros
    C, tc, _ = native.contract_host(A, B, native.SPLIT_TF32X3)
    assert tc
    assert np.array_equal(C, A @ B)


def test_wide_sums(native):
    # one term of 1 and one of 2^-20 .. 2^-40, in different chunks of K: the sum
    # needs up to 41 bits, more than the leading float has
    M, N, K = 64, 64, 128
    A = np.zeros((M, K), dtype=complex)
    B = np.zeros((K, N), dtype=complex)
    A[:, 0] = 1.0
    A[:, 100] = 2.0 ** -(20.0 + np.arange(M) % 21) * np.where(np.arange(M) % 2, -1.0, 1.0)
    B[0] = np.where(np.arange(N) % 3, 3.0, -5.0) + 1j
    B[100] = 1.0 - 3j
    C, tc, _ = native.contract_host(A, B, native.SPLIT_TF32X3)
    assert tc
    assert np.array_equal(C, A @ B)
