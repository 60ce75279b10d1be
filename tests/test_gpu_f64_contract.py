"""FP64 contractions against the host product in 64 bits, at the shapes where
the kernels change over: a single output, ragged K slices of the direct kernel
(fewer values than slices, K not a multiple), one output more than a block,
outputs at the direct / tiled border.  Tolerance: rounding of a K-term FP64
dot product in two summation orders, 1e-13 sqrt(K) of max|A B|."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def native():
    import __graft_entry__ as g
    g.build()
    from paper_2210_03763_gb300 import native as nat
    return nat


SHAPES = [(1, 1, 1), (1, 1, 700), (3, 3, 2), (9, 9, 9), (9, 729, 18), (12, 12, 145), (129, 1, 31), (64, 64, 64),
          (81, 5, 65), (257, 130, 17), (1000, 9, 3)]


def _check(native, M, N, K):
    rng = np.random.default_rng(M + 7 * N + 13 * K)
    A = rng.uniform(-1, 1, (M, K)) + 1j * rng.uniform(-1, 1, (M, K))
    B = rng.uniform(-1, 1, (K, N)) + 1j * rng.uniform(-1, 1, (K, N))
    ref = A @ B
    C, tc, _ = native.contract_host(A, B, native.FP64)
    assert not tc
    assert np.max(abs(C - ref)) <= 1e-13 * np.sqrt(K) * np.max(abs(ref))


@pytest.mark.parametrize("M,N,K", SHAPES)
def test_direct_contraction_vs_host_product(native, M, N, K):
    _check(native, M, N, K)
