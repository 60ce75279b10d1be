"""H_eff in FP64 on a tensor graded along one leg: the batched, strided and
accumulating contractions of a node, elements far below the tensor's largest
included.  At the root, where applying H_eff moves no gauge, from the product
state |0...0>, whose bond bases are unit vectors: its operators couple few
indices, so H_eff X is graded as X is.

Reference: by linearity the sum over the leg's index of H_eff applied to one
slice at a time, where no graded sum occurs.  Both sides have the error bound of
FMA chains, some 10^3 2^-53 of the sum of products' sizes; sum_k |y_k| is that
sum up to what cancels within a slice (block terms against pair terms, a factor
of 10^2 at most here): 1e-11 sum_k |y_k|."""
import numpy as np
import pytest

from paper_2210_03763_gb300 import workloads as W

pytestmark = pytest.mark.gpu
CHI = 200


@pytest.fixture(scope="module")
def ctx():
    import __graft_entry__ as ge
    ge.build()
    from paper_2210_03763_gb300 import native
    g = native.TTN(4, 4, CHI)
    g.set_hamiltonian(W.square_lattice(4, 4), 20.0)
    g.apply_pulse(W.random_constant_schedule(16, 1))
    g.set_product_state(np.tile([1.0, 0.0, 0.0], (16, 1)))
    yield g
    g.close()


@pytest.mark.parametrize("leg", [0, 1])
def test_heff_of_a_graded_tensor(ctx, leg):
    root = ctx.num_nodes() - 1
    d = ctx.node_info(root)[0]
    assert d == (CHI, CHI, 1)
    rng = np.random.default_rng(leg)
    shape = [1, 1, 1]
    shape[leg] = CHI
    X = (rng.normal(size=d) + 1j * rng.normal(size=d)) * (2.0 ** (-0.4 * np.arange(CHI))).reshape(shape)
    y = ctx.apply_heff(root, X)
    ref, size = np.zeros_like(y), np.zeros(d)
    for k in range(CHI):
        S = np.zeros_like(X)
        i = (slice(None),) * leg + (k,)
        S[i] = X[i]
        yk = ctx.apply_heff(root, S)
        ref += yk
        size += abs(yk)
    err = np.max(abs(y - ref) / size)
    assert err <= 1e-11, err
