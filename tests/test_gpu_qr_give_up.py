"""A block of the cooperative QR column loop whose bounded barrier wait runs out
at the last barrier leaves rows of Q unwritten while every other block
finishes: the call reports it, and the next one runs normally.  (The hook ends
the block at that place without any wait running out.)"""
import os
import tempfile

import numpy as np
import pytest

from paper_2210_03763_gb300 import workloads as W

pytestmark = pytest.mark.gpu
TIMEOUT = 6


@pytest.fixture()
def native():
    import __graft_entry__ as g
    g.build()
    from paper_2210_03763_gb300 import native as nat
    nat.inject(nat.INJECT_NONE)
    yield nat
    nat.inject(nat.INJECT_NONE)


@pytest.mark.parametrize("M,D", [(300, 20), (2000, 17), (100, 12)])
def test_qr_reports_a_block_that_gave_up(native, M, D):
    rng = np.random.default_rng(M)
    A = rng.normal(size=(M, D)) + 1j * rng.normal(size=(M, D))
    native.inject(native.INJECT_QR_GIVE_UP, 1)
    with pytest.raises(native.TTNError) as e:
        native.selftest_qr(A)
    assert e.value.code == TIMEOUT
    Q, R, nd, _ = native.selftest_qr(A)
    assert nd == 0 and np.max(abs(Q @ R - A)) < 1e-12 * np.max(abs(A)) * D


def test_step_reports_it_and_continues_after_a_reload(native):
    def ctx():
        g = native.TTN(3, 3, 16)
        g.set_hamiltonian(W.square_lattice(3, 3), 20.0)
        g.apply_pulse(W.random_constant_schedule(9, 1))
        g.set_product_state(W.random_product_amps(9, 2))
        return g

    g, ref = ctx(), ctx()
    with tempfile.TemporaryDirectory() as td:
        path = os.path.join(td, "s.ttn")
        g.step(0.02)
        g.save(path)
        native.inject(native.INJECT_QR_GIVE_UP, 1)
        with pytest.raises(native.TTNError) as e:
            g.step(0.02)
        assert e.value.code == TIMEOUT
        g.load(path)
        ref.load(path)
    g.step(0.02)
    ref.step(0.02)
    assert all(np.array_equal(g.get_node(k), ref.get_node(k)) for k in range(g.num_nodes()))
    g.close()
    ref.close()
