"""The matvec counter counts what ran.  A Krylov run launches as many steps as
its node took last time before it looks at a status, so the first short step
after a long one runs more products than the second."""
import pytest

from paper_2210_03763_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def test_matvecs_beyond_the_last_needed_step_are_counted():
    import __graft_entry__ as ge
    ge.build()
    from paper_2210_03763_gb300 import native
    g = native.TTN(3, 3, 16)
    g.set_hamiltonian(W.square_lattice(3, 3), 20.0)
    g.apply_pulse(W.random_constant_schedule(9, 1))
    g.set_product_state(W.random_product_amps(9, 2))
    g.step(0.2)
    counts = []
    for _ in range(2):
        g.reset_stats()
        g.step(1e-4)
        counts.append(g.stats()["matvecs"])
    assert counts[0] > counts[1] > 0
    g.close()
