"""FP64 calls whose contractions run on the tensor cores (gemm_digits.cu) report
a pipeline wait that ran out, and work again afterwards (the hook makes the
drain warps of the next tensor-core contraction wait 1 ms on a barrier that
nothing arrives at)."""
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


def _ctx(native, chi=64):
    g = native.TTN(4, 4, chi)
    g.set_hamiltonian(W.square_lattice(4, 4), 20.0)
    g.apply_pulse(W.random_constant_schedule(16, 1))
    g.set_product_state(W.random_product_amps(16, 2))
    return g


CALLS = {
    "step": lambda n, g, h: g.step(0.02),
    "measure": lambda n, g, h: g.measure(0),
    "overlap": lambda n, g, h: g.overlap(h),
    "refresh": lambda n, g, h: g.refresh_envs(),
    "compress": lambda n, g, h: g.compress_into(_ctx(n, 16)),
    "contract": lambda n, g, h: n.contract_host(np.ones((600, 64)), np.ones((64, 400)), n.FP64),
    "qr": lambda n, g, h: n.selftest_qr(np.random.default_rng(0).normal(size=(2048, 48))),
}


@pytest.mark.parametrize("name", sorted(CALLS))
def test_call_reports_the_timeout(native, name):
    g, h = _ctx(native), _ctx(native)
    CALLS[name](native, g, h)
    native.inject(native.INJECT_TC_STALL, 1)
    with pytest.raises(native.TTNError) as e:
        CALLS[name](native, g, h)
    assert e.value.code == TIMEOUT
    native.inject(native.INJECT_NONE)
    g.set_product_state(W.random_product_amps(16, 2))
    CALLS[name](native, g, h)
    assert abs(g.norm() - 1.0) < 1e-9
    g.close()
    h.close()
