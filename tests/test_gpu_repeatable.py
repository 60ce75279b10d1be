"""A step is a function of the state: the same state gives the same bits in a
fresh context, in one that has run other states before, and after save and
load."""
import os
import tempfile

import numpy as np
import pytest

from paper_2210_03763_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def native():
    import __graft_entry__ as g
    g.build()
    from paper_2210_03763_gb300 import native as nat
    return nat


def _ctx(native, prec, chi=48):
    g = native.TTN(4, 3, chi)
    g.set_precision(prec)
    g.set_hamiltonian(W.square_lattice(4, 3), 20.0)
    g.apply_pulse(W.cz_layer_workload(4, 3, 2.0 ** 1.5)[0])
    return g


def _product(g, seed):
    g.set_product_state(W.random_product_amps(g.N, seed))


def _entangled(g, seed, falloff):
    """Isometric nodes, a root whose spectrum falls from 1 to 10^-falloff."""
    rng = np.random.default_rng(seed)
    leaf, root = g.leaf_atoms(), g.num_nodes() - 1

    def normal(*s):
        return rng.normal(size=s) + 1j * rng.normal(size=s)

    for k in range(root + 1):
        (d0, d1, d2), ch = g.node_info(k)
        if k == root:
            n = min(d0, d1)
            U, V = np.linalg.qr(normal(d0, n))[0], np.linalg.qr(normal(d1, n))[0]
            X = ((U * 10.0 ** (-falloff * np.arange(n) / max(1, n - 1))) @ V.T)[:, :, None]
            X = X / np.linalg.norm(X)
        else:
            A = normal(d0, d1, d2)
            for u in (0, 1):
                if ch[u] < 0 and leaf[-ch[u] - 1] < 0:
                    A[(slice(None),) * u + (slice(1, None),)] = 0
            X = np.linalg.qr(A.reshape(d0 * d1, d2, order="F"))[0].reshape(d0, d1, d2, order="F")
        g.set_node(k, X)
    g.refresh_envs()


def _bits(g):
    return [g.get_node(k) for k in range(g.num_nodes())] + [g.measure(0), g.measure(2)]


def _same(a, b):
    return all(np.array_equal(x, y) for x, y in zip(a, b))


STATES = {"product": lambda g: _product(g, 3), "flat": lambda g: _entangled(g, 4, 0.5),
          "falling": lambda g: _entangled(g, 5, 6.0)}


@pytest.mark.parametrize("prec", ["FP64", "SPLIT_TF32X3"])
@pytest.mark.parametrize("before,state", [("product", "flat"), ("product", "falling"), ("falling", "product"),
                                          ("falling", "flat"), ("flat", "product")])
def test_used_context_steps_as_a_fresh_one(native, prec, before, state):
    p = getattr(native, prec)
    fresh, used = _ctx(native, p), _ctx(native, p)
    STATES[before](used)
    for _ in range(2):
        used.step(0.02)
    STATES[state](used)
    STATES[state](fresh)
    for _ in range(2):
        used.step(0.02)
        fresh.step(0.02)
        assert _same(_bits(used), _bits(fresh))
    used.close()
    fresh.close()


@pytest.mark.parametrize("state", ["product", "falling"])
def test_run_continues_after_save_and_load(native, state):
    g, h = _ctx(native, native.FP64), _ctx(native, native.FP64)
    STATES[state](g)
    for _ in range(3):
        g.step(0.02)
    with tempfile.TemporaryDirectory() as td:
        path = os.path.join(td, "s.ttn")
        g.save(path)
        h.load(path)
    for _ in range(2):
        g.step(0.02)
        h.step(0.02)
        assert _same(_bits(g), _bits(h))
    g.close()
    h.close()
