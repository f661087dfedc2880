"""Simple-cubic Ising sweeps whose tiles have more pairs to unite than the pair
list holds: low temperatures from an ordered start, on tiles that cover the
lattice, wrap, and reach past it.  Spins, labels, measurements and sums equal
the graph oracle's bit for bit."""
import numpy as np
import pytest

import oracle
import paper_1612_08312_gb300 as pyro

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("L", [2, 8, 15, 16, 17, 33, 66, 80])
@pytest.mark.parametrize("bonds", [1.0, 0.95])
def test_more_pairs_than_the_list_holds(L, bonds):
    rng = np.random.default_rng(L)
    mask = None if bonds == 1.0 else (rng.random(3 * L ** 3) < bonds).astype(np.uint8)
    bi, bj = oracle.sc_edges(L)
    g = pyro.Graph(pyro.ISING, 7 + L, sc_L=L, start="up", bond_mask=mask)
    o = oracle.GraphOracle(L ** 3, bi, bj, oracle.ISING, 7 + L, "up", edge_mask=mask)
    for beta in (1.0, 0.8, 1.3, 2.0, 40.0, 1.0):
        g.sweep(beta)
        o.sweep(beta)
        assert (g.spins() == o.spins()).all()
        assert (g.labels() == o.labels()).all()
        assert g.measure() == o.measure()
    assert g.stats() == o.stats()
    g.close()


def test_a_lowered_union_bound_is_reported_there_too():
    g = pyro.Graph(pyro.ISING, 5, sc_L=16, start="up")
    try:
        pyro.pyro_debug_set(pyro.DEBUG_UNITE_BOUND, 0)
        g.sweep(1.0)
        with pytest.raises(pyro.PyroError) as ei:
            g.stats()
        assert ei.value.code == pyro.E_NOCONVERGE
    finally:
        pyro.pyro_debug_set(pyro.DEBUG_UNITE_BOUND, 4096)
    g.close()
