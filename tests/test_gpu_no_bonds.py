"""Ising sweeps at beta = 0, where the labelling has a form of its own, between
sweeps with bonds: spins, labels, measurements and sums equal the oracle's bit
for bit, on tiles that divide L, reach past it and cover it."""
import pytest

import oracle
import paper_1612_08312_gb300 as pyro

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("L,tile", [(1, (0, 0, 0)), (5, (0, 0, 0)), (8, (0, 0, 0)), (8, (1, 1, 1)), (8, (2, 1, 1)),
                                    (16, (8, 8, 4)), (33, (0, 0, 0)), (40, (8, 8, 8))])
def test_sweeps_without_bonds(L, tile):
    g = pyro.Lattice(L, pyro.ISING, 6 + L, start="random", tile=tile)
    o = oracle.Oracle(L, pyro.ISING, 6 + L, "random")
    for beta in (0.0, 0.0, 0.2373, 0.0, 1e-12, 0.4, 0.0):
        g.sweep(beta)
        o.sweep(beta)
        assert (g.spins() == o.spins()).all()
        assert (g.labels() == o.labels()).all()
        assert g.measure() == o.measure()
    assert g.stats() == o.stats()
    g.close()
