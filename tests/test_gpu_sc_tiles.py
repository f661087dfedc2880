"""The simple-cubic Ising sweep at the edges of its segments (16 sites) and
tiles: spins, labels and measurements of every sweep equal the graph oracle's
bit for bit, and the same lattice handed over as a bond list gives the same
chain."""
import numpy as np
import pytest

import oracle
import paper_1612_08312_gb300 as pyro
import workloads

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("L", [2, 3, 15, 16, 17, 18, 31, 32, 33, 48, 50])
@pytest.mark.parametrize("masks", [False, True])
def test_every_sweep(L, masks):
    rng = np.random.default_rng(L)
    site = bond = None
    if masks:
        site = (rng.random(L ** 3) < 0.85).astype(np.uint8)
        bond = (rng.random(3 * L ** 3) < 0.9).astype(np.uint8)
    beta = 1 / (4.511524 if not masks else 3.4)
    bi, bj = oracle.sc_edges(L)
    g = pyro.Graph(pyro.ISING, 3 * L + 1, sc_L=L, start="random", site_mask=site, bond_mask=bond)
    o = oracle.GraphOracle(L ** 3, bi, bj, oracle.ISING, 3 * L + 1, "random", site_mask=site, edge_mask=bond)
    assert (g.labels() == np.arange(L ** 3)).all()
    assert (g.spins() == o.spins()).all()
    for _ in range(3):
        g.sweep(beta)
        o.sweep(beta)
        assert (g.spins() == o.spins()).all()
        assert (g.labels() == o.labels()).all()
        assert g.measure() == o.measure()
    assert g.stats() == o.stats()
    s = workloads.random_ising(L ** 3, L)
    g.set_spins(s)
    assert (g.spins() == s).all()
    g.close()


@pytest.mark.parametrize("L", [20, 64, 90])
def test_equals_the_bond_list(L):
    bi, bj = oracle.sc_edges(L)
    a = pyro.Graph(pyro.ISING, 5, sc_L=L, start="random")
    b = pyro.Graph(pyro.ISING, 5, nsites=L ** 3, bond_i=bi, bond_j=bj, start="random")
    for beta in (0.0, 0.2216, 0.3, 50.0):
        a.sweep(beta, 2)
        b.sweep(beta, 2)
        assert (a.spins() == b.spins()).all()
        assert (a.labels() == b.labels()).all()
    assert a.stats() == b.stats()
    a.close()
    b.close()
