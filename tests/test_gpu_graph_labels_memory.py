"""Labels of the simple-cubic Ising lattice need no device memory beyond what
the lattice holds since its creation: with every allocation failing they are
returned all the same, and the sweep after them runs."""
import numpy as np
import pytest

import oracle
import paper_1612_08312_gb300 as pyro

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("L", [5, 20, 40])
def test_labels_without_an_allocation(L):
    beta = 0.2216
    bi, bj = oracle.sc_edges(L)
    g = pyro.Graph(pyro.ISING, 3, sc_L=L, start="random")
    o = oracle.GraphOracle(L ** 3, bi, bj, oracle.ISING, 3, "random")
    g.sweep(beta)
    o.sweep(beta)
    try:
        pyro.pyro_debug_set(pyro.DEBUG_FAIL_ALLOCS, 1000)
        labels = g.labels()
        g.sweep(beta)
    finally:
        pyro.pyro_debug_set(pyro.DEBUG_FAIL_ALLOCS, 0)
    assert (labels == o.labels()).all()
    o.sweep(beta)
    assert (g.labels() == o.labels()).all()
    g.close()


def test_creation_fails_when_any_allocation_does():
    """One allocation more at creation: its failure is reported as the others'
    are, and nothing is left behind."""
    for k in range(1, 4):
        pyro.pyro_debug_set(pyro.DEBUG_FAIL_ALLOCS, k)
        try:
            with pytest.raises(pyro.PyroError):
                pyro.Graph(pyro.ISING, 3, sc_L=8, start="random")
        finally:
            pyro.pyro_debug_set(pyro.DEBUG_FAIL_ALLOCS, 0)
    pyro.Graph(pyro.ISING, 3, sc_L=8, start="random").close()
