"""The tile a lattice reports is accepted back: by another lattice of the same
size, by its workspace size and by batches of that size, whether or not its
edges divide L."""
import pytest

import oracle
import paper_1612_08312_gb300 as pyro
import workloads

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("model", [pyro.ISING, pyro.HEIS])
@pytest.mark.parametrize("L", [3, 7, 9, 12, 16, 21])
def test_reported_tile(model, L):
    beta = 1 / workloads.TC[model]
    a = pyro.Lattice(L, model, 4, precision=pyro.FP64, start="random")
    tile = a.tile
    b = pyro.Lattice(L, model, 4, precision=pyro.FP64, start="random", tile=tile)
    c = pyro.Replicas([L], [beta], model, precision=pyro.FP64, start="random", seed=4, tile=tile)
    assert b.tile == tile
    assert pyro.pyro_workspace_bytes(L, model, precision=pyro.FP64, tile=tile) == \
        pyro.pyro_workspace_bytes(L, model, precision=pyro.FP64)
    o = oracle.Oracle(L, model, 4, "random")
    o.sweep(beta, 2)
    for g in (a, b):
        g.sweep(beta, 2)
        assert (g.labels() == o.labels()).all()
    d = pyro.Replicas([L] * 5, [beta] * 5, model, precision=pyro.FP64, start="random", seed=4, tile=tile)
    for g in (c, d):
        g.sweep(2)
        assert (g.spins(0) == a.spins()).all()
    for g in (a, b, c, d):
        g.close()


@pytest.mark.parametrize("tile", [(8, 8, 4), (2, 1, 1), (1, 4, 1)])
def test_other_tiles_must_divide(tile):
    assert pyro.Lattice(9, pyro.ISING, 3).tile != tile
    with pytest.raises(pyro.PyroError):
        pyro.Lattice(9, pyro.ISING, 3, tile=tile)
