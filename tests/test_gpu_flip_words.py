"""Flip bits of a tile, 17 bits a cell, put together a warp at a time: tiles of
1 to 512 cells, so parts of a warp, one warp and several, on every model's
flip.  Ising bit for bit against the oracle, FP64 to 1e-12, as elsewhere."""
import numpy as np
import pytest

import oracle
import paper_1612_08312_gb300 as pyro

pytestmark = pytest.mark.gpu

TILES = [(1, 1, 1), (2, 1, 1), (2, 2, 1), (2, 2, 2), (4, 2, 2), (4, 4, 2), (4, 4, 4), (8, 4, 4), (8, 8, 4), (8, 8, 8)]


@pytest.mark.parametrize("tile", TILES)
@pytest.mark.parametrize("model", [pyro.ISING, pyro.XY, pyro.HEIS])
def test_flips_of_every_tile_size(model, tile):
    g = pyro.Lattice(8, model, 21, precision=pyro.FP64, start="random", tile=tile)
    o = oracle.Oracle(8, model, 21, "random")
    beta = {pyro.ISING: 1 / 4.2, pyro.XY: 1 / 2.0, pyro.HEIS: 1 / 1.3}[model]
    for _ in range(2):
        g.sweep(beta)
        o.sweep(beta)
        assert np.abs(g.spins() - o.spins()).max() <= (0 if model == pyro.ISING else 1e-12)
    g.close()
