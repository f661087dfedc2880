"""Tiles with an edge of more than 32 cells, along each axis: the crossing
pairs name their cell in the tile by its coordinates.  Spins and labels equal
the oracle's, Ising bit for bit, FP64 n-vectors to 1e-12."""
import numpy as np
import pytest

import oracle
import paper_1612_08312_gb300 as pyro
import workloads

pytestmark = pytest.mark.gpu


def run(model, L, tile, sweeps):
    g = pyro.Lattice(L, model, 12, precision=pyro.FP64, start="random", tile=tile)
    o = oracle.Oracle(L, model, 12, "random")
    beta = 1 / workloads.TC[model]
    for _ in range(sweeps):
        g.sweep(beta)
        o.sweep(beta)
        assert (g.labels() == o.labels()).all()
        assert np.abs(g.spins() - o.spins()).max() <= (0 if model == pyro.ISING else 1e-12)
    g.close()


@pytest.mark.parametrize("tile", [(64, 2, 2), (2, 64, 2), (2, 2, 64), (64, 8, 1), (1, 64, 8), (8, 1, 64), (64, 1, 1)])
def test_ising_l64(tile):
    run(pyro.ISING, 64, tile, 2)


@pytest.mark.parametrize("tile", [(128, 2, 2), (2, 128, 2), (1, 2, 128)])
def test_ising_l128(tile):
    run(pyro.ISING, 128, tile, 1)


@pytest.mark.parametrize("model", [pyro.XY, pyro.HEIS])
@pytest.mark.parametrize("tile", [(64, 2, 2), (1, 64, 2), (2, 1, 64)])
def test_fp64_l64(model, tile):
    run(model, 64, tile, 1)
