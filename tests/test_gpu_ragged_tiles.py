"""Lattice sizes that the default labelling tile does not divide: the last
tile of an axis reaches past the lattice, and a tile longer than the lattice
wraps onto itself.  Every sweep is compared with the oracle: spins, labels and
measurements, Ising bit for bit and FP64 n-vectors to 1e-12."""
import numpy as np
import pytest

import oracle
import workloads

pytestmark = pytest.mark.gpu

pyro = pytest.importorskip("paper_1612_08312_gb300")


@pytest.mark.parametrize("L", [3, 5, 7, 9, 10, 13, 15, 17, 18, 23, 31, 33])
def test_ising_default_tile(L):
    g = pyro.Lattice(L, pyro.ISING, 40 + L, start="random")
    o = oracle.Oracle(L, oracle.ISING, 40 + L, "random")
    beta = 1 / workloads.TC[1]
    for _ in range(3):
        g.sweep(beta)
        o.sweep(beta)
        assert (g.spins() == o.spins()).all()
        assert (g.labels() == o.labels()).all()
        assert g.measure() == o.measure()
    assert g.stats() == o.stats()
    g.close()


@pytest.mark.parametrize("model", [pyro.XY, pyro.HEIS])
@pytest.mark.parametrize("L", [3, 5, 9, 11, 14, 17])
def test_fp64_default_tile(model, L):
    g = pyro.Lattice(L, model, 70 + L, precision=pyro.FP64, start="random")
    o = oracle.Oracle(L, model, 70 + L, "random")
    beta = 1 / workloads.TC[model]
    for _ in range(2):
        g.sweep(beta)
        o.sweep(beta)
        assert np.abs(g.spins() - o.spins()).max() <= 1e-12
        assert (g.labels() == o.labels()).all()
        assert np.allclose(g.measure(), o.measure(), rtol=1e-12, atol=0)
    g.close()


def test_fp32_energy_of_a_ragged_lattice():
    """FP32 measurement against a float64 sum over the same spins: a cell adds
    64 float32 terms, a relative error below 64 * 2^-24 < 4e-6 of the sum of
    magnitudes, which 3 N |J| bounds."""
    L = 11
    g = pyro.Lattice(L, pyro.HEIS, 9, start="random")
    g.sweep(1 / workloads.TC[3], 3)
    s = g.spins()
    o = oracle.Oracle(L, oracle.HEIS, 9, "random")
    o.set_spins(s)
    E, Eo = g.measure()[0], o.measure()[0]
    assert abs(E - Eo) <= 4e-6 * 3 * s.shape[0]
    g.close()


def test_batch_of_sizes_without_a_common_divisor():
    Ls = [5, 8, 9, 14]
    betas = [1 / 4.2, 1 / 4.21394, 1 / 4.23, 1 / 4.0]
    b = pyro.Replicas(Ls, betas, pyro.ISING, start="random", seed=6)
    b.sweep(34)  # a graph chunk and two single sweeps
    alls = b.stats_all()
    for r, L in enumerate(Ls):
        o = oracle.Oracle(L, oracle.ISING, pyro.replica_seed(6, r), "random")
        o.sweep(betas[r], 34)
        assert (b.spins(r) == o.spins()).all()
        assert alls[r] == o.stats()
    b.close()


def test_autotuned_tile_of_an_odd_size():
    """The autotuner's answer for a size no power of two divides is accepted
    back (zeros name the default tile), and other non-dividing tiles are not."""
    tile, ms = pyro.pyro_autotune(9, pyro.ISING, pyro.FP64, 0.2373, 2)
    assert ms > 0 and all(t == 0 or 9 % t == 0 for t in tile)
    g = pyro.Lattice(9, pyro.ISING, 3, start="random", tile=tile)
    o = oracle.Oracle(9, oracle.ISING, 3, "random")
    g.sweep(0.2373, 3)
    o.sweep(0.2373, 3)
    assert (g.spins() == o.spins()).all()
    with pytest.raises(pyro.PyroError):
        pyro.Lattice(9, pyro.ISING, 3, tile=(8, 8, 4))
    g.close()
