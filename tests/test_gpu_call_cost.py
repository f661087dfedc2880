"""A call of a few sweeps replays graphs: what it costs the host is a graph
launch a sweep, not every kernel's launch, so that one thread can drive several
small lattices.  Six launches a sweep take about ten times as long as one graph
launch; the bound is half."""
import time

import pytest

import oracle
import paper_1612_08312_gb300 as pyro

pytestmark = pytest.mark.gpu


def host_time(lattices, n):
    """Seconds of the enqueueing calls alone, best of ten, with little queued."""
    best = float("inf")
    for _ in range(10):
        t = time.perf_counter()
        for g in lattices:
            g.sweep(0.2373, n)
        best = min(best, time.perf_counter() - t)
        for g in lattices:
            g.sync()
    return best


@pytest.mark.parametrize("n", [2, 7, 31])
def test_calls_of_a_few_sweeps_replay_graphs(n):
    on = [pyro.Lattice(8, pyro.ISING, 1 + k, start="random") for k in range(4)]
    off = [pyro.Lattice(8, pyro.ISING, 1 + k, start="random") for k in range(4)]
    for g in off:
        g.set_graphs(False)
    host_time(on, n), host_time(off, n)  # captures, first launches
    assert host_time(on, n) < 0.5 * host_time(off, n)
    assert len({g.launches for g in on + off}) == 1  # the count is of kernels, either way
    o = oracle.Oracle(8, oracle.ISING, 2, "random")
    o.sweep(0.2373, 20 * n)
    for g in (on[1], off[1]):
        assert (g.spins() == o.spins()).all() and (g.labels() == o.labels()).all()
        assert g.stats() == o.stats()
    for g in on + off:
        g.close()
