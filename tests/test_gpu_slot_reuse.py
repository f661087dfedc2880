"""The table of crossing clusters is reused from sweep to sweep and from call to
call without any clearing, so entries of an earlier, larger use must never be
read: sizes that change in the allocation-free call's one scratch array, and
temperatures that change the number of slots on one lattice.  Bit for bit
against the oracle."""
import numpy as np
import pytest

import oracle
import paper_1612_08312_gb300 as pyro

pytestmark = pytest.mark.gpu


def packed(s):
    return ((s == -1).astype(np.uint16).reshape(-1, 16) << np.arange(16, dtype=np.uint16)).sum(1).astype(np.uint16)


def test_sizes_alternate_in_one_scratch_array():
    import torch
    stream = torch.cuda.current_stream().cuda_stream
    for call, (L, beta) in enumerate([(32, 0.2373), (5, 0.2373), (16, 0.6), (32, 0.05), (12, 0.0), (32, 0.2373),
                                      (16, 0.2373), (31, 0.2), (8, 0.2373), (17, 0.2373), (32, 0.2373)]):
        o = oracle.Oracle(L, oracle.ISING, 3 + call, "random")
        spins = torch.from_numpy(packed(o.spins()).view(np.int16)).cuda()
        labels = torch.empty(16 * L ** 3, dtype=torch.int32, device="cuda")
        meas = torch.empty(4, dtype=torch.float64, device="cuda")
        pyro.pyro_ising_sweep_noalloc(spins.data_ptr(), spins.data_ptr(), labels.data_ptr(), meas.data_ptr(), L, beta,
                                      3 + call, 0, stream)
        o.sweep(beta)
        assert (spins.cpu().numpy().view(np.uint16) == packed(o.spins())).all()
        assert (labels.cpu().numpy() == o.labels()).all()
        assert tuple(meas.cpu().tolist()[:3]) == o.measure()


BETAS = (0.02, 0.2373, 0.5, 0.02, 0.35, 0.0, 0.2373, 0.1, 0.6)


@pytest.mark.parametrize("L", [16, 21])
@pytest.mark.parametrize("model", [pyro.ISING, pyro.HEIS])
def test_temperatures_alternate_on_one_lattice(model, L):
    g = pyro.Lattice(L, model, 9, precision=pyro.FP64, start="random")
    o = oracle.Oracle(L, model, 9, "random")
    for beta in BETAS:
        beta *= 1 if model == pyro.ISING else 3
        g.sweep(beta)
        o.sweep(beta)
        assert (g.labels() == o.labels()).all()
        assert np.abs(g.spins() - o.spins()).max() <= (0 if model == pyro.ISING else 1e-12)
    g.close()


def test_temperatures_alternate_on_the_simple_cubic_lattice():
    L = 37
    bi, bj = oracle.sc_edges(L)
    g = pyro.Graph(pyro.ISING, 9, sc_L=L, start="random")
    o = oracle.GraphOracle(L ** 3, bi, bj, oracle.ISING, 9, "random")
    for beta in BETAS:
        g.sweep(beta)
        o.sweep(beta)
        assert (g.labels() == o.labels()).all() and (g.spins() == o.spins()).all()
    g.close()
