"""The allocation-free sweep on lattices its tile does not divide, and on spin
arrays of any alignment: the measurement reads four cells at a time only where
L and the tile's rows are multiples of 4 and the array starts on 8 bytes, and
must give the same sums everywhere else.  Spins, labels and measurement are
the oracle's, bit for bit."""
import numpy as np
import pytest

import oracle
import paper_1612_08312_gb300 as pyro

pytestmark = pytest.mark.gpu


def packed(s):
    return ((s == -1).astype(np.uint16).reshape(-1, 16) << np.arange(16, dtype=np.uint16)).sum(1).astype(np.uint16)


@pytest.mark.parametrize("offset", [0, 1, 2, 3])  # cells of 2 bytes
@pytest.mark.parametrize("L", [1, 2, 4, 5, 8, 12, 20, 32])
def test_noalloc_sizes_and_alignment(L, offset):
    import torch
    o = oracle.Oracle(L, oracle.ISING, 5, "random")
    buf = torch.zeros(L ** 3 + 8, dtype=torch.int16, device="cuda")
    spins = buf[offset:offset + L ** 3]
    labels = torch.empty(16 * L ** 3, dtype=torch.int32, device="cuda")
    meas = torch.empty(4, dtype=torch.float64, device="cuda")
    spins.copy_(torch.from_numpy(packed(o.spins()).view(np.int16)))
    assert buf.data_ptr() % 8 == 0
    for sweep in range(2):
        pyro.pyro_ising_sweep_noalloc(spins.data_ptr(), spins.data_ptr(), labels.data_ptr(), meas.data_ptr(), L,
                                      1 / 4.2, 5, sweep, torch.cuda.current_stream().cuda_stream)
        o.sweep(1 / 4.2)
        assert (spins.cpu().numpy().view(np.uint16) == packed(o.spins())).all()
        assert (labels.cpu().numpy() == o.labels()).all()
        assert tuple(meas.cpu().tolist()[:3]) == o.measure()
    assert (buf[:offset] == 0).all() and (buf[offset + L ** 3:] == 0).all()


@pytest.mark.parametrize("L,tile", [(4, (4, 4, 4)), (4, (2, 2, 2)), (8, (8, 1, 1)), (16, (4, 8, 8)), (24, (8, 8, 4)),
                                    (32, (32, 2, 2)), (12, (1, 4, 4)),
                                    (16, (8, 8, 8)), (32, (2, 16, 16))])
def test_measurement_of_given_tiles(L, tile):
    g = pyro.Lattice(L, pyro.ISING, 8, start="random", tile=tile)
    o = oracle.Oracle(L, oracle.ISING, 8, "random")
    assert g.measure() == o.measure()
    g.sweep(1 / 4.2)
    o.sweep(1 / 4.2)
    assert g.measure() == o.measure()
    g.close()
