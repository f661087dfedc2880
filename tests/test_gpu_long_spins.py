"""FP64 n-vectors of any length: a caller may set spins that are no unit
vectors, and their bonds are decided by the FP64 rule like any other's.  Here
every spin is long across the sweep's axis and short along it, so that an
approximation of the projections good for unit vectors only decides many bonds
otherwise.  Labels equal the oracle's; spins to 1e-12 of their length.  Set
through every way in: spins, state and the caller's own workspace."""
import ctypes

import numpy as np
import pytest

import oracle
import paper_1612_08312_gb300 as pyro

pytestmark = pytest.mark.gpu

LENGTH = 1e6


def long_spins(N, model, axis, seed):
    rng = np.random.default_rng(seed)
    along = rng.uniform(-1.2, 1.2, N)
    v = rng.normal(size=(N, model))
    v -= np.outer(v @ axis, axis)
    v *= LENGTH / np.linalg.norm(v, axis=1)[:, None]
    return v + np.outer(along, axis)


@pytest.mark.parametrize("model", [pyro.XY, pyro.HEIS])
@pytest.mark.parametrize("L,way", [(4, "spins"), (6, "spins"), (8, "spins"), (8, "state"), (8, "workspace")])
def test_bonds_of_long_spins(model, L, way):
    import torch

    seed, beta, ws = 31 + L, 0.8, None
    o = oracle.Oracle(L, model, seed, "up")
    o.sweep(beta)
    s = long_spins(o.N, model, o.axis(), L)
    o.sweep_count = 0
    o.set_spins(s)
    o.sweep(beta)
    kw = dict(precision=pyro.FP64, start="up")
    if way == "workspace":
        ws = torch.empty(pyro.pyro_workspace_bytes(L, model, precision=pyro.FP64), dtype=torch.uint8, device="cuda")
        kw.update(workspace=ws.data_ptr(), workspace_bytes=ws.numel())
    g = pyro.Lattice(L, model, seed, **kw)
    planes = np.ascontiguousarray(s.T)
    if way == "spins":
        g.set_spins(s)
    elif way == "state":
        assert pyro.lib().pyro_set_state(g.h, planes.ctypes.data_as(ctypes.c_void_p), planes.nbytes) == 0
        g.sync()
    else:
        ws[256:256 + planes.nbytes].copy_(torch.from_numpy(planes.view(np.uint8).reshape(-1)))
        torch.cuda.synchronize()
    assert (g.spins() == s).all()
    g.sweep(beta)
    assert (g.labels() == o.labels()).all()
    assert np.abs(g.spins() - o.spins()).max() <= 1e-12 * LENGTH
    # unit vectors beside them take the fast path in other tiles only
    o.sweep(beta)
    g.sweep(beta)
    assert (g.labels() == o.labels()).all()
    g.close()
