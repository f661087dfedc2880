"""The simple-cubic Ising sweep at the largest edge the interface takes, 1,290:
bond ids pass 2^32, sites end just below 2^31 and the last segment of a row is
short.  No oracle holds this lattice, so outputs are checked on samples drawn
over the whole range and at its ends: the start, bonds and flips from cuRAND's
Philox in the documented layout, the labels' properties, and E and M recomputed
from the spins."""
import math

import numpy as np
import pytest

import paper_1612_08312_gb300 as pyro
import refmath

pytestmark = pytest.mark.gpu
BOND, FLIP, INIT, TIE = 1, 2, 4, 5  # stream tags


def bond_ends(L, e):
    i, d = e // 3, e % 3
    x, y, z = i % L, (i // L) % L, i // (L * L)
    return i, (x + (d == 0)) % L + L * ((y + (d == 1)) % L + L * ((z + (d == 2)) % L))


def energy_and_magnetisation(s, L):
    import torch
    t = torch.from_numpy(s).cuda().view(L, L, L)
    e = m = 0
    for z in range(0, L, 30):
        top = min(L, z + 30)
        a = t[z:top].to(torch.int32)
        up = t[torch.arange(z + 1, top + 1, device="cuda") % L].to(torch.int32)
        m += int(a.sum())
        e += int((a * torch.roll(a, -1, 2)).sum()) + int((a * torch.roll(a, -1, 1)).sum()) + int((a * up).sum())
    return -float(e), m


@pytest.mark.parametrize("L", [66, 1290])
def test_sampled_sweeps(L):
    if refmath.curand_philox_lib() is None:
        pytest.skip("nvcc not available to build the cuRAND host probe")
    N, seed = L ** 3, 5
    rng = np.random.default_rng(0)
    g = pyro.Graph(pyro.ISING, seed, sc_L=L, start="random")
    s0 = g.spins()
    i = np.concatenate([rng.integers(0, N, 200000), np.arange(N - 5000, N), np.arange(5000)])
    assert (s0[i] == np.where(refmath.stream_bits(seed, 0xFFFFFFFF, INIT, i) == 1, -1, 1)).all()
    for beta in (1 / 4.511524, 0.4):
        g.sweep(beta, 2)
        s0, k = g.spins(), g.sweep_count
        g.sweep(beta, 1)
        s1, lab = g.spins(), g.labels()
        for a in range(0, N, 1 << 27):
            b = min(N, a + (1 << 27))
            assert (lab[a:b] <= np.arange(a, b, dtype=np.int64)).all() and (lab[a:b] >= 0).all()
        j = np.concatenate([rng.integers(0, N, 1000000), np.arange(N - 100000, N)])
        assert (lab[lab[j]] == lab[j]).all()
        e = np.concatenate([rng.integers(0, 3 * N, 400000), np.arange(3 * N - 200000, 3 * N)])
        if 3 * N > (1 << 32) + 3 * L:
            e = np.concatenate([e, (1 << 32) + rng.integers(-3 * L, 3 * L, 50000)])
        bi, bj = bond_ends(L, e)
        w = (refmath.stream_bytes(seed, k, BOND, e).astype(np.int64) << 24) | \
            (refmath.stream_words(seed, k, TIE, e).astype(np.int64) & 0xFFFFFF)
        same = s0[bi] == s0[bj]
        active = same & (w < math.floor(-math.expm1(-2 * beta) * 2 ** 32))
        assert active.sum() > 100000
        assert (lab[bi[active]] == lab[bj[active]]).all() and (lab[bi[~same]] != lab[bj[~same]]).all()
        q = np.concatenate([rng.integers(0, N, 300000), np.arange(N - 100000, N)])
        flip = refmath.stream_bits(seed, k, FLIP, lab[q].astype(np.int64))
        assert (s1[q] == np.where(flip == 1, -s0[q], s0[q])).all()
        E, M = energy_and_magnetisation(s1, L)
        m = abs(M) / N
        assert g.measure() == (E, m * m, (m * m) * (m * m))
    g.close()
