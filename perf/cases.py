"""The work that users of this framework have it do, as measurable cases.

A case is a dict of plain values.  Its "kind" says which public entry points
a pass calls:

  lattice  Lattice.sweep (one pyrochlore lattice in caller-owned device
           memory), with the pass's statistics if "stats" is true: the run
           loop of a single large or small system;
  noalloc  pyro_ising_sweep_noalloc: one sweep embedded in a program that
           owns all device memory, labels and measurement returned;
  batch    Replicas.reset_stats / sweep / stats_all: one bin of a finite-
           size-scaling run over several sizes and temperatures;
  graph    Graph.sweep, stats and spins: the generic-lattice path on the
           simple-cubic lattice, implicit or as an explicit bond list,
           optionally site-diluted.

Temperatures are the critical ones the workloads use; single lattices start
from a correlated configuration drawn from the seed, batches (whose starts
the library draws) are equilibrated for a few sweeps first.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_1612_08312_gb300 as pyro

ISING, XY, HEIS = 1, 2, 3
# critical temperatures: pyrochlore, simple cubic, and the site-diluted
# simple-cubic lattice of occupation 0.8 (scaled from the Ising one)
TC = {ISING: 4.21394, XY: 2.0285, HEIS: 1.31695}
TC_SC = {ISING: 4.511524, XY: 2.20182, HEIS: 1.4430}
TC_DIL = {ISING: 3.5, XY: 1.71, HEIS: 1.12}
EQ_SWEEPS = 20  # a batch's sweeps before the first timed bin


def listed():
    return [
        # one sweep of the smallest workload lattice: launch and latency bound
        dict(name="ising L8 sweep", kind="lattice", model=ISING, L=8, fp64=False, sweeps=1, stats=False),
        # a bin of the small sizes of a finite-size-scaling run
        dict(name="ising small-size bin", kind="batch", model=ISING, sizes="8,12,16", temps=4, fp64=False, sweeps=16),
        # a sweep inside a program that may not allocate
        dict(name="ising L24 noalloc", kind="noalloc", model=ISING, L=24),
        # an odd lattice size, in bins of four sweeps
        dict(name="ising L45 bin", kind="lattice", model=ISING, L=45, fp64=False, sweeps=4, stats=True),
        # the 48 replicas (six sizes, eight temperatures) of the batched workload
        dict(name="ising 48 replicas", kind="batch", model=ISING, sizes="16,24,32,48,64,96", temps=8, fp64=False,
             sweeps=2),
        # the headline lattice, sweep by sweep
        dict(name="ising L256 sweep", kind="lattice", model=ISING, L=256, fp64=False, sweeps=1, stats=False),
        # the XY workload, every sweep's observables read back
        dict(name="xy L64 fp32", kind="lattice", model=XY, L=64, fp64=False, sweeps=1, stats=True),
        # the large Heisenberg workload
        dict(name="heisenberg L128 fp32", kind="lattice", model=HEIS, L=128, fp64=False, sweeps=1, stats=True),
        # the full-precision form, on a size that is no power of two
        dict(name="heisenberg L50 fp64", kind="lattice", model=HEIS, L=50, fp64=True, sweeps=1, stats=True),
        # Heisenberg replicas of two sizes
        dict(name="heisenberg 16 replicas", kind="batch", model=HEIS, sizes="32,64", temps=8, fp64=False, sweeps=2),
        # the comparison lattice: four sweeps, then the configuration is saved
        dict(name="simple cubic L256", kind="graph", model=ISING, L=256, fp64=True, sweeps=4, bonds="implicit", p=1.0),
        # a diluted lattice handed over as a bond list
        dict(name="diluted list L128", kind="graph", model=ISING, L=128, fp64=True, sweeps=4, bonds="list", p=0.8),
    ]


def _loguniform(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["lattice", "lattice", "lattice", "batch", "graph", "noalloc"])
    if kind == "noalloc":
        return dict(kind=kind, model=ISING, L=_loguniform(rng, 3, 32))
    model = rng.choice([ISING, ISING, XY, HEIS])
    fp64 = model != ISING and rng.random() < 0.3
    if kind == "lattice":
        L = _loguniform(rng, 4, 192 if model == ISING else (64 if fp64 else 112))
        return dict(kind=kind, model=model, L=L, fp64=fp64, sweeps=rng.choice([1, 1, 2, 5]) if L < 64 else 1,
                    stats=rng.random() < 0.5)
    if kind == "batch":
        top = 80 if model == ISING else 40
        sizes = sorted({_loguniform(rng, 6, top) for _ in range(rng.choice([2, 3, 4]))})
        return dict(kind=kind, model=model, sizes=",".join(map(str, sizes)), temps=rng.choice([2, 3, 5, 8]), fp64=fp64,
                    sweeps=rng.choice([1, 2, 4, 33]) if max(sizes) < 24 else rng.choice([1, 2, 4]))
    bonds = rng.choice(["implicit", "implicit", "list"])
    L = _loguniform(rng, 6, 96 if bonds == "list" else (256 if model == ISING else 128))
    return dict(kind=kind, model=model, L=L, fp64=fp64 or model == ISING, sweeps=rng.choice([1, 2, 4]), bonds=bonds,
                p=rng.choice([1.0, 1.0, 0.8, 0.9]))


def _beta(case):
    if case["kind"] == "graph":
        return 1.0 / (TC_SC if case["p"] == 1.0 else TC_DIL)[case["model"]]
    return 1.0 / TC[case["model"]]


def _field(L, per_cell, nc, seed):
    """nc components over L^3 cells of per_cell sites, (L^3 per_cell, nc) float64
    on the GPU: a Gaussian field with a 1 / k^2 spectrum (the correlations of a
    critical system) plus as much independent noise on every site."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    k2 = sum(torch.minimum(a, L - a) ** 2 for a in torch.meshgrid(
        *[torch.arange(L, device="cuda", dtype=torch.float64)] * 3, indexing="ij"))
    k2[0, 0, 0] = 1.0
    out = torch.empty((L ** 3 * per_cell, nc), dtype=torch.float64, device="cuda")
    for c in range(nc):
        w = torch.randn((L, L, L), generator=g, device="cuda", dtype=torch.float64)
        s = torch.fft.ifftn(torch.fft.fftn(w) / k2.sqrt()).real.reshape(-1, 1)
        s = s / s.std().clamp_min(1e-12)
        n = torch.randn((L ** 3, per_cell), generator=g, device="cuda", dtype=torch.float32)
        out[:, c] = (s + 0.9 * n).reshape(-1)
    return out


def _start(case, seed):
    """The starting configuration: (N,) int8 of +-1 or (N, n) unit vectors whose
    components are float32 values, held in float64."""
    n = case["model"]
    v = _field(case["L"], 1 if case["kind"] == "graph" else 16, n, seed)
    if n == ISING:
        return torch.where(v[:, 0] < 0, -1, 1).to(torch.int8)
    return (v / v.norm(dim=1, keepdim=True)).float().double()


def _packed(s):
    """Ising spins as the library packs them: bit b of word c is 1 iff site 16 c + b is -1."""
    bits = (s.reshape(-1, 16) < 0).to(torch.int32) << torch.arange(16, device="cuda", dtype=torch.int32)
    return bits.sum(dim=1, dtype=torch.int32).to(torch.int16)


def _mask(case, seed):
    return (np.random.default_rng(seed).random(case["L"] ** 3) < case["p"]).astype(np.uint8)


def _sc_bonds(L):
    i = np.arange(L ** 3, dtype=np.int32)
    x, y, z = i % L, (i // L) % L, i // (L * L)
    nb = np.stack([i - x + (x + 1) % L, i + L * ((y + 1) % L - y), i + L * L * ((z + 1) % L - z)], axis=1)
    return np.repeat(i, 3), nb.reshape(-1).astype(np.int32)


class _State:
    """What a user's program holds: the handle and the buffers it is given."""

    def __init__(self, case):
        self.case, self.beta = case, _beta(case)


def prepare(case, seed):
    st = _State(case)
    L, model, kind = case.get("L"), case["model"], case["kind"]
    prec = pyro.FP64 if case.get("fp64") else pyro.FP32
    if kind == "batch":
        Ls, betas = _replicas(case)
        st.rep = pyro.Replicas(Ls, betas, model, precision=prec, start="random", seed=seed)
        st.rep.sweep(EQ_SWEEPS)
        st.rep.sync()
        return st
    s = _start(case, seed)
    if kind == "noalloc":
        st.spins, st.seed, st.sweep = _packed(s), seed, 0
        st.labels = torch.empty(16 * L ** 3, dtype=torch.int32, device="cuda")
        st.meas = torch.empty(4, dtype=torch.float64, device="cuda")
        torch.cuda.synchronize()
        return st
    if kind == "graph":
        kw = dict(sc_L=L)
        if case["bonds"] == "list":
            bi, bj = _sc_bonds(L)
            kw = dict(nsites=L ** 3, bond_i=bi, bond_j=bj)
        if case["p"] < 1.0:
            kw["site_mask"] = _mask(case, seed)
        st.graph = pyro.Graph(model, seed, precision=prec, **kw)
        st.graph.set_spins(s.cpu().numpy())
        # the saved configuration goes to pinned memory
        st.out = torch.empty(s.shape, dtype=s.dtype, pin_memory=True)
        return st
    nbytes = pyro.pyro_workspace_bytes(L, model, prec)
    ws = torch.empty(nbytes, dtype=torch.uint8, device="cuda")
    torch.cuda.synchronize()
    st.lat = pyro.Lattice(L, model, seed, precision=prec, workspace=ws.data_ptr(), workspace_bytes=nbytes)
    st.ws = ws
    state = _packed(s) if model == ISING else s.T.contiguous().to(torch.float64 if prec == pyro.FP64 else torch.float32)
    host = state.cpu()
    pyro.pyro_set_state(st.lat.h, host.data_ptr(), host.numel() * host.element_size())
    st.lat.sync()
    # the spins live in the caller's memory, 256 bytes after its start
    st.spins = ws[256:256 + host.numel() * host.element_size()].view(host.dtype).view(host.shape)
    return st


def _replicas(case):
    Ls = [int(x) for x in case["sizes"].split(",")]
    tc, k = TC[case["model"]], case["temps"]
    Ts = [tc * (1.0 + 0.012 * (q - (k - 1) / 2) / max(k - 1, 1)) for q in range(k)]
    return [L for L in Ls for _ in Ts], [1.0 / T for _ in Ls for T in Ts]


def _values(stats):
    """Per-sweep means' sums, without the count."""
    return [stats[k] for k in ("sum_E", "sum_E2", "sum_m2", "sum_m4", "sum_absm")]


def run(st):
    case, kind = st.case, st.case["kind"]
    if kind == "noalloc":
        pyro.pyro_ising_sweep_noalloc(st.spins.data_ptr(), st.spins.data_ptr(), st.labels.data_ptr(),
                                      st.meas.data_ptr(), case["L"], st.beta, st.seed, st.sweep)
        st.sweep += 1
        return {"spins": st.spins, "labels": st.labels, "meas": st.meas}
    if kind == "batch":
        st.rep.reset_stats()
        st.rep.sweep(case["sweeps"])
        return {"stats": np.array([_values(s) for s in st.rep.stats_all()])}
    if kind == "graph":
        st.graph.reset_stats()
        st.graph.sweep(st.beta, case["sweeps"])
        out = st.graph.spins(out=st.out.numpy())
        return {"spins": out, "stats": np.array(_values(st.graph.stats()))}
    if not case["stats"]:
        st.lat.sweep(st.beta, case["sweeps"])
        return {"spins": st.spins}
    st.lat.reset_stats()
    st.lat.sweep(st.beta, case["sweeps"])
    return {"spins": st.spins, "stats": np.array(_values(st.lat.stats()))}


def _sites(case):
    if case["kind"] == "batch":
        return sum(16 * L ** 3 for L in _replicas(case)[0])
    return case["L"] ** 3 * (1 if case["kind"] == "graph" else 16)


def work(case):
    """The spins read and written once a sweep (packed Ising bits, generic
    Ising bytes, n components), an explicit bond list read once a sweep, the
    labels where they are returned; three bonds a site: a random word's share
    (ten rounds of Philox serve sixteen bonds), the projections, the products
    and the exponentials."""
    n, N, k = case["model"], _sites(case), case.get("sweeps", 1)
    site = n * (8 if case.get("fp64") else 4) if n > 1 else (1 if case["kind"] == "graph" else 0.125)
    b = 2.0 * site * N * k
    if case["kind"] == "graph":
        b += (24.0 * N * k if case["bonds"] == "list" else 0) + site * N
    if case["kind"] == "noalloc":
        b += 4.0 * N
    flops = N * k * (3 * 5 + 3 * 2 + (0 if n == 1 else (2 * n - 1) + 3 * 4 + 3 * 2 * n + 3 * n))
    return {"bytes": b, "flops": float(flops)}


# ------------------------------------------------------------- 64-bit form --
_M32 = 0xFFFFFFFF


def _philox(j, sweep, tag, seed):
    """Philox4x32-10 (Salmon et al., SC'11) of the counters (j, sweep, tag): four
    int64 tensors of 32-bit words."""
    c = [j & _M32, (j >> 32) & _M32, torch.full_like(j, sweep & _M32), torch.full_like(j, tag)]
    k0, k1 = seed & _M32, (seed >> 32) & _M32
    for r in range(10):
        if r:
            k0, k1 = (k0 + 0x9E3779B9) & _M32, (k1 + 0xBB67AE85) & _M32
        a, b = c[0] * 0xD2511F53, c[2] * 0xCD9E8D57  # wrap modulo 2^64
        c = [((b >> 32) & _M32) ^ c[1] ^ k0, b & _M32, ((a >> 32) & _M32) ^ c[3] ^ k1, a & _M32]
    return c


def _axis(n, sweep, seed):
    """The sweep's reflection axis: rejection in the square, Marsaglia's vector for n = 3."""
    for t in range(256):
        w = _philox(torch.tensor([t], device="cuda"), sweep, 3, seed)
        u = [(int(w[k]) - (int(w[k]) >> 31 << 32)) * 2.0 ** -31 for k in (0, 1)]
        q = u[0] * u[0] + u[1] * u[1]
        if 0.0 < q < 1.0:
            if n == 2:
                return [u[0] / math.sqrt(q), u[1] / math.sqrt(q)]
            t = math.sqrt(1.0 - q)
            return [2.0 * u[0] * t, 2.0 * u[1] * t, 1.0 - 2.0 * q]
    return [1.0, 0.0, 0.0][:n]


def _pyro_bonds(L):
    """Both sites of the 48 L^3 pyrochlore bonds in the order of their ids."""
    c = torch.arange(L ** 3, device="cuda")
    x, y, z = c % L, (c // L) % L, c // (L * L)
    a = [(0, 0, 0), (0, 1, 1), (1, 0, 1), (1, 1, 0)]
    slots = [[(0, 1, 1), (1, 2, 1), (2, 3, 1), (0, 3, 1)], [(0, 2, 1), (1, 3, 1), (0, 2, 0), (1, 3, 0)],
             [(0, 1, 0), (1, 2, 0), (2, 3, 0), (0, 3, 0)]]

    def site(f, v, up):
        if up or v == 0:
            return 16 * c + 4 * f + v
        h = [int(a[f][d] == 0 and a[v][d] == 1) for d in range(3)]
        return 16 * ((x - h[0]) % L + L * ((y - h[1]) % L + L * ((z - h[2]) % L))) + 4 * (f ^ v) + v

    i = torch.empty((L ** 3, 48), dtype=torch.int64, device="cuda")
    j = torch.empty_like(i)
    for g in range(3):
        for f in range(4):
            for q in range(4):
                va, vb, up = slots[g][q]
                i[:, 16 * g + 4 * f + q] = site(f, va, up)
                j[:, 16 * g + 4 * f + q] = site(f, vb, up)
    return i.reshape(-1), j.reshape(-1)


def _clusters(N, i, j):
    """The smallest site of each site's cluster under the edges (i, j)."""
    lab = torch.arange(N, device="cuda")
    while True:
        a, b = lab[i], lab[j]
        live = a != b
        if not bool(live.any()):
            return lab
        a, b, i, j = a[live], b[live], i[live], j[live]
        lab.scatter_reduce_(0, torch.maximum(a, b), torch.minimum(a, b), "amin")
        while True:
            up = lab[lab]
            if bool((up == lab).all()):
                break
            lab = up


def _sweep64(s, i, j, ids, occ, n, beta, sweep, seed):
    """One sweep in 64 bits; the new spins and the clusters' labels."""
    N = s.shape[0]
    if n == 1:
        ok = s[i] == s[j]
        thr = torch.full((1,), math.floor(-math.expm1(-2.0 * beta) * 2.0 ** 32), dtype=torch.int64, device="cuda")
        thr = thr.expand(ids.shape[0])
    else:
        r = _axis(n, sweep, seed)
        p = sum(s[:, k] * r[k] for k in range(n))
        x = p[i] * p[j]
        ok = x > 0
        thr = torch.floor(-torch.expm1(-2.0 * beta * x) * 2.0 ** 32).clamp_min(0).to(torch.int64)
    i, j, ids, thr = i[ok], j[ok], ids[ok], thr[ok]
    w = torch.stack(_philox(torch.arange(int(ids.max()) // 16 + 1 if len(ids) else 1, device="cuda"), sweep, 1, seed), 1)
    top = (w.reshape(-1)[ids >> 2] >> (8 * (ids & 3))) & 0xFF
    on = top < (thr >> 24)
    tie = (top == (thr >> 24)).nonzero().reshape(-1)
    t = torch.stack(_philox(ids[tie] >> 2, sweep, 5, seed), 1)
    on[tie] = (t.gather(1, (ids[tie] & 3).reshape(-1, 1)).reshape(-1) & 0xFFFFFF) < (thr[tie] & 0xFFFFFF)
    lab = _clusters(N, i[on], j[on])
    f = torch.stack(_philox(torch.arange((N + 127) // 128, device="cuda"), sweep, 2, seed), 1).reshape(-1)
    flip = ((f[lab >> 5] >> (lab & 31)) & 1).bool() & occ
    if n == 1:
        return torch.where(flip, -s, s), lab
    new = s - 2.0 * p[:, None] * torch.tensor(r, dtype=torch.float64, device="cuda")
    new = new / new.norm(dim=1, keepdim=True)
    return torch.where(flip[:, None], new, s), lab


def _observables(s, i, j, occ):
    """E, M^2 / N_occ^2 and its square (J = 1), and M_x."""
    v = s.double().reshape(s.shape[0], -1)
    E = -sum(float((v[i, k] * v[j, k]).sum()) for k in range(v.shape[1]))
    M = (v * occ[:, None]).sum(0)
    m2 = float((M * M).sum()) / max(int(occ.sum()), 1) ** 2
    return E, m2, m2 * m2, float(M[0])


def exact(case, seed):
    kind, n, N = case["kind"], case["model"], _sites(case)
    if kind == "batch" or N > 40_000_000:
        return None
    s = _start(case, seed)
    occ = torch.ones(N, dtype=torch.bool, device="cuda")
    if kind == "graph":
        i, j = (torch.from_numpy(a).cuda().long() for a in _sc_bonds(case["L"]))
        if case["p"] < 1.0:
            occ = torch.from_numpy(_mask(case, seed)).cuda().bool()
    else:
        i, j = _pyro_bonds(case["L"])
    ids = torch.arange(i.shape[0], device="cuda")
    here = occ[i] & occ[j]
    i, j, ids = i[here], j[here], ids[here]
    sums = np.zeros(5)
    for k in range(case.get("sweeps", 1)):
        s, lab = _sweep64(s, i, j, ids, occ, n, _beta(case), k, seed)
        E, m2, m4, Mx = _observables(s, i, j, occ)
        sums += [E, E * E, m2, m4, math.sqrt(m2)]
    if kind == "noalloc":
        return {"spins": _packed(s), "labels": lab.int(), "meas": torch.tensor([E, m2, m4, Mx], dtype=torch.float64)}
    if kind == "graph":
        return {"spins": s.cpu().numpy(), "stats": sums}
    spins = _packed(s) if n == ISING else s.T.contiguous()
    return {"spins": spins, "stats": sums} if case["stats"] else {"spins": spins}
