"""The kernels' normalisation against the plain quotient by the root, on the
GPU, bit for bit: squared lengths through the whole range of the short forms
and past it, components of every size, powers of two and their neighbours,
zeros and denormals."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

import paper_1612_08312_gb300 as pyro

pytestmark = pytest.mark.gpu
HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def probe(tmp_path_factory):
    so = str(tmp_path_factory.mktemp("probe") / "normalise_probe.so")
    b = pyro._build
    subprocess.check_call([b.nvcc(), *b.ARCH, *b.NVFLAGS, "-shared", "-o", so,
                           os.path.join(HERE, "helpers", "normalise_probe.cu"), "-lcudart"])
    lib = ctypes.CDLL(so)
    lib.probe_normalise.argtypes = [ctypes.c_int, ctypes.c_int, ctypes.c_void_p, ctypes.c_void_p, ctypes.c_void_p,
                                    ctypes.c_long]
    return lib


def vectors(nc, f, n, rng):
    """Unit vectors scaled to squared lengths of up to 1.2 times the short
    form's range of units in the last place from 1, some with a component that
    is zero, tiny, denormal, a power of two or next to one."""
    eps, span = (2.0 ** -23, 1024) if f == np.float32 else (2.0 ** -52, 128)
    v = rng.normal(size=(n, nc))
    kind = rng.integers(0, 8, n)
    small = np.choose(kind, [0.0, 1e-20, 1e-30, 3e-39, 5e-310, 2.0 ** -rng.integers(0, 30, n).astype(float), 1.0, 1.0])
    axis = rng.integers(0, nc, n)
    rows = np.arange(n)
    fixed = kind < 6
    v[rows[fixed], axis[fixed]] = 0.0
    rest = np.where(fixed, np.sqrt(np.maximum(1.0 - small ** 2, 0.0)), 1.0)
    v *= (rest / np.linalg.norm(v, axis=1))[:, None]
    v[rows[fixed], axis[fixed]] = small[fixed] * rng.choice([-1, 1], fixed.sum())
    v *= np.sqrt(1.0 + rng.uniform(-1.2, 1.2, n) * span * eps)[:, None]
    t = v.astype(f)
    near = (kind == 5) & (rng.random(n) < 0.6)
    away = rng.choice([-2, 2], n).astype(f)
    t[rows[near], axis[near]] = np.nextafter(t[rows[near], axis[near]], away[near])
    return t


@pytest.mark.parametrize("nc", [2, 3])
@pytest.mark.parametrize("bits", [32, 64])
def test_bits_of_the_normalisation(probe, nc, bits):
    import torch
    f, i = (np.float32, np.int32) if bits == 32 else (np.float64, np.int64)
    n = 1 << 21
    t = vectors(nc, f, n, np.random.default_rng(nc + bits))
    a = torch.from_numpy(t).cuda()
    fast, plain = torch.empty_like(a), torch.empty_like(a)
    torch.cuda.synchronize()
    assert probe.probe_normalise(nc, bits, a.data_ptr(), fast.data_ptr(), plain.data_ptr(), n) == 0
    x, y = fast.cpu().numpy(), plain.cpu().numpy()
    assert np.isfinite(y).all()
    differ = (x.view(i) != y.view(i)).any(axis=1)
    assert not differ.any(), f"{differ.sum()} of {n}, first {t[differ][0]!r}: {x[differ][0]!r} {y[differ][0]!r}"
    # the short form was taken, and left, by a good part of them
    q = (t.astype(np.float64) ** 2).sum(1)
    units = np.abs(q - 1) / (2.0 ** -23 if bits == 32 else 2.0 ** -52)
    assert (units < 100).sum() > n // 20 and (units > (1024 if bits == 32 else 128)).sum() > n // 20
