"""Host-side check of the n-vector bond shortcut's margin: q = 256 p - b, from
one fast exponential (relative error 2^-22) of the FP32-staged projections,
never contradicts the exact rule, w < floor(p 2^32) with top byte b of w.

The margin is 1e-3 for FP32 spins and 1e-3 + 4e-4 K2 for FP64 spins, whose
projections are staged in FP32 with an error of at most 3e-7 each."""
import numpy as np
import pytest

F = np.float32


@pytest.mark.parametrize("fp64", [False, True])
@pytest.mark.parametrize("K2", [0.3, 1.5186, 20.0, 2000.0])
def test_shortcut_never_contradicts_the_exact_rule(fp64, K2):
    rng = np.random.default_rng(int(K2 * 10) + fp64)
    margin = F(1e-3) + (F(4e-4) * F(K2) if fp64 else F(0))
    K2l = F(K2) * F(1.44269504)
    n = 200000
    b = rng.integers(0, 256, n)
    # products of projections: all of [-1, 1], and close to the bytes' edges
    edge = -np.log1p(-np.minimum(b + rng.integers(0, 2, n), 255) / 256.0) / K2
    x = np.where(rng.random(n) < 0.5, rng.uniform(-1, 1, n), edge + rng.normal(0, 3e-6, n))
    pa = rng.uniform(0.5, 1.0, n) if fp64 else rng.uniform(0.5, 1.0, n).astype(F)
    pb = np.clip(x / pa, -1, 1)
    if not fp64:
        pb = pb.astype(F)
    off = rng.uniform(-3e-7, 3e-7, (2, n)) if fp64 else np.zeros((2, n))
    fa, fb = (pa + off[0]).astype(F), (pb + off[1]).astype(F)
    # one fused multiply-add: 8 - y log2 e, so that the exponential is 256 exp(-y)
    arg = (8.0 - (fa * K2l).astype(np.float64) * fb.astype(np.float64)).astype(F)
    for err in (-1, 0, 1):
        with np.errstate(over="ignore"):
            e = (np.exp2(arg.astype(np.float64)) * (1 + err * 2.0 ** -22)).astype(F)
            q = -(e - (256 - b).astype(F))
        on, never = q > F(1) + margin, q < -margin
        if fp64:
            xs = pa * pb
            p = -np.expm1(-K2 * xs)
        else:
            xs = pa * pb  # float32 product
            p = (-np.expm1(-(F(K2) * xs).astype(np.float64))).astype(F).astype(np.float64)
            p = p * (1 + err * 2.0 ** -23)  # expm1f is within an ulp
        thr = np.where(xs > 0, np.floor(np.clip(p, 0, 1) * 2.0 ** 32), 0.0)
        assert (thr[on] >= (b[on] + 1) * 2.0 ** 24).all()
        assert (thr[never] <= b[never] * 2.0 ** 24).all()
        assert (on | never).any()
