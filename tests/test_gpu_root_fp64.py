"""The square root of the FP64 column-march kernels against IEEE arithmetic.

Along x the field comes in groups a, a, c, c and b points along x.  A cell
between a face of zero difference and the face a | c has M = +-cx F(a | c), in
which every operation but the root is one rounded product (a fused
multiply-add with a zero addend rounds like the product): numpy gives the same
bits for the same root, so M tells which root the kernel took.

Bound: the kernel refines the hardware's reciprocal square root r by one
third-order step from t = x r, e = 1 - t r (exact but for its rounding, so
that the rounding of t drops out).  With |e| <= 2^-19 the remainder 5 e^3 / 16
is below 2^-58 of the root, 0.02 ulp, and the last addition rounds once:
0.52 ulp in all."""
from fractions import Fraction

import numpy as np
import pytest

from gpu_util import host
from test_gpu_parity import rk  # noqa: F401  (fixture)

pytestmark = pytest.mark.gpu

KAPPA0, DX = 0.01, 0.125
NK = -0.25 * KAPPA0 * (0.25 / DX)           # constant kappa; slopes in units of 1 / (4 dx)


def _upper_and_lower(rk, shape, a, c, b0, **phys):  # noqa: F811
    """M of the cells below and above the a | c faces, one per group."""
    import torch
    T = np.stack([a, a, c, c], axis=1).reshape(shape)
    b = np.zeros((len(shape),) + shape)
    b[0] = np.repeat(b0, 4).reshape(shape)
    plan = rk.Plan(shape, "f64", params=dict(kappa_par0=KAPPA0, dx=(DX,) * len(shape), **phys))
    Td = torch.from_numpy(T).cuda()
    M = torch.empty_like(Td)
    plan.apply_M(Td, torch.from_numpy(b).cuda(), M)
    got = host(M).reshape(-1, 4)
    return got[:, 1], got[:, 2]


@pytest.mark.parametrize("shape", [(512, 128), (8, 64, 128)])
def test_root_within_its_bound(rk, shape):  # noqa: F811
    """Temperatures from 2^-38 to 2^83, even and odd exponents."""
    rng = np.random.default_rng(3)
    n = int(np.prod(shape)) // 4
    scale = np.exp2(rng.integers(-60, 60, n).astype(np.float64))
    a = rng.integers(1 << 22, 1 << 23, n) * scale
    c = a + np.exp2(rng.integers(0, 20, n).astype(np.float64)) * scale
    lo, hi = _upper_and_lower(rk, shape, a, c, np.ones(n), kappa_model="spitzer")
    assert np.array_equal(lo, -hi)
    Ts, X = a + c, 4.0 * (4.0 * (c - a))
    nk = -0.25 * KAPPA0 * 0.17677669529663688110 * (0.25 / DX)      # -kappa0 2^-2.5 / 4
    cx = -nk * (1.0 / DX)
    root = np.sqrt(Ts)
    off = np.nonzero(lo != cx * (Ts * Ts * root * X))[0]
    assert len(off) <= n // 100
    for i in off:
        errs = []
        for q in (np.nextafter(root[i], np.inf), np.nextafter(root[i], 0.0)):
            if cx * (Ts[i] * Ts[i] * q * X[i]) == lo[i]:
                errs.append(abs((Fraction(q) ** 2 - Fraction(Ts[i])) / (2 * Fraction(q) * Fraction(np.spacing(q)))))
        assert errs and min(errs) <= Fraction(52, 100)


def test_root_at_the_ends_of_its_range(rk):  # noqa: F811
    """Saturated flux at constant kappa: F = T15 X / (sat |V| + T15) with
    |V| = root(X^2), T15 = Ts root(Ts).  b scales X, so X^2 runs from zero
    through the subnormal numbers, the smallest normal one and 1 up to
    infinity; the last groups have Ts < 0.  The roots differ by at most one ulp
    each, the sum is fused in the kernel, and quotient and products round once:
    8 ulp between the two."""
    ex = np.concatenate([np.arange(-1090.0, -1000.0, 0.5), np.arange(-1000.0, 1010.0, 10.0), np.arange(1010.0, 1040.0, 0.5)])
    n = 480
    b0 = np.exp2(np.resize(ex, n) / 4.0) * 0.5 * 1.1         # X = 4 (c - a) (2 b0)^2 and X^2 ~ 2^ex
    a, c = np.full(n, 1.0), np.full(n, 1.5)
    a[-4:], c[-4:] = -2.0, -1.0
    for phi in (0.3, 1e-160, 1e160):
        with np.errstate(all="ignore"):
            q0 = 5.0 * phi
            sat = -NK / (q0 * 0.35355339059327376220)
            Ts, Bn = a + c, b0 + b0
            X = Bn * (Bn * (4.0 * (c - a)))
            T15 = Ts * np.sqrt(Ts)
            want = -NK * (1.0 / DX) * (T15 * X / (sat * np.sqrt(X * X) + T15))
        lo, hi = _upper_and_lower(rk, (1, 4 * n), a, c, b0, kappa_model="const", saturate=True, phi=phi)
        good = np.isfinite(want)
        assert good.sum() > 300
        assert np.array_equal(np.isnan(lo), np.isnan(want)) and np.array_equal(np.isnan(hi), np.isnan(want))
        assert np.array_equal(lo[~good & ~np.isnan(want)], want[~good & ~np.isnan(want)])
        assert np.all(np.abs(lo[good] - want[good]) <= 8 * np.spacing(np.abs(want[good])))
        assert np.array_equal(lo[good], -hi[good])
