"""Stage kernels that march: several planes (2D: rows) a block, chunk lengths
that do not divide the grid, one block over all of it -- ring-buffer slots,
carried faces and prefetched rows past the first -- against the FP64 oracle.
M is one launch of the kernel under test; the super-step of three stages runs
on the caller's rows, the one of five on padded rows where the width is not a
multiple of four."""
import numpy as np
import pytest

from gpu_util import (F32_FLUX_TOL, F32_LIMITER_MAX, F32_STATE_MAX, F32_STATE_REL_L2, F64_TOL, host, norm_max, rel_l2,
                      rounded, torch_dev)
from oracle import Problem
from test_gpu_parity import _fields, rk  # noqa: F401  (fixture)

pytestmark = pytest.mark.gpu

SPITZ = dict(kappa_model="spitzer", kappa_par0=0.01, kappa_perp_ratio=1e-4)
PHYS = {
    "spitzer": SPITZ,
    "sat": dict(kappa_model="spitzer", kappa_par0=0.01, saturate=True, phi=0.3),
    "sat_upwind": dict(SPITZ, saturate=True, phi=0.05, sat_upwind=True),
    "mc": dict(SPITZ, limiter="mc"),
    "mc_sat": dict(SPITZ, saturate=True, phi=0.3, limiter="mc"),
}
# shape (z, y, x) or (y, x), boundary, chunk lengths
F32_3D = [((19, 11, 67), "periodic", (2, 5, 16)), ((19, 11, 67), "dirichlet", (2, 7, 19)),      # GEN, PAD
          ((23, 9, 130), "periodic", (7,)), ((23, 17, 41), "dirichlet", (5, 16)),
          ((19, 11, 68), "dirichlet", (2, 5, 16)), ((40, 8, 132), "dirichlet", (7, 40)),        # DIR
          ((21, 9, 68), "periodic", (2, 5, 16))]                                                 # periodic row pairs
F64_3D = [((19, 11, 37), "periodic", (2, 5, 19)), ((23, 17, 20), "dirichlet", (3, 7)), ((31, 33, 9), "periodic", (4, 31))]
TWO_D = [((57, 67), "periodic", (2, 5, 14)), ((57, 66), "dirichlet", (3, 8)), ((64, 61), "dirichlet", (7, 64)),
         ((45, 120), "periodic", (1, 4, 45)), ((45, 33), "dirichlet", (6,))]


def _cases():
    out = []
    for dtype, group in (("f32", F32_3D + TWO_D), ("f64", F64_3D + TWO_D)):
        for k, (shape, bc, chunks) in enumerate(group):
            for q, phys in enumerate(PHYS):
                out.append((dtype, shape, bc, chunks, phys, (k + q) % 2 == 0))
    return out


@pytest.mark.parametrize("dtype,shape,bc,chunks,phys,cubic", _cases())
def test_march_against_oracle(rk, orc, dtype, shape, bc, chunks, phys, cubic):  # noqa: F811
    import torch
    nd = len(shape)
    h = 1.0 / max(shape)
    prm = dict(PHYS[phys], bc=bc, bc_value=0.95, dx=(h,) * nd if cubic else tuple(h * f for f in (1.0, 1.1, 0.9)[:nd]))
    T, b = _fields(shape)
    P = Problem(shape, **prm)
    Td, bd = torch_dev(T, dtype), torch_dev(b, dtype)
    T, b = rounded(T, dtype), rounded(b, dtype)
    M_ref = orc.apply_M(P, T, b)
    dt = 3.5 * orc.dt_expl(P, T)
    ref = {3: orc.super_step(P, T, b, 0.5 * dt, 3)[0], 5: orc.super_step(P, T, b, dt, 5)[0]}
    plan = rk.Plan(shape, dtype, params=prm)
    limited = phys.startswith("mc")
    M = torch.empty_like(Td)
    for chunk in chunks:
        plan.set_variant(0, chunk)
        plan.apply_M(Td, bd, M)
        # a limited slope near a kink may take the other branch in FP32
        tol = F64_TOL if dtype == "f64" else (F32_LIMITER_MAX if limited else F32_FLUX_TOL)
        assert np.abs(host(M) - M_ref).max() < tol * np.abs(M_ref).max(), chunk
        for s, want in ref.items():
            X = Td.clone()
            plan.super_step_s((0.5 if s == 3 else 1.0) * dt, s, X, bd)
            got = host(X)
            if dtype == "f64":
                assert norm_max(got, want) < F64_TOL, (chunk, s)
            else:
                assert rel_l2(got, want) < F32_STATE_REL_L2, (chunk, s)
                assert norm_max(got, want) < (F32_LIMITER_MAX if limited else F32_STATE_MAX), (chunk, s)
    assert plan.check() == 0
