"""The kernels of the automatic choice off the packed tiles' grids -- the
row-pair kernel's builds for any width and either boundary (FP32 3D), the
column-march kernels (FP64 3D, 2D) and the packed 2D kernel -- against the FP64 oracle at the edges of
their tiles: one cell, widths and heights one below, at and one above a tile,
odd widths, single planes; cubic and non-cubic cells, both boundaries,
saturated (both readings of c_iso) and MC-limited fluxes."""
import pytest

from gpu_util import F32_LIMITER_MAX, F32_STATE_MAX, F32_STATE_REL_L2, F64_TOL, host, norm_max, rel_l2, rounded, torch_dev
from oracle import Problem
from test_gpu_parity import _fields, rk  # noqa: F401  (fixture)

pytestmark = pytest.mark.gpu

SPITZ = dict(kappa_model="spitzer", kappa_par0=0.01, kappa_perp_ratio=1e-4)
PHYS = {
    "spitzer": SPITZ,
    "const": dict(kappa_par0=0.02, kappa_perp_ratio=0.1),
    "sat": dict(kappa_model="spitzer", kappa_par0=0.01, saturate=True, phi=0.3),
    "sat_const": dict(kappa_par0=0.02, kappa_perp_ratio=0.1, saturate=True, phi=0.003),
    "sat_upwind": dict(kappa_model="spitzer", kappa_par0=0.01, saturate=True, phi=0.05, sat_upwind=True),
    "mc": dict(SPITZ, limiter="mc"),
}
SHAPES_F32 = [(1, 1, 3), (2, 1, 1), (3, 9, 5), (5, 8, 63), (4, 7, 65), (20, 17, 66), (3, 16, 130), (9, 2, 129),
              (3, 1, 4), (5, 8, 64), (12, 9, 68), (4, 17, 128)]
SHAPES_F64 = [(1, 1, 1), (2, 1, 3), (3, 9, 5), (4, 33, 17), (20, 16, 31), (6, 8, 33), (3, 40, 9)]
SHAPES_2D = [(1, 1), (2, 3), (5, 30), (7, 31), (40, 32), (9, 62), (130, 63)]


def _cases():
    out = []
    for dtype, shapes in (("f32", SHAPES_F32 + SHAPES_2D), ("f64", SHAPES_F64 + SHAPES_2D)):
        for k, shape in enumerate(shapes):
            for q, phys in enumerate(PHYS):
                # boundaries and cell shapes alternate over shapes and physics
                for bc in (("periodic", "dirichlet") if k % 2 == 0 else (("periodic", "dirichlet")[q % 2],)):
                    out.append((dtype, shape, phys, bc, (k + q) % 3 != 0))
    return out


@pytest.mark.parametrize("dtype,shape,phys,bc,cubic", _cases())
def test_automatic_kernel_against_oracle(rk, orc, dtype, shape, phys, bc, cubic):  # noqa: F811
    nd = len(shape)
    h = 1.0 / max(shape)
    prm = dict(PHYS[phys], bc=bc, bc_value=0.95, dx=(h,) * nd if cubic else tuple(h * f for f in (1.0, 1.1, 0.9)[:nd]))
    T, b = _fields(shape)
    P = Problem(shape, **prm)
    Td, bd = torch_dev(T, dtype), torch_dev(b, dtype)
    T, b = rounded(T, dtype), rounded(b, dtype)
    plan = rk.Plan(shape, dtype, params=prm)
    dt = 20 * orc.dt_expl(P, T)
    for _ in range(2):
        s = plan.super_step(dt, Td, bd)
        T, sref = orc.super_step(P, T, b, dt)
        assert s == sref
    got = host(Td)
    assert plan.check() == 0
    if dtype == "f64":
        assert norm_max(got, T) < F64_TOL
    else:
        assert rel_l2(got, T) < F32_STATE_REL_L2
        assert norm_max(got, T) < (F32_LIMITER_MAX if phys == "mc" else F32_STATE_MAX)


@pytest.mark.parametrize("dtype,shape", [("f32", (5, 9, 67)), ("f64", (5, 9, 33)), ("f32", (9, 33)), ("f64", (9, 33))])
def test_bad_cells_are_reported(rk, dtype, shape):  # noqa: F811
    """A NaN in the last cell of an odd row and a stage that leaves T <= 0
    raise the status bits; the clean field raises none."""
    import torch
    T, b = _fields(shape)
    Td, bd = torch_dev(T, dtype), torch_dev(b, dtype)
    plan = rk.Plan(shape, dtype, params=dict(SPITZ, dx=(1.0 / max(shape),) * len(shape)))
    dt = 20 * plan.dt_expl(Td)
    plan.super_step_s(dt, 5, Td, bd)
    assert plan.check() == 0
    bad = Td.clone()
    bad.view(-1)[-1] = float("nan")
    plan.super_step_s(dt, 2, bad, bd)
    assert plan.check() == 3                     # RKL_ERR_NONFINITE
    neg = torch.ones_like(Td)
    neg.view(-1)[-1] = -1e-3
    plan.super_step_s(1e-9 * dt, 2, neg, torch.zeros_like(bd))
    assert plan.check() == 4                     # RKL_ERR_NONPOSITIVE_T


def test_new_ensemble_schedule_same_bits(rk):  # noqa: F811
    """The schedule an ensemble starts with (row-pair tiles, a tile length
    from its sizes) advances it to the bits of the paired-cell schedule."""
    import torch
    from test_gpu_ensemble import _build, _periodic_specs
    got = []
    for sched in (None, (1, 32)):
        ens, T_all, b_all, _, _, dts = _build(rk, _periodic_specs())
        if sched:
            ens.set_schedule(*sched)
        ens.super_step(dts, T_all, b_all)
        assert ens.check() == 0
        got.append(T_all.clone())
    assert torch.equal(got[0], got[1])
