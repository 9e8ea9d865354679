"""Face fluxes, the advection step and the time-step statistics on grids at the
edges of their kernels' choice -- rows shorter and longer than a tile, full and
part tiles, odd plane counts, walls -- against the FP64 oracle, and their time
on narrow grids."""
import numpy as np
import pytest

from gpu_util import F32_FLUX_TOL, F64_TOL, host, norm_max, rounded, torch_dev
from oracle import Problem
from test_gpu_parity import _fields, rk  # noqa: F401  (fixture)

pytestmark = pytest.mark.gpu

SPITZ = dict(kappa_model="spitzer", kappa_par0=0.01, kappa_perp_ratio=1e-4)
# (z, y, x).  On a chip of 152 SMs the rows of 7 and 4 cells are past the line
# from which FP32 takes one thread per cell; (41, 256, 256) has full tiles only
# and enough of them for the FP64 march.
SHAPES = [(1, 1, 1), (41, 256, 256), (5, 9, 33), (3, 7, 31), (9, 8, 8), (41, 280, 7), (11, 500, 4), (2, 3, 1)]


@pytest.mark.parametrize("bc", ["periodic", "dirichlet"])
@pytest.mark.parametrize("dtype", ["f32", "f64"])
@pytest.mark.parametrize("shape", SHAPES)
def test_flux_and_advect_against_oracle(rk, orc, shape, dtype, bc):  # noqa: F811
    import torch
    prm = dict(SPITZ, bc=bc, bc_value=0.95)
    P = Problem(shape, **prm)
    T, b = _fields(shape)
    rng = np.random.default_rng(5)
    u = rng.normal(size=(3,) + shape)
    T, b, u = rounded(T, dtype), rounded(b, dtype), rounded(u, dtype)
    plan = rk.Plan(shape, dtype, params=prm)
    Td, bd, ud = torch_dev(T, dtype), torch_dev(b, dtype), torch_dev(u, dtype)
    F = [torch.empty_like(Td) for _ in range(3)]
    plan.flux(Td, bd, *F)
    want = orc.flux(P, T, b)
    scale = max(np.abs(w).max() for w in want) or 1.0
    for got, w in zip(F, want):
        assert np.abs(host(got) - w).max() <= (F32_FLUX_TOL if dtype == "f32" else F64_TOL) * scale
    dt = orc.dt_hyp(P, u, 0.8)
    assert plan.dt_hyperbolic(ud, 0.8) == pytest.approx(dt, rel=1e-6 if dtype == "f32" else 1e-14)
    out = torch.empty_like(Td)
    plan.advect(dt, ud, Td, out)
    # a few roundings of numbers up to |T| + dt |div|
    assert norm_max(host(out), orc.advect(P, T, u, dt)) < (2e-6 if dtype == "f32" else 1e-14)


@pytest.mark.parametrize("dtype", ["f32", "f64"])
def test_dt_hyperbolic_reports_nan_and_reads_any_alignment(rk, dtype):  # noqa: F811
    """Cell counts and addresses that rule the 16-byte reads out; a NaN in the
    last cell of each component."""
    import torch
    dt_ = torch.float32 if dtype == "f32" else torch.float64
    for shape, skip in [((3, 5, 7), 0), ((4, 4, 4), 1), ((4, 4, 4), 0), ((40, 50, 33), 3)]:
        n = int(np.prod(shape))
        g = torch.Generator("cuda").manual_seed(2)
        u = torch.randn(3 * n + skip, generator=g, device="cuda", dtype=dt_)[skip:].view((3,) + shape)
        dx = (0.5, 0.25, 0.125)
        plan = rk.Plan(shape, dtype, params=dict(SPITZ, dx=dx))
        rate = sum(u[d].double().abs() / dx[d] for d in range(3)).max().item()
        assert plan.dt_hyperbolic(u, 0.8) == pytest.approx(0.8 / rate, rel=1e-6 if dtype == "f32" else 1e-14)
        for d in range(3):
            v = u.clone()
            v[d].view(-1)[-1] = float("nan")
            with pytest.raises(rk.RklError) as ei:
                plan.dt_hyperbolic(v, 0.8)
            assert ei.value.status == rk._lib.RKL_ERR_NONFINITE


def _best_us(call):
    import torch
    best = 1e300
    for _ in range(20):
        e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        e0.record()
        for _ in range(5):
            call()
        e1.record()
        torch.cuda.synchronize()
        best = min(best, e0.elapsed_time(e1) * 200.0)
    return best


@pytest.mark.parametrize("dtype", ["f32", "f64"])
def test_narrow_grids_cost_what_their_cells_cost(rk, dtype):  # noqa: F811
    """A million cells as 10^6 rows of one cell take at most three times (FP32:
    six) as long as 1000 rows of 1000; with one lane of 32 busy it was 14 to 30."""
    import torch
    us = {}
    for shape in [(1000, 1000, 1), (1, 1000, 1000)]:
        plan = rk.Plan(shape, dtype, params=SPITZ)
        dt_ = torch.float32 if dtype == "f32" else torch.float64
        T = 1.0 + 0.1 * torch.rand(shape, device="cuda", dtype=dt_)
        b = torch.rand((3,) + shape, device="cuda", dtype=dt_)
        out = [torch.empty_like(T) for _ in range(3)]
        us[shape[2]] = (_best_us(lambda: plan.flux(T, b, *out)), _best_us(lambda: plan.advect(1e-6, b, T, out[0])))
    # FP32: the marching kernels are about 3 times as fast per cell on wide grids
    limit = 6.0 if dtype == "f32" else 3.0
    for narrow, wide in zip(us[1], us[1000]):
        assert narrow < limit * wide, us
