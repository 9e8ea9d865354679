"""Device memory of a plan whose width is not a multiple of four: the
row-padded copies of T and b come with the first super-step that uses them."""
import pytest

from test_gpu_parity import rk  # noqa: F401  (fixture)

pytestmark = pytest.mark.gpu


def test_padded_copies_are_allocated_on_use(rk):  # noqa: F811
    import torch
    shape = (200, 250, 255)                              # 51 MB an array
    array = 4 * 200 * 250 * 256                          # with padded rows
    params = dict(kappa_model="spitzer", kappa_par0=0.01, kappa_perp_ratio=1e-4)
    g = torch.Generator("cuda").manual_seed(1)
    T = 1.0 + 0.2 * torch.rand(shape, generator=g, device="cuda")
    b = torch.randn((3,) + shape, generator=g, device="cuda")
    b /= b.square().sum(0).sqrt()
    M = torch.empty_like(T)
    # everything that the library loads lazily is there before the first count
    warm = rk.Plan(shape, "f32", params=params)
    dt = 0.5 * warm.dt_expl(T)
    warm.apply_M(T, b, M)
    for s in (3, 6):
        warm.super_step_s(dt, s, T.clone(), b)
    assert warm.check() == 0
    warm.close()
    X = T.clone()
    torch.cuda.synchronize()

    def held(start):
        torch.cuda.synchronize()
        return start - torch.cuda.mem_get_info()[0]

    start = torch.cuda.mem_get_info()[0]
    plan = rk.Plan(shape, "f32", params=params)
    plan.apply_M(X, b, M)
    plan.super_step_s(dt, 3, X, b)
    assert held(start) < 4.5 * array
    plan.super_step_s(dt, 6, X, b)
    assert 7.5 * array < held(start) < 8.5 * array
    assert plan.check() == 0
    plan.close()
    assert held(start) < 0.5 * array
