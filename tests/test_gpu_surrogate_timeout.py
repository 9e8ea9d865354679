"""A bounded wait that gave up is reported by every call that hands out or
uses gradients, and no parameter changes."""
import numpy as np
import pytest

from test_gpu_surrogate_exact import rk  # noqa: F401  (fixture)

pytestmark = pytest.mark.gpu

SHAPE = (8, 16, 32)


@pytest.mark.parametrize("backend", [0, 1])
def test_timeout_stops_the_gradients(rk, backend):  # noqa: F811
    import torch
    lib = rk._lib
    nz, ny, nx = SHAPE
    sur = lib.rkl_sur_create(nz, ny, nx, (1.0 / nx, 1.0 / ny, 1.0 / nz), torch.cuda.current_stream().cuda_stream)
    lib.rkl_sur_set_backend(sur, backend)
    rng = np.random.default_rng(1)
    for l in range(6):
        co, ci = lib.rkl_sur_layer_shape(l)
        w = rng.normal(scale=np.sqrt(2.0 / (27 * ci)), size=(27, co, ci)).astype(np.float32)
        lib.rkl_sur_set_params(sur, l, w, np.zeros(co, dtype=np.float32))
    T = torch.rand(SHAPE, device="cuda") + 1.0
    b = torch.rand((3,) + SHAPE, device="cuda")
    target = 1e-3 * torch.randn(SHAPE, device="cuda")
    dz = torch.zeros((nz * ny * nx, 32), device="cuda", dtype=torch.bfloat16)

    def params():
        return [lib.rkl_sur_get_params(sur, l) for l in range(6)]

    def fails(call, *args):
        with pytest.raises(rk.RklError) as ei:
            call(sur, *args)
        assert ei.value.status == lib.RKL_ERR_TIMEOUT

    lib.rkl_sur_features(sur, T, b, 0.01, True, 100.0)
    lib.rkl_sur_train_step(sur, 2e-3, target, 1e-3)
    lib.rkl_sur_check(sur)
    before = params()

    lib.rkl_sur_selftest_timeout(sur)
    fails(lib.rkl_sur_get_grads, 2)
    fails(lib.rkl_sur_adam, 1e-3)
    fails(lib.rkl_sur_train_step, 2e-3, target, 1e-3)
    fails(lib.rkl_sur_check)
    # a layer's own gradient call, then Adam without a read in between
    lib.rkl_sur_layer_weight_grad(sur, 2, dz, dz)
    lib.rkl_sur_selftest_timeout(sur)
    fails(lib.rkl_sur_adam, 1e-3)
    fails(lib.rkl_sur_backward, target)
    fails(lib.rkl_sur_check)
    for (w0, b0), (w1, b1) in zip(before, params()):
        assert np.array_equal(w0, w1) and np.array_equal(b0, b1)

    # cleared: the pass runs again
    lib.rkl_sur_train_step(sur, 2e-3, target, 1e-3)
    lib.rkl_sur_get_grads(sur, 2)
    lib.rkl_sur_check(sur)
    assert any(not np.array_equal(w0, w1) for (w0, _), (w1, _) in zip(before, params()))
    lib.rkl_sur_destroy(sur)
