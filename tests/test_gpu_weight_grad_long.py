"""Weight and bias gradients of one layer where a CTA's run of steps is long
(every barrier goes through many phases, runs cross tile columns and end inside
one) and where the halo wraps onto the tile itself, exactly: small integer
operands make every product and sum an integer below 2^24."""
import numpy as np
import pytest

from test_gpu_surrogate_exact import rk  # noqa: F401  (fixture)

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape", [(4, 8, 16), (12, 24, 16), (4, 16, 16), (100, 64, 96), (128, 128, 128)])
@pytest.mark.parametrize("layer", [0, 2, 5])
def test_weight_grad_exact(rk, shape, layer):  # noqa: F811
    import torch
    lib = rk._lib
    nz, ny, nx = shape
    V = nz * ny * nx
    co, ci = lib.rkl_sur_layer_shape(layer)
    sur = lib.rkl_sur_create(nz, ny, nx, (1.0, 1.0, 1.0), torch.cuda.current_stream().cuda_stream)
    g = torch.Generator("cuda").manual_seed(7)
    # |sum| <= 4 V of values in [-2, 2]: below 2^24 for V <= 2^21
    dz = torch.randint(-2, 3, (V, co), generator=g, device="cuda").double()
    x = torch.randint(-2, 3, (V, ci), generator=g, device="cuda").double()
    lib.rkl_sur_layer_weight_grad(sur, layer, dz.bfloat16(), x.bfloat16())
    gw, gb = lib.rkl_sur_get_grads(sur, layer)
    lib.rkl_sur_check(sur)
    lib.rkl_sur_destroy(sur)
    box = x.view(nz, ny, nx, ci)
    for o in range(27):
        off = (o // 9 - 1, (o // 3) % 3 - 1, o % 3 - 1)
        want = dz.T @ torch.roll(box, [-v for v in off], (0, 1, 2)).reshape(V, ci)
        assert np.array_equal(gw[o].astype(np.float64), want.cpu().numpy()), off
    assert np.array_equal(gb.astype(np.float64), dz.sum(0).cpu().numpy())
