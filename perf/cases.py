"""Performance cases of the RKL2 conduction library: the calls that programs
built on it make, from a 2D ring of ten thousand cells to a 512^3 box.

A case is a dict of plain values; its "kind" is one of

* "step"      one RKL2 super-step of one grid (Plan.dt_expl, Plan.super_step)
* "split"     one operator-split step: donor-cell advection over dt_h and the
              conduction super-step (SplitDriver.step)
* "ensemble"  one super-step of many uneven problems (Ensemble.super_step)
* "layer"     one hidden layer of the surrogate network: forward, backward
              data and weight gradient (rkl_sur_layer_*)
* "train"     one training pass of the surrogate: features, forward, backward

Fields are drawn on the GPU from a seed: b a unit field (the normalised curl
of a random vector potential with |A_k|^2 ~ k^(-17/3) on shells 2 <= |k| <= 8,
or the azimuthal ring field), T a same-spectrum scalar field, a hot blob or a
hot sector.
"""
from __future__ import annotations

import math
import random

import numpy as np
import torch

import paper_1702_05487_gb300 as rk
from paper_1702_05487_gb300 import _lib
from paper_1702_05487_gb300.split import SplitDriver

SIZES = (32, 48, 64, 96, 128, 192)          # sides of an ensemble's problems


def listed():
    return [
        # the paper's 2D ring test in its own FP64 and Dirichlet walls: the
        # smallest call, 14 stages of ten thousand cells
        dict(name="ring100_f64", kind="step", field="ring", nx=100, ny=100, nz=0, dtype="f64", bc="dirichlet",
             kappa="const", perp=0.0, saturate=False, limiter=False, ratio=50.0, energies=False),
        # a 2D run at production resolution, ragged, FP32, saturated
        dict(name="plane_f32", kind="step", field="tangled", nx=1530, ny=1071, nz=0, dtype="f32", bc="periodic",
             kappa="spitzer", perp=1e-4, saturate=True, limiter=False, ratio=60.0, energies=False),
        # a small 3D box (test problems, parameter scans): 20 short stages
        dict(name="tangled64", kind="step", field="tangled", nx=64, ny=64, nz=64, dtype="f32", bc="periodic",
             kappa="spitzer", perp=1e-4, saturate=False, limiter=False, ratio=100.0, energies=False),
        # the ordinary production box: tangled field, Spitzer conductivity
        dict(name="tangled256", kind="step", field="tangled", nx=256, ny=256, nz=256, dtype="f32", bc="periodic",
             kappa="spitzer", perp=1e-4, saturate=False, limiter=False, ratio=100.0, energies=False),
        # the largest: saturated conduction out of a hot blob, 28 stages
        dict(name="blob512", kind="step", field="blob", nx=512, ny=512, nz=512, dtype="f32", bc="periodic",
             kappa="spitzer", perp=0.0, saturate=True, limiter=False, ratio=200.0, energies=False),
        # monotonicity-preserving run (MC limiter at every face) that logs
        # the energy before and after each super-step
        dict(name="limited_energies", kind="step", field="tangled", nx=224, ny=192, nz=160, dtype="f32",
             bc="periodic", kappa="spitzer", perp=1e-4, saturate=False, limiter=True, ratio=80.0, energies=True),
        # a box whose sides are whatever the physics asked for
        dict(name="ragged_f32", kind="step", field="tangled", nx=201, ny=150, nz=99, dtype="f32", bc="periodic",
             kappa="spitzer", perp=1e-4, saturate=False, limiter=False, ratio=60.0, energies=False),
        # a reference run in double precision
        dict(name="box_f64", kind="step", field="tangled", nx=112, ny=96, nz=80, dtype="f64", bc="periodic",
             kappa="spitzer", perp=1e-4, saturate=False, limiter=False, ratio=30.0, energies=False),
        # the operator-split loop of a host code, walls at a fixed temperature
        dict(name="split_walls", kind="split", nx=192, ny=128, nz=96, dtype="f32", bc="dirichlet", kappa="const",
             perp=1e-2, saturate=False, limiter=False, ratio=60.0),
        # a parameter study: 24 uneven problems advanced together
        dict(name="ensemble24", kind="ensemble", count=24, draw=4),
        # one hidden layer of the surrogate on its 128^3 patch
        dict(name="layer128", kind="layer", layer=2, nx=128, ny=128, nz=128),
        # one training pass of the whole network
        dict(name="train_96", kind="train", nx=96, ny=96, nz=96),
    ]


def _log_int(rng: random.Random, lo: int, hi: int) -> int:
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng: random.Random):
    kind = rng.choice(("plane", "box", "box", "box", "f64", "split", "ensemble", "layer", "train"))
    phys = dict(kappa=rng.choice(("spitzer", "spitzer", "const")), perp=rng.choice((0.0, 1e-4, 1e-2)),
                saturate=rng.random() < 0.4, limiter=rng.random() < 0.25, bc=rng.choice(("periodic", "periodic", "dirichlet")))
    ratio = round(math.exp(rng.uniform(math.log(20.0), math.log(200.0))), 2)
    if kind == "plane":
        f64 = rng.random() < 0.4
        hi = 400 if f64 else 2000
        return dict(kind="step", field="tangled", nx=_log_int(rng, 64, hi), ny=_log_int(rng, 64, hi), nz=0,
                    dtype="f64" if f64 else "f32", ratio=ratio, energies=rng.random() < 0.3, **phys)
    if kind == "box":
        n = [_log_int(rng, 32, 256) for _ in range(3)]
        if rng.random() < 0.7:                      # most programs pick a multiple of four
            n[0] = max(32, n[0] // 4 * 4)
        return dict(kind="step", field=rng.choice(("tangled", "blob")), nx=n[0], ny=n[1], nz=n[2], dtype="f32",
                    ratio=ratio, energies=rng.random() < 0.3, **phys)
    if kind == "f64":
        n = [_log_int(rng, 24, 100) for _ in range(3)]
        return dict(kind="step", field="tangled", nx=n[0], ny=n[1], nz=n[2], dtype="f64", ratio=min(ratio, 60.0),
                    energies=False, **phys)
    if kind == "split":
        n = [_log_int(rng, 32, 256) for _ in range(3)]
        n[0] = max(32, n[0] // 4 * 4)
        return dict(kind="split", nx=n[0], ny=n[1], nz=n[2], dtype="f32", ratio=ratio, **phys)
    if kind == "ensemble":
        return dict(kind="ensemble", count=_log_int(rng, 4, 40), draw=rng.randrange(10, 1 << 20))
    n = [16 * rng.randint(2, 9), 16 * rng.randint(2, 9), 4 * rng.randint(8, 34)]
    if rng.random() < 0.15:
        n[1] += 8                                   # sides that the wide blocks do not tile
    if kind == "layer":
        return dict(kind="layer", layer=rng.choice((1, 2, 3, 4)), nx=n[0], ny=n[1], nz=n[2])
    return dict(kind="train", nx=n[0], ny=n[1], nz=n[2])


# --------------------------------------------------------------------------
# inputs

def _gen(seed: int):
    return torch.Generator().manual_seed(int(seed))


def _waves(shape, gen, count: int, slope: float = -17.0 / 3.0):
    """`count` half spectra of random shell modes on a periodic grid of the
    given C-order shape, and the wavevector of every entry (x, y(, z))."""
    nd = len(shape)
    half = list(shape[:-1]) + [shape[-1] // 2 + 1]
    kmax = [min(8, (n - 1) // 2) for n in shape]
    ks = [torch.arange(-m, m + 1) for m in kmax[:-1]] + [torch.arange(0, kmax[-1] + 1)]
    grid = torch.meshgrid(*ks, indexing="ij")
    k2 = sum(g.double() ** 2 for g in grid)
    amp = torch.where((k2 >= 4) & (k2 <= 64), k2.clamp(min=1.0) ** (slope / 4.0), torch.zeros(()).double())
    box = amp * torch.complex(torch.randn((count,) + amp.shape, generator=gen, dtype=torch.float64),
                              torch.randn((count,) + amp.shape, generator=gen, dtype=torch.float64))
    index = torch.meshgrid(*[k % n for k, n in zip(ks, shape)], indexing="ij")
    kvec = [g.double() for g in reversed(grid)]
    return half, index, box, kvec[:nd]


def _synth(shape, half, index, modes):
    spec = torch.zeros(half, dtype=torch.complex64, device="cuda")
    spec[tuple(i.cuda() for i in index)] = modes.to(torch.complex64).cuda()
    return torch.fft.irfftn(spec, s=shape, norm="forward")


def _unit_field(shape, gen):
    """Unit field [ndim][...], normalised curl of a random vector potential."""
    nd = len(shape)
    half, index, A, k = _waves(shape, gen, 3 if nd == 3 else 1)
    if nd == 2:
        modes = [1j * k[1] * A[0], -1j * k[0] * A[0]]
    else:
        modes = [1j * (k[1] * A[2] - k[2] * A[1]), 1j * (k[2] * A[0] - k[0] * A[2]), 1j * (k[0] * A[1] - k[1] * A[0])]
    b = torch.stack([_synth(shape, half, index, m) for m in modes])
    mag = b.square().sum(0).sqrt_()
    b /= mag.clamp_(min=1e-6 * float(mag.mean()))
    return b


def _scalar(shape, gen):
    half, index, S, _ = _waves(shape, gen, 1)
    f = _synth(shape, half, index, S[0])
    return f / f.abs().max()


def _fields(case, shape, seed):
    gen = _gen(seed)
    nd = len(shape)
    if case["field"] == "ring":
        # the ring on [-1, 1]^2; the hot sector's angle varies with the seed
        a = float(torch.rand((), generator=gen)) * 2.0 * math.pi - math.pi
        y, x = torch.meshgrid(*[-1.0 + (torch.arange(n).double().cuda() + 0.5) * (2.0 / n) for n in shape],
                              indexing="ij")
        r = (x * x + y * y).sqrt()
        da = torch.remainder(torch.atan2(y, x) - a + math.pi, 2.0 * math.pi) - math.pi
        T = torch.where((r > 0.5) & (r < 0.7) & (da.abs() < math.pi / 12), 12.0, 10.0).double()
        return T, torch.stack([-y / r.clamp(min=1e-12), x / r.clamp(min=1e-12)])
    b = _unit_field(shape, gen)
    if case["field"] == "blob":
        h = 1.0 / max(shape)
        at = torch.rand(nd, generator=gen).tolist()
        r2 = 0.0
        for d, n in enumerate(shape):
            c = (torch.arange(n).cuda() + 0.5) / n - at[d]
            c = (c - torch.round(c)) * (n * h)
            r2 = r2 + (c * c).view([-1 if e == d else 1 for e in range(nd)])
        T = 1.0 + 9.0 * torch.exp(-r2 / 0.01)
    else:
        T = 1.0 + 0.2 * _scalar(shape, gen)
    return T, b


def _shape(case):
    return (case["nz"], case["ny"], case["nx"]) if case["nz"] else (case["ny"], case["nx"])


def _params(case):
    shape = _shape(case)
    L = 2.0 if case.get("field") == "ring" else 1.0
    h = L / max(shape)
    return dict(dx=(h,) * len(shape), bc=case["bc"], bc_value=10.0 if case.get("field") == "ring" else 1.0,
                kappa_model=case["kappa"], kappa_par0=0.01, kappa_perp_ratio=case["perp"],
                saturate=case["saturate"], phi=0.3, rho=1.0, limiter="mc" if case["limiter"] else "none")


def _step_inputs(case, seed):
    T, b = _fields(dict(field="tangled", **case) if "field" not in case else case, _shape(case), seed)
    dt = torch.float64 if case["dtype"] == "f64" else torch.float32
    return T.to(dt).contiguous(), b.to(dt).contiguous()


def _flow(case, seed):
    """Cell-centred ABC flow [3][z][y][x] with seeded phases, scaled so that
    dt_h (C_h = 0.8) is `ratio` explicit conduction steps at T = 1.2."""
    p = (torch.rand(3, generator=_gen(seed + 77), dtype=torch.float64) * 2 * math.pi).tolist()
    z, y, x = torch.meshgrid(*[2 * math.pi * (torch.arange(n).double().cuda() + 0.5) / n for n in _shape(case)],
                             indexing="ij")
    u = torch.stack([torch.sin(z + p[0]) + torch.cos(y + p[1]), torch.sin(x + p[1]) + torch.cos(z + p[2]),
                     torch.sin(y + p[2]) + torch.cos(x + p[0])])
    prm = _params(case)
    rate = float(u.abs().sum(0).max()) / prm["dx"][0]
    return (u * (0.8 / (case["ratio"] * _dt_expl(prm, 1.2)) / rate)).float().contiguous()


def _problems(case):
    rng = np.random.default_rng(case["draw"])
    out = []
    for _ in range(case["count"]):
        nx, ny, nz = (int(v) for v in rng.choice(SIZES, 3))
        h = 1.0 / max(nx, ny, nz)
        out.append(((nz, ny, nx), dict(dx=(h, h, h), kappa_model="spitzer", kappa_par0=float(rng.uniform(1e-3, 1e-1)),
                                       kappa_perp_ratio=1e-4), float(rng.uniform(20.0, 400.0))))
    return out


def _ensemble_inputs(case, seed):
    fields = []
    for p, (shape, prm, ratio) in enumerate(_problems(case)):
        gen = _gen(1000 * seed + p)
        b = _unit_field(shape, gen)
        T = (1.0 + 0.2 * _scalar(shape, gen)).float()
        fields.append((T, b.float(), ratio * _dt_expl(prm, float(T.max()))))
    return fields


def _layer_inputs(case, seed):
    """A hidden layer's BF16 weights (as a checkpoint holds them) and bias,
    its input activations (after a ReLU), the mask of the layer below and the
    gradient that comes back."""
    co, ci = _lib.rkl_sur_layer_shape(case["layer"])
    V = case["nx"] * case["ny"] * case["nz"]
    gen = torch.Generator("cuda").manual_seed(int(seed))
    w = torch.randn((27, co, ci), generator=gen, device="cuda") * math.sqrt(2.0 / (27 * ci))
    w = w.bfloat16().float()
    bias = 0.1 * torch.randn(co, generator=gen, device="cuda")
    x = torch.randn((V, ci), generator=gen, device="cuda").relu_().bfloat16()
    dz = (1e-3 * torch.randn((V, co), generator=gen, device="cuda")).bfloat16()
    return w, bias, x, dz


SUR_FLUX, SUR_HEAD, SUR_RATIO = 0.0625, 1e-4, 100.0


def _train_inputs(case, seed):
    """A patch (T, b), the training target and the network's parameters."""
    shape = _shape(case)
    gen = _gen(seed)
    b = _unit_field(shape, gen).contiguous()
    T = (1.0 + 0.2 * _scalar(shape, gen)).contiguous()
    target = (0.01 * _scalar(shape, gen)).contiguous()
    params = []
    for l in range(6):
        co, ci = _lib.rkl_sur_layer_shape(l)
        rci, rco = (9 if l == 0 else ci), (3 if l == 5 else co)
        w = torch.zeros((27, co, ci))
        w[:, :rco, :rci] = torch.randn((27, rco, rci), generator=gen) * math.sqrt(2.0 / (27 * rci))
        params.append((w.bfloat16().float().numpy(), np.zeros(co, dtype=np.float32)))
    return T, b, target, params


def _train_params(case):
    shape = _shape(case)
    return dict(dx=(1.0 / max(shape),) * 3, kappa_model="spitzer", kappa_par0=0.01, kappa_perp_ratio=1e-4)


# --------------------------------------------------------------------------
# the calls

class _Sur:
    """Surrogate handle that is given back with the state."""

    def __init__(self, case, dx):
        self.handle = _lib.rkl_sur_create(case["nz"], case["ny"], case["nx"], dx,
                                          torch.cuda.current_stream().cuda_stream)

    def __del__(self):
        try:
            _lib.rkl_sur_destroy(self.handle)
        except Exception:
            pass


def prepare(case, seed):
    kind = case["kind"]
    st = dict(case=case)
    if kind == "step":
        st["T"], st["b"] = _step_inputs(case, seed)
        st["plan"] = rk.Plan(_shape(case), case["dtype"], params=_params(case))
    elif kind == "split":
        st["T"], st["b"] = _step_inputs(case, seed)
        st["other"] = torch.empty_like(st["T"])
        st["u"] = _flow(case, seed)
        st["driver"] = SplitDriver(_shape(case), case["dtype"], params=_params(case))
    elif kind == "ensemble":
        fields = _ensemble_inputs(case, seed)
        st["ens"] = rk.Ensemble([(s, prm) for s, prm, _ in _problems(case)])
        st["T0"] = torch.cat([T.reshape(-1) for T, _, _ in fields])
        st["T"] = torch.empty_like(st["T0"])
        st["b"] = torch.cat([b.reshape(-1) for _, b, _ in fields])
        st["dt"] = [dt for _, _, dt in fields]
    elif kind == "layer":
        w, bias, st["x"], st["dz"] = _layer_inputs(case, seed)
        st["sur"] = _Sur(case, (1.0 / max(_shape(case)),) * 3)
        _lib.rkl_sur_set_params(st["sur"].handle, case["layer"], w.cpu().numpy(), bias.cpu().numpy())
        st["y"], st["dx"] = torch.empty_like(st["dz"]), torch.empty_like(st["x"])
    else:
        st["T"], st["b"], st["target"], params = _train_inputs(case, seed)
        prm = _train_params(case)
        st["plan"] = rk.Plan(_shape(case), "f32", params=prm)
        st["sur"] = _Sur(case, prm["dx"])
        for l, (w, b) in enumerate(params):
            _lib.rkl_sur_set_params(st["sur"].handle, l, w, b)
        st["dT"] = torch.empty_like(st["T"])
    return st


def run(st):
    case = st["case"]
    kind = case["kind"]
    if kind == "step":
        # super-steps of a fixed multiple of the explicit step, the state in place
        dt = case["ratio"] * st["plan"].dt_expl(st["T"])
        got = st["plan"].super_step(dt, st["T"], st["b"], energies=case["energies"])
        return dict(T=st["T"], s=got[0], before=got[1], after=got[2]) if case["energies"] else dict(T=st["T"], s=got)
    if kind == "split":
        T, dt, s = st["driver"].step(st["T"], st["other"], st["b"], st["u"])
        st["T"], st["other"] = T, st["T"]
        return dict(T=T, dt=dt, s=s)
    if kind == "ensemble":
        # every entry of the study starts from the stored initial fields
        st["T"].copy_(st["T0"])
        return dict(s=st["ens"].super_step(st["dt"], st["T"], st["b"]), T=st["T"])
    sur = st["sur"].handle
    if kind == "layer":
        l = case["layer"]
        _lib.rkl_sur_layer_forward(sur, l, st["x"], st["y"])
        _lib.rkl_sur_layer_backward_data(sur, l, st["dz"], st["x"], st["dx"])
        _lib.rkl_sur_layer_weight_grad(sur, l, st["dz"], st["x"])
        gw, gb = _lib.rkl_sur_get_grads(sur, l)
        return dict(y=st["y"], dx=st["dx"], gw=gw, gb=gb)
    dt = SUR_RATIO * st["plan"].dt_expl(st["T"])
    _lib.rkl_sur_features_flux(sur, st["plan"].handle, st["T"], st["b"], SUR_RATIO, SUR_FLUX * dt / SUR_HEAD)
    _lib.rkl_sur_forward(sur, SUR_HEAD, st["dT"])
    loss = _lib.rkl_sur_backward(sur, st["target"])
    grads = [_lib.rkl_sur_get_grads(sur, l) for l in range(6)]
    return dict(dT=st["dT"], loss=loss, gw=[g[0] for g in grads], gb=[g[1] for g in grads])


def _stages(ratio):
    return 1 + int(0.5 * (-1.0 + math.sqrt(9.0 + 16.0 * ratio)))


def _step_work(cells, nd, s, esize, saturate, limiter):
    """s stages of one grid.  Every stage reads the stage before it and b, and
    from the second on Y_{j-2}, Y_0 and M(Y_0); it writes Y_j (the first one
    M(Y_0) too)."""
    words = cells * ((3 + nd) + (s - 1) * (5 + nd))
    face = 14 + 8 * (nd - 1) + 4 + (20 if saturate else 0) + (16 * (nd - 1) if limiter else 0)
    return dict(bytes=float(words * esize), flops=float(cells * s * (nd * (face + 2) + 9)))


def work(case):
    kind = case["kind"]
    if kind == "ensemble":
        got = [_step_work(math.prod(s), 3, _stages(r), 4, False, False) for s, _, r in _problems(case)]
        return {k: sum(g[k] for g in got) for k in ("bytes", "flops")}
    if kind in ("layer", "train"):
        V = case["nx"] * case["ny"] * case["nz"]
        if kind == "layer":                         # x, dz (twice needed, read once), y, dx, the gradients
            return dict(bytes=float(V * 64 * 4 + 27 * 32 * 32 * 4), flops=float(3 * 2 * 27 * 32 * 32 * V))
        per = 2 * 27 * (9 * 32 + 4 * 32 * 32 + 32 * 3)
        # T, b, target read, dT written; five hidden activations of 32 BF16
        # channels written and read back (forward, mask and weight gradient)
        return dict(bytes=float(V * (4 * 6 + 5 * 64 * 2)), flops=float(V * (3 * per - 2 * 27 * 9 * 32)))
    cells = math.prod(_shape(case))
    nd = len(_shape(case))
    es = 8 if case["dtype"] == "f64" else 4
    w = _step_work(cells, nd, _stages(case["ratio"]), es, case["saturate"], case["limiter"])
    if kind == "split":                             # u read, T read and written once more
        w = dict(bytes=w["bytes"] + cells * es * (nd + 2), flops=w["flops"] + cells * 10 * nd)
    return w


# --------------------------------------------------------------------------
# the same results in 64 bits with plain torch

def _kappa(prm, T):
    if prm["kappa_model"] == "spitzer":
        return prm["kappa_par0"] * T * T * (T.sqrt() if torch.is_tensor(T) else math.sqrt(T))
    return prm["kappa_par0"] * (torch.ones_like(T) if torch.is_tensor(T) else 1.0)


def _dt_expl(prm, Tmax):
    inv = sum(1.0 / h ** 2 for h in prm["dx"])
    return 0.5 / (_kappa(prm, Tmax) * (1.0 + prm["kappa_perp_ratio"]) * inv)


def _pad(A, bc, value):
    """A with one ghost cell on every side; value None copies the nearest cell."""
    for d in range(A.dim()):
        n = A.shape[d]
        lo, hi = A.narrow(d, 0, 1), A.narrow(d, n - 1, 1)
        if bc == "periodic":
            lo, hi = hi, lo
        elif value is not None:
            lo = hi = torch.full_like(lo, value)
        A = torch.cat([lo, A, hi], d)
    return A


def _mc(a, b):
    m = torch.minimum(0.5 * (a + b).abs(), 2.0 * torch.minimum(a.abs(), b.abs()))
    return torch.where(a * b > 0, torch.copysign(m, a), torch.zeros_like(m))


def _faces(T, bp, prm, axis):
    """Flux on the n + 1 faces normal to `axis` (a component index, x first)."""
    nd = T.dim()
    Tp = _pad(T, prm.get("bc", "periodic"), prm.get("bc_value", 0.0))
    dim = nd - 1 - axis

    def cut(A, side, comp=None, shift=0):
        for d in range(nd):
            n = A.shape[d] - 2
            if d == dim:
                A = A.narrow(d, side, n + 1)
            else:
                A = A.narrow(d, 1 + (shift if comp is not None and d == nd - 1 - comp else 0), n)
        return A

    dx = prm["dx"]
    TL, TR = cut(Tp, 0), cut(Tp, 1)
    grad, bf = {axis: (TR - TL) / dx[axis]}, {}
    for e in range(nd):
        if e != axis:
            up, dn = [cut(Tp, s, e, 1) for s in (0, 1)], [cut(Tp, s, e, -1) for s in (0, 1)]
            if prm.get("limiter") == "mc":
                grad[e] = _mc(_mc(up[0] - TL, TL - dn[0]), _mc(up[1] - TR, TR - dn[1])) / dx[e]
            else:
                grad[e] = (up[0] + up[1] - dn[0] - dn[1]) / (4.0 * dx[e])
        bf[e] = 0.5 * (cut(bp[e], 0) + cut(bp[e], 1))
    Tf = 0.5 * (TL + TR)
    kpar = _kappa(prm, Tf)
    bdg = sum(bf[e] * grad[e] for e in range(nd))
    F = -kpar * bf[axis] * bdg - prm["kappa_perp_ratio"] * kpar * grad[axis]
    if prm.get("saturate"):
        mag = F * F
        for e in range(nd):
            if e != axis:
                mag += (kpar * bf[e] * bdg + prm["kappa_perp_ratio"] * kpar * grad[e]) ** 2
        q = 5.0 * prm["phi"] * prm["rho"] * Tf * Tf.sqrt()
        F = q / (q + mag.sqrt_()) * F
    return F


def _M(T, bp, prm):
    out = torch.zeros_like(T)
    for axis in range(T.dim()):
        F = _faces(T, bp, prm, axis)
        d = T.dim() - 1 - axis
        out -= (F.narrow(d, 1, T.shape[d]) - F.narrow(d, 0, T.shape[d])) / prm["dx"][axis]
    return out


def _super_step(T, b, prm, dt, s):
    bp = [_pad(c, prm.get("bc", "periodic"), None) for c in b.double()]
    bj = lambda j: 1.0 / 3.0 if j <= 2 else (j * j + j - 2.0) / (2.0 * j * (j + 1.0))  # noqa: E731
    w1 = 4.0 / (s * s + s - 2.0)
    Y0 = T
    MY0 = _M(Y0, bp, prm)
    Ym, Y = Y0, Y0 + bj(1) * w1 * dt * MY0
    for j in range(2, s + 1):
        mu, nu = (2.0 * j - 1.0) / j * bj(j) / bj(j - 1), -(j - 1.0) / j * bj(j) / bj(j - 2)
        Yn = mu * Y + nu * Ym
        Yn += (1.0 - mu - nu) * Y0
        Yn += mu * w1 * dt * _M(Y, bp, prm)
        Yn -= (1.0 - bj(j - 1)) * mu * w1 * dt * MY0
        Ym, Y = Y, Yn
    return Y


def _advect(T, u, prm, dt):
    out = T.clone()
    nd = T.dim()
    Tp = _pad(T, prm["bc"], prm["bc_value"])
    for axis in range(nd):
        up = _pad(u[axis].double(), prm["bc"], None)
        d = nd - 1 - axis

        def inner(A, side):
            for e in range(nd):
                A = A.narrow(e, side, T.shape[e] + 1) if e == d else A.narrow(e, 1, T.shape[e])
            return A
        uf = 0.5 * (inner(up, 0) + inner(up, 1))
        F = uf * torch.where(uf >= 0, inner(Tp, 0), inner(Tp, 1))
        out -= dt * (F.narrow(d, 1, T.shape[d]) - F.narrow(d, 0, T.shape[d])) / prm["dx"][axis]
    return out


def _shifted(x, shape, o):
    """x[v + offset o] for channels-last x of a periodic patch."""
    d = (o // 9 - 1, (o // 3) % 3 - 1, o % 3 - 1)
    return torch.roll(x.view(shape + (-1,)), [-v for v in d], (0, 1, 2)).reshape(x.shape)


def _conv(x, w, shape):
    out = torch.zeros((x.shape[0], w.shape[1]), dtype=torch.float64, device=x.device)
    for o in range(27):
        out.addmm_(_shifted(x, shape, o), w[o].T)
    return out


def _conv_back(dz, w, shape):
    out = torch.zeros((dz.shape[0], w.shape[2]), dtype=torch.float64, device=dz.device)
    for o in range(27):
        out.addmm_(_shifted(dz, shape, 26 - o), w[o])
    return out


def _conv_grad(dz, x, shape):
    return torch.stack([dz.T @ _shifted(x, shape, o) for o in range(27)])


def exact(case, seed):
    kind = case["kind"]
    if kind == "step":
        T, b = _step_inputs(case, seed)
        prm = _params(case)
        T = T.double()
        dt = case["ratio"] * _dt_expl(prm, float(T.max()))
        Y = _super_step(T, b, prm, dt, _stages(case["ratio"]))
        if not case["energies"]:
            return dict(T=Y, s=None)
        dV = math.prod(prm["dx"])
        return dict(T=Y, s=None, before=float(T.sum()) * dV, after=float(Y.sum()) * dV)
    if kind == "split":
        T, b = _step_inputs(case, seed)
        u = _flow(case, seed)
        prm = _params(case)
        dt = 0.8 / float((u.double().abs().sum(0) / prm["dx"][0]).max())
        A = _advect(T.double(), u, prm, dt)
        return dict(T=_super_step(A, b, prm, dt, _stages(dt / _dt_expl(prm, float(A.max())))), dt=dt, s=None)
    if kind == "ensemble":
        out = []
        for (T, b, dt), (_, prm, _) in zip(_ensemble_inputs(case, seed), _problems(case)):
            s = _stages(dt / _dt_expl(prm, float(T.max())))
            out.append(_super_step(T.double(), b, prm, dt, s).reshape(-1))
        return dict(s=None, T=torch.cat(out))
    shape = _shape(case)
    if kind == "layer":
        w, bias, x, dz = _layer_inputs(case, seed)
        w, x, dz = w.double(), x.double(), dz.double()
        return dict(y=torch.relu(_conv(x, w, shape) + bias.double()), dx=_conv_back(dz, w, shape) * (x > 0),
                    gw=_conv_grad(dz, x, shape), gb=dz.sum(0))
    # the whole network without any 16-bit storage between the layers: dT
    # only (the gradients' own accuracy is that of the layers' case)
    T, b, target, params = _train_inputs(case, seed)
    prm = _train_params(case)
    T64 = T.double()
    dt = SUR_RATIO * _dt_expl(prm, float(T64.max()))
    bp = [_pad(c, "periodic", None) for c in b.double()]
    x = torch.zeros(shape + (16,), dtype=torch.float64, device="cuda")
    x[..., 0] = T64 - 1.0
    for c in range(3):
        x[..., 1 + c] = b[c]
        F = _faces(T64, bp, prm, c)
        x[..., 6 + c] = SUR_FLUX * dt / SUR_HEAD * F.narrow(2 - c, 1, shape[2 - c])
    x[..., 4] = torch.log10(_kappa(prm, T64)) + 2.0
    x[..., 5] = SUR_RATIO / 100.0
    a = x.reshape(-1, 16)
    for l, (w, _) in enumerate(params):
        a = _conv(a, torch.from_numpy(w).cuda().double(), shape)
        a = torch.relu_(a) if l < 5 else a
    G = a.view(shape + (-1,))
    dT = -SUR_HEAD * sum((G[..., c] - torch.roll(G[..., c], 1, 2 - c)) / prm["dx"][c] for c in range(3))
    none = [None] * 6
    return dict(dT=dT, loss=0.5 * float((dT - target.double()).square().mean()), gw=none, gb=none)
