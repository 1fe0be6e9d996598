"""The workloads whose speed is followed, each one pass through the public entry points.

Six kinds of work, as programs of this package do them:

  pic      advance one run by some steps (pic_step) and read the field back
  load     take a run's particles from host memory, advance it one step, read the field back
  batch    advance an ensemble of trench runs (pic_batch_step), read every member's field
  deposit  the stand-alone deposit of device-resident particles (pic_deposit_static)
  unet     the warm-start network: a forward pass, or the loss and every gradient
  layer    one layer of that network through its own entry point

`exact` restates each in FP64 with torch and numpy alone.
"""
from __future__ import annotations

import ctypes
import math
from types import SimpleNamespace

import numpy as np
import torch

import paper_1610_03918_gb300 as pg

# ---------------------------------------------------------------------------
# the cases
# ---------------------------------------------------------------------------


def _pic(name, kind, nx, ny, **kw):
    c = dict(name=name, kind=kind, nx=nx, ny=ny, px=False, py=True, depth=0, y0=0, width=0, phi_el=-20.0,
             rf=0.0, recycle=False, mass=1836.0, tau=0.1, ppc=64, surface=False, sort_every=8, steps=16)
    c.update(kw)
    return c


def listed():
    return [
        # The paper's own run: a small box advanced thousands of steps, where a
        # step is a few short kernels and its time is latency and launches.
        # 8-step sorts, RF electrode, recycled ions.
        _pic("paper_80x30", "pic", 80, 30, depth=20, y0=5, width=15, phi_el=0.0, rf=5.0, recycle=True,
             mass=3672.0, tau=1.0, ppc=100),
        # The doubly periodic box of the energy and oscillation checks (singular system).
        _pic("periodic_64x64", "pic", 64, 64, px=True, phi_el=0.0, ppc=50),
        # All four walls grounded and absorbing.
        _pic("bounded_256x256", "pic", 256, 256, py=False, phi_el=0.0, ppc=100),
        # The headline production run: 85M particles, bottom charging, sorted
        # every 24 steps (about what its own tuning chooses).
        _pic("trench_1024x512", "pic", 1024, 512, depth=200, y0=251, width=10, ppc=100, surface=True,
             sort_every=24, steps=24),
        # A run (re)started or driven from host memory: the whole state from
        # pinned buffers, one step, the field back.
        _pic("load_512x256", "load", 512, 256, depth=100, y0=118, width=20, ppc=64, surface=True, steps=1),
        # The trench-width sweep: members of different grids advanced together.
        dict(name="ensemble_8", kind="batch", members=8, ppc=16, sort_every=24, steps=24),
        # Deposit of another program's particles on the trench grid.
        dict(name="deposit_8M", kind="deposit", nx=1024, ny=512, px=False, py=True, n=8_388_608),
        # The learned guess of one solve at the trench grid.
        dict(name="forward_1032x512", kind="unet", batch=1, height=1032, width=512, grad=False),
        # One pass of training at the trench grid (the batch it is trained with).
        dict(name="gradients_b4", kind="unet", batch=4, height=1032, width=512, grad=True),
        # Single layers of the network: the top level's 32 -> 32 convolution ...
        dict(name="conv_top", kind="layer", op="conv", batch=1, height=1032, width=512, cin=32, cout=32),
        # ... a deep one, 256 channels of [upsampled | skip] -> 128, batch 4 ...
        dict(name="conv_deep", kind="layer", op="conv", batch=4, height=258, width=128, cin=256, cout=128),
        # ... and the weight gradient of a middle one.
        dict(name="wgrad_mid", kind="layer", op="wgrad", batch=4, height=516, width=256, cin=64, cout=64),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _fit(nx, ny, px, py, even):
    """The nearest sizes the solver's hierarchy takes: halved together while both are even
    (a periodic half must stay even), what is left has to be small."""
    step = 2 if even else 1
    while True:
        a, b = max(step, nx - nx % step), max(step, ny - ny % step)
        ca, cb = a, b
        while ca % 2 == 0 and cb % 2 == 0 and min(ca, cb) >= 4 and not (px and ca % 4) and not (py and cb % 4):
            ca, cb = ca // 2, cb // 2
        if (ca + 1) * (cb + 1) <= 2500:
            return a, b
        step *= 2


def _draw_pic(rng, kind):
    most = 12_000_000                       # particles of one species
    nx, ny = _log(rng, 32, 600), _log(rng, 24, 512)
    box = rng.choice(["trench", "trench", "trench", "plates", "bounded", "periodic"])
    if box in ("trench", "plates") and rng.random() < 0.4:
        ny = 1 << rng.randint(5, 9)
    nx, ny = _fit(nx, ny, box == "periodic", box != "bounded", box != "bounded")
    ppc = max(4, min(_log(rng, 8, 120), most // (nx * ny)))
    steps = rng.choice([4, 8, 12])
    c = _pic(None, kind, nx, ny, ppc=ppc, sort_every=rng.choice([8, 24]), steps=1 if kind == "load" else steps)
    del c["name"]
    if box == "trench":
        width = rng.randint(2, max(2, min(40, ny // 3)))
        c.update(depth=max(3, int(0.2 * nx)), width=width, y0=(ny - width) // 2, surface=rng.random() < 0.7)
        if rng.random() < 0.3:
            c.update(phi_el=0.0, rf=5.0, recycle=True, mass=3672.0, tau=1.0)
    elif box == "plates":
        c.update(phi_el=rng.choice([-20.0, -5.0]))
    elif box == "bounded":
        c.update(py=False, phi_el=0.0)
    else:
        c.update(px=True, phi_el=0.0)
    return c


def draw(rng):
    kind = rng.choice(["pic", "pic", "pic", "load", "batch", "deposit", "unet", "layer", "layer", "layer"])
    if kind in ("pic", "load"):
        return _draw_pic(rng, kind)
    if kind == "batch":
        return dict(kind=kind, members=rng.randint(2, 10), ppc=rng.randint(4, 16), sort_every=rng.choice([8, 24]),
                    steps=rng.choice([8, 16, 24]))
    if kind == "deposit":
        return dict(kind=kind, nx=_log(rng, 20, 1000), ny=_log(rng, 20, 1000), px=rng.random() < 0.3,
                    py=rng.random() < 0.7, n=_log(rng, 10_000, 12_000_000))
    if kind == "unet":
        grad = rng.random() < 0.4
        h, w = 8 * _log(rng, 4, 129), 8 * _log(rng, 3, 64)
        return dict(kind=kind, batch=rng.randint(1, 4 if grad else 2), height=h, width=w, grad=grad)
    op = rng.choice(["conv", "conv", "wgrad", "upconv", "upback", "upwgrad"])
    level = rng.randint(0, 3)
    h, w = max(8, _log(rng, 30, 1032) >> level), max(8, _log(rng, 20, 512) >> level)
    co = 32 << level
    ci = rng.choice([co, max(32, co // 2), min(256, 2 * co)])
    if op.startswith("up"):
        ci, co = (64 << min(level, 2)), (32 << min(level, 2))
    return dict(kind=kind, op=op, batch=rng.randint(1, 4), height=h, width=w, cin=ci, cout=co)


# ---------------------------------------------------------------------------
# particle runs
# ---------------------------------------------------------------------------


def _workload(c):
    """The description of a run that pg.Sim takes."""
    return SimpleNamespace(
        name="run", nx=c["nx"], ny=c["ny"], periodic_x=c["px"], periodic_y=c["py"], dt=0.1, phi_top=0.0,
        phi_electrode=c["phi_el"], trench_depth=c["depth"], trench_y0=c["y0"], trench_width=c["width"],
        ppc=c["ppc"], surface_charge=c["surface"], poisson_rtol=1e-6, sort_every=c["sort_every"],
        phi_rf_amp=c["rf"], omega_rf=0.01 if c["rf"] else 0.0, recycle=c["recycle"], source_x0=0, source_x1=0,
        recycle_seed=11, charge=(-1.0, 1.0), alpha=(-1.0, 1.0 / c["mass"]),
        vth=(1.0, math.sqrt(c["tau"] / c["mass"])))


_GRIDS = [(128, 256), (256, 256), (256, 512), (512, 512)]   # (y cells, x cells) of the width sweep


def _member(c, k):
    wy, hx = _GRIDS[k % 4]
    width = 1 + int(round(39 * k / 47))
    return _pic("m", "pic", hx, wy, depth=int(round(0.195 * hx)), y0=(wy - width) // 2, width=width, ppc=c["ppc"],
                surface=True, sort_every=c["sort_every"], steps=c["steps"])


def _conductor(c):
    m = np.zeros((c["nx"], c["ny"]), bool)
    if c["depth"]:
        m[c["nx"] - c["depth"]:] = True
        if c["width"]:
            m[c["nx"] - c["depth"]:, c["y0"]:c["y0"] + c["width"]] = False
    return m


def _dev():
    return torch.device("cuda" if torch.cuda.is_available() else "cpu")


def _particles(c, seed, s):
    """ppc particles per plasma cell, uniform in the cell, Maxwellian: x, y, vx, vy (FP64, on the GPU)."""
    d = _dev()
    g = torch.Generator(device=d).manual_seed(1000 * int(seed) + s)
    cells = torch.from_numpy(np.argwhere(~_conductor(c))).to(d).double().repeat_interleave(c["ppc"], 0)
    n = cells.shape[0]
    vth = 1.0 if s == 0 else math.sqrt(c["tau"] / c["mass"])
    r = [torch.rand(n, generator=g, device=d, dtype=torch.float64) for _ in range(2)]
    v = [vth * torch.randn(n, generator=g, device=d, dtype=torch.float64) for _ in range(2)]
    return [cells[:, 0] + r[0], cells[:, 1] + r[1], v[0], v[1]]


def _n_particles(c):
    return int((~_conductor(c)).sum()) * c["ppc"]


def _field(sim):
    # the field is held in FP32 on the device; the read-back hands it over in FP64 arrays
    return np.stack(sim.efield()).astype(np.float32)


def _make_sim(c, seed):
    sim = pg.Sim(_workload(c), capacity=_n_particles(c), hit_capacity=1 << 16)
    for s in (0, 1):
        sim.load(s, *[a.cpu().numpy() for a in _particles(c, seed, s)], v_at_t0=True)
    sim.step(0)
    return sim


# ---------------------------------------------------------------------------
# the network and its layers
# ---------------------------------------------------------------------------
_CH = (32, 64, 128, 256)


def _layers():
    """(kind, cin, cout) in parameter order."""
    out, prev = [], 2
    for ch in _CH:
        out += [("conv", prev, ch), ("conv", ch, ch)]
        prev = ch
    for lv in (2, 1, 0):
        out += [("up", _CH[lv + 1], _CH[lv]), ("conv", 2 * _CH[lv], _CH[lv]), ("conv", _CH[lv], _CH[lv])]
    return out + [("head", _CH[0], 1)]


def _params(seed):
    """He-initialised weights, small biases: the flat FP32 vector the network takes."""
    rng = np.random.default_rng([int(seed), 5])
    parts = []
    for kind, ci, co in _layers():
        n, fan = {"conv": (co * 9 * ci, 9 * ci / 2), "up": (4 * ci * co, ci / 2), "head": (ci, ci)}[kind]
        parts += [rng.standard_normal(n) / math.sqrt(fan), 0.05 * rng.standard_normal(co)]
    return np.concatenate(parts).astype(np.float32)


def _net_inputs(c, seed):
    """(rho / max |rho|, conductor mask) and a smooth target."""
    d = _dev()
    g = torch.Generator(device=d).manual_seed(int(seed))
    B, H, W = c["batch"], c["height"], c["width"]
    x = torch.zeros((B, H, W, 2), device=d)
    x[..., 0] = torch.randn((B, H, W), generator=g, device=d).clamp_(-4, 4) * 0.25
    x[:, 0, :, 1] = 1.0
    x[:, H - H // 5:, :, 1] = 1.0
    x[:, H - H // 5:, W // 2 - 4:W // 2 + 4, 1] = 0.0
    x[..., 0] *= 1.0 - x[..., 1]
    i = torch.arange(H, device=d).view(1, H, 1) / H
    j = torch.arange(W, device=d).view(1, 1, W) / W
    ph = torch.rand((B, 1, 1), generator=g, device=d)
    t = torch.sin(math.pi * i) * (0.5 + 0.3 * torch.cos(2 * math.pi * (j + ph))) + torch.zeros_like(x[..., 0])
    return x.contiguous(), t.contiguous()


def _layer_inputs(c, seed):
    """A layer's input tensor, output-side gradient and weights (activations after a ReLU: half zeros)."""
    d = _dev()
    g = torch.Generator(device=d).manual_seed(int(seed))
    B, H, W, ci, co = (c[k] for k in ("batch", "height", "width", "cin", "cout"))
    up = c["op"].startswith("up")

    def act(h, w, ch):
        return torch.randn((B, h, w, ch), generator=g, device=d).clamp_(min=0).to(torch.bfloat16)

    x = act(H, W, ci)
    dy = (torch.randn((B, 2 * H if up else H, 2 * W if up else W, co), generator=g, device=d) * 1e-2)
    dy = (dy * (torch.rand(dy.shape, generator=g, device=d) < 0.5)).to(torch.bfloat16)
    w = torch.randn((4 * ci * co if up else co * 9 * ci,), generator=g, device=d) / math.sqrt((ci if up else 9 * ci) / 2)
    b = 0.1 * torch.randn((co,), generator=g, device=d)
    return x, dy, w, b


_I, _P = ctypes.c_int32, ctypes.c_void_p
_ARGS = {
    "pic_conv3x3_bf16": [_I, _I, _I, _I, _P, _I, _I, _I, _P, _P, _I, _P, _I, _I, _I, _P],
    "pic_conv3x3_wgrad_bf16": [_I, _I, _I, _I, _P, _P, _I, _I, _I, _I, _P, _P],
    "pic_upconv_bf16": [_I, _I, _I, _I, _P, _I, _P, _P, _P, _I, _I, _I, _P],
    "pic_upconv_back_bf16": [_I, _I, _I, _I, _P, _I, _I, _I, _P, _P, _I, _P],
    "pic_upconv_wgrad_bf16": [_I, _I, _I, _I, _P, _I, _P, _I, _I, _I, _P, _P, _P],
    "pic_deposit_static": [_I, _I, _I, _I, ctypes.c_int64, _P, _P, ctypes.c_double, _P, _P],
}


def _entry(name):
    f = getattr(pg.load_library(), name)
    f.argtypes, f.restype = _ARGS[name], ctypes.c_int
    return f


def _ok(st, name):
    if st != pg.PIC_OK:
        raise pg.PicError(st, name)


# ---------------------------------------------------------------------------
# prepare and run
# ---------------------------------------------------------------------------


def prepare(case, seed):
    kind = case["kind"]
    if kind == "pic":
        return SimpleNamespace(c=case, sim=_make_sim(case, seed))
    if kind == "load":
        host = []
        for s in (0, 1):
            host.append([a.cpu().pin_memory() for a in _particles(case, seed, s)])
        ids = torch.arange(host[0][0].numel(), dtype=torch.int32).pin_memory()
        return SimpleNamespace(c=case, host=host, ids=ids.numpy().view(np.uint32),
                               sim=pg.Sim(_workload(case), capacity=_n_particles(case), hit_capacity=1 << 16))
    if kind == "batch":
        mem = [_member(case, k) for k in range(case["members"])]
        b = pg.Batch([_workload(m) for m in mem], capacities=[_n_particles(m) for m in mem], hit_capacity=1 << 12)
        for k, (m, view) in enumerate(zip(mem, b.members)):
            for s in (0, 1):
                view.load(s, *[a.cpu().numpy() for a in _particles(m, 64 * int(seed) + k, s)], v_at_t0=True)
        b.step(0)
        return SimpleNamespace(c=case, batch=b)
    if kind == "deposit":
        x, y = _deposit_inputs(case, seed)
        return SimpleNamespace(c=case, x=x, y=y, f=_entry("pic_deposit_static"))
    if kind == "unet":
        net = pg.Unet(case["batch"], case["height"], case["width"])
        net.set_params(_params(seed))
        x, t = _net_inputs(case, seed)
        return SimpleNamespace(c=case, net=net, x=x, t=t)
    x, dy, w, b = _layer_inputs(case, seed)
    op, co, ci = case["op"], case["cout"], case["cin"]
    name = {"conv": "pic_conv3x3_bf16", "wgrad": "pic_conv3x3_wgrad_bf16", "upconv": "pic_upconv_bf16",
            "upback": "pic_upconv_back_bf16", "upwgrad": "pic_upconv_wgrad_bf16"}[op]
    if op == "conv":
        w = w.to(torch.bfloat16)
        out = [torch.empty(x.shape[:3] + (co,), dtype=torch.bfloat16, device=x.device)]
    elif op == "upconv":
        out = [torch.empty(dy.shape, dtype=torch.bfloat16, device=x.device)]
    elif op == "upback":
        out = [torch.empty(x.shape, dtype=torch.bfloat16, device=x.device)]
    else:
        out = [torch.empty(w.shape, device=x.device)]
        if op == "upwgrad":
            out.append(torch.empty((co,), device=x.device))
    return SimpleNamespace(c=case, x=x, dy=dy, w=w, b=b, out=out, name=name, f=_entry(name))


def _deposit_inputs(c, seed):
    """Positions all over the grid, a few of them outside it (dropped, or wrapped where periodic)."""
    d = _dev()
    g = torch.Generator(device=d).manual_seed(int(seed))
    u = [torch.rand(c["n"], generator=g, device=d, dtype=torch.float64) for _ in range(2)]
    return [(1.002 * u[0] - 0.001) * c["nx"], (1.002 * u[1] - 0.001) * c["ny"]]


def run(state):
    c = state.c
    kind = c["kind"]
    if kind == "pic":
        state.sim.step(c["steps"])
        return _field(state.sim)
    if kind == "load":
        for s in (0, 1):
            state.sim.load(s, *[a.numpy() for a in state.host[s]], ids=state.ids)
        state.sim.step(c["steps"])
        return _field(state.sim)
    if kind == "batch":
        state.batch.step(c["steps"])
        return [_field(m) for m in state.batch.members]
    stream = torch.cuda.current_stream().cuda_stream
    if kind == "deposit":
        rho = torch.empty((c["nx"] + (not c["px"]), c["ny"] + (not c["py"])), dtype=torch.float64, device="cuda")
        _ok(state.f(c["nx"], c["ny"], int(c["px"]), int(c["py"]), c["n"], state.x.data_ptr(), state.y.data_ptr(),
                    0.01, rho.data_ptr(), stream), "pic_deposit_static")
        return rho
    if kind == "unet":
        if not c["grad"]:
            return state.net.forward(state.x)
        loss, grad = state.net.gradients(state.x, state.t)
        return [loss, grad]
    B, H, W, ci, co, op = (c[k] for k in ("batch", "height", "width", "cin", "cout", "op"))
    x, dy, w, b, out = (t.data_ptr() if isinstance(t, torch.Tensor) else t
                        for t in (state.x, state.dy, state.w, state.b, state.out))
    if op == "conv":
        st = state.f(0, B, H, W, x, ci, 0, ci, w, b, 1, out[0].data_ptr(), co, 0, co, stream)
    elif op == "upconv":
        st = state.f(0, B, H, W, x, ci, w, b, out[0].data_ptr(), co, 0, co, stream)
    elif op == "upback":
        st = state.f(0, B, H, W, dy, co, 0, co, w, out[0].data_ptr(), ci, stream)
    else:
        for o in out:
            o.zero_()                       # the gradients are added to what is there
        if op == "wgrad":
            st = state.f(0, B, H, W, dy, x, ci, 0, ci, co, out[0].data_ptr(), stream)
        else:
            st = state.f(0, B, H, W, x, ci, dy, co, 0, co, out[0].data_ptr(), out[1].data_ptr(), stream)
    _ok(st, state.name)
    return out


# ---------------------------------------------------------------------------
# what a pass cannot do without
# ---------------------------------------------------------------------------


def _pic_work(c):
    n, nodes = 2 * _n_particles(c), c["nx"] * c["ny"]
    # a step moves 20 bytes of state per particle in and out; per node the
    # deposit is written and read (two 8-byte sums), the potential read and
    # written (8 bytes each way) and the field written and read (8 bytes)
    step = dict(bytes=40 * n + 64 * nodes, flops=60 * n + 200 * nodes)
    w = {k: c["steps"] * v for k, v in step.items()}
    if c["kind"] == "load":
        w["bytes"] += 36 * n + 24 * n       # the host state in, the device state out
    w["bytes"] += 16 * nodes                # the field handed back
    return w


def _conv_flops(c):
    if c["op"].startswith("up"):
        return 2 * 4 * c["cin"] * c["cout"] * c["batch"] * c["height"] * c["width"]
    return 2 * 9 * c["cin"] * c["cout"] * c["batch"] * c["height"] * c["width"]


def work(case):
    kind = case["kind"]
    if kind in ("pic", "load"):
        return _pic_work(case)
    if kind == "batch":
        ws = [_pic_work(_member(case, k)) for k in range(case["members"])]
        return {k: sum(w[k] for w in ws) for k in ("bytes", "flops")}
    if kind == "deposit":
        return dict(bytes=16 * case["n"] + 8 * case["nx"] * case["ny"], flops=20 * case["n"])
    if kind == "unet":
        px = case["batch"] * case["height"] * case["width"]
        fl, k, acts = 0, 0, 0.0
        for i, (what, ci, co) in enumerate(_layers()):
            lv = i // 2 if i < 8 else (2 - (i - 8) // 3 if what != "head" else 0)
            p = px / 4 ** lv
            fl += {"conv": 18, "up": 2, "head": 2}[what] * ci * co * p
            k += ({"conv": 9, "up": 4, "head": 1}[what] * ci + 1) * co
            acts += 2 * co * p
        if case["grad"]:   # gradients of data and weights; every activation kept and read once more
            return dict(bytes=12 * px + 4 * k + 4 * k + 2 * acts, flops=3 * fl)
        return dict(bytes=12 * px + 2 * k, flops=fl)
    B, H, W, ci, co = (case[k] for k in ("batch", "height", "width", "cin", "cout"))
    px, q = B * H * W, 4 if case["op"].startswith("up") else 1
    nw = (4 if q == 4 else 9) * ci * co
    data = 2 * px * ci + 2 * q * px * co
    wb = {"conv": 2, "wgrad": 4, "upconv": 4, "upback": 4, "upwgrad": 4}[case["op"]]
    return dict(bytes=data + wb * nw, flops=_conv_flops(case))


# ---------------------------------------------------------------------------
# the same in FP64
# ---------------------------------------------------------------------------


def _basis(n, periodic, d):
    """Orthonormal eigenvectors (columns over all nodes) and eigenvalues of the 1-D second
    difference with periodic ends, or with zero at both end nodes of n cells."""
    if not periodic:
        i = torch.arange(n + 1, device=d, dtype=torch.float64)[:, None]
        k = torch.arange(1, n, device=d, dtype=torch.float64)[None, :]
        return math.sqrt(2.0 / n) * torch.sin(math.pi * i * k / n), 2 - 2 * torch.cos(math.pi * k[0] / n)
    i = torch.arange(n, device=d, dtype=torch.float64)[:, None]
    k = torch.arange(n, device=d)
    m = ((k + 1) // 2).double()
    a = 2 * math.pi * i * m / n
    v = torch.where(k % 2 == 1, torch.cos(a), torch.sin(a))
    v[:, 0] = 1.0
    if n % 2 == 0:
        v[:, n - 1] = torch.cos(math.pi * i[:, 0])
    return v / v.norm(dim=0), 2 - 2 * torch.cos(2 * math.pi * m / n)


class _Exact:
    """The step loop in FP64: bilinear weighting, leapfrog, absorption at the first
    conductor or wall face, Dirichlet Poisson solve, field by open edges."""

    def __init__(self, c):
        d = self.d = _dev()
        self.c = c
        nx, ny, px, py = c["nx"], c["ny"], c["px"], c["py"]
        self.shape = (nx + (not px), ny + (not py))
        cond = _conductor(c)
        D = np.zeros(self.shape, bool)
        g, el = np.zeros(self.shape), np.zeros(self.shape)
        if not py:
            D[:, 0] = D[:, -1] = True
        if not px:
            D[0] = D[-1] = True
            g[0], g[-1], el[-1] = 0.0, c["phi_el"], 1.0
        ci, cj = np.nonzero(cond)
        for a in (0, 1):
            for b in (0, 1):
                at = ((ci + a) % self.shape[0] if px else ci + a, (cj + b) % self.shape[1] if py else cj + b)
                D[at], g[at], el[at] = True, c["phi_el"], 1.0
        t = lambda a: torch.from_numpy(a).to(d)   # noqa: E731
        self.free, self.g0, self.el = t(~D), t(np.where(D, g, 0.0)), t(el)
        self.plasma = t(~cond)
        pad = np.zeros((nx + 2, ny + 2), bool)
        pad[1:-1, 1:-1] = ~cond
        if px:
            pad[0], pad[-1] = pad[-2], pad[1]
        if py:
            pad[:, 0], pad[:, -1] = pad[:, -2], pad[:, 1]
        n0, n1 = self.shape   # an edge is open when a plasma cell borders it
        up = pad[1:, :-1] | pad[1:, 1:]        # from node (i, j) to (i + 1, j)
        rt = pad[:-1, 1:] | pad[1:, 1:]        # from node (i, j) to (i, j + 1)
        self.ox, self.oy = t(up[:n0, :n1]), t(rt[:n0, :n1])
        self.vx, lx = _basis(nx, px, d)
        self.vy, ly = _basis(ny, py, d)
        lam = lx[:, None] + ly[None, :]
        self.ilam = torch.where(lam > 1e-14, 1 / lam.clamp(min=1e-14), torch.zeros_like(lam))
        self.phi = self.g0.clone()
        self.bottom = torch.zeros((2, ny), device=d, dtype=torch.float64)
        self.n = 0

    def shift(self, a, dim, by):
        """a at the neighbour by along dim (zero beyond a wall)."""
        r = torch.roll(a, -by, dim)
        if not (self.c["px"], self.c["py"])[dim]:
            r.select(dim, -1 if by > 0 else 0).zero_()
        return r

    def lap(self, a):
        return 4 * a - sum(self.shift(a, k, s) for k in (0, 1) for s in (-1, 1))

    def solve(self, rho):
        g = self.g0 + (self.c["rf"] * math.sin(0.01 * 0.1 * self.n)) * self.el
        b = (rho - self.lap(torch.where(self.free, torch.zeros_like(g), g))) * self.free
        if self.c["px"] and self.c["py"]:
            b = b - b.mean()
        x = torch.where(self.free, self.phi, torch.zeros_like(g))
        r = b - self.lap(x) * self.free
        p, rz_old, stop = None, 1.0, 1e-12 * float(b.norm())
        for _ in range(400):
            if float(r.norm()) <= stop:
                break
            z = self.vx @ ((self.vx.T @ r @ self.vy) * self.ilam) @ self.vy.T * self.free
            rz = (r * z).sum()
            p = z if p is None else z + (rz / rz_old) * p
            q = self.lap(p) * self.free
            al = rz / (p * q).sum()
            x, r, rz_old = x + al * p, r - al * q, rz
        self.phi = torch.where(self.free, x, g)
        e = []
        for k, o in ((0, self.ox), (1, self.oy)):
            dphi = torch.where(o, self.shift(self.phi, k, 1) - self.phi, torch.zeros_like(g))
            of = o.double()
            if not (self.c["px"], self.c["py"])[k]:   # no edge beyond the last node
                dphi.select(k, -1).zero_()
                of.select(k, -1).zero_()
            s, cnt = dphi + self.shift(dphi, k, -1), of + self.shift(of, k, -1)
            e.append(torch.where(cnt > 0, -s / cnt.clamp(min=1), torch.zeros_like(s)))
        self.e = e

    def corners(self, x, y):
        i, j = x.floor(), y.floor()
        fx, fy = x - i, y - j
        i, j = i.long(), j.long()
        for a in (0, 1):
            for b in (0, 1):
                ii, jj = (i + a) % self.shape[0], (j + b) % self.shape[1]
                yield ii * self.shape[1] + jj, (fx if a else 1 - fx) * (fy if b else 1 - fy)

    def deposit(self, p):
        rho = torch.zeros(self.shape[0] * self.shape[1], device=self.d, dtype=torch.float64)
        for s, q in ((0, -1.0), (1, 1.0)):
            for at, w in self.corners(p[s][0], p[s][1]):
                rho.index_add_(0, at, w * (q / self.c["ppc"]))
        rho = rho.view(self.shape)
        if self.c["surface"]:
            sig = 0.5 * (self.bottom[1] - self.bottom[0]) / self.c["ppc"]
            row = torch.zeros(self.c["ny"] + 1, device=self.d, dtype=torch.float64)
            row[:-1] += sig
            row[1:] += sig
            if self.c["py"]:
                row[0] += row[-1]
                row = row[:-1]
            rho[self.c["nx"] - 1] += row
        return rho

    def gather(self, x, y):
        e = [torch.zeros_like(x), torch.zeros_like(x)]
        for at, w in self.corners(x, y):
            for k in (0, 1):
                e[k] += w * self.e[k].reshape(-1)[at]
        return e

    def is_plasma(self, i, j):
        c = self.c
        if c["px"]:
            i = i % c["nx"]
        if c["py"]:
            j = j % c["ny"]
        inside = (i >= 0) & (i < c["nx"]) & (j >= 0) & (j < c["ny"])
        return inside & self.plasma[i.clamp(0, c["nx"] - 1), j.clamp(0, c["ny"] - 1)]

    def move(self, s, p):
        """One leapfrog step of a species [x, y, vx, vy, id] (moves of at most one cell)."""
        x, y, vx, vy, ids = p
        al = (-1.0, 1.0 / self.c["mass"])[s]
        ex, ey = self.gather(x, y)
        vx, vy = vx + al * 0.1 * ex, vy + al * 0.1 * ey
        x1, y1 = x + 0.1 * vx, y + 0.1 * vy
        i, j = x.floor().long(), y.floor().long()
        cx, cy = x1.floor().long() - i, y1.floor().long() - j
        tx = ((i + (cx > 0)).double() - x).abs() * vy.abs()
        ty = ((j + (cy > 0)).double() - y).abs() * vx.abs()
        xfirst = (cx != 0) & ((cy == 0) | (tx <= ty))
        ia, ja = torch.where(xfirst, i + cx, i), torch.where(xfirst, j, j + cy)
        first, second = self.is_plasma(ia, ja), self.is_plasma(i + cx, j + cy)
        dead = ~(first & second)
        if self.c["surface"]:
            # through the x = nx face: by the x crossing, in the column it happens in
            hit = dead & (i + cx >= self.c["nx"]) & (xfirst | first)
            col = torch.where(xfirst, j, j + cy)[hit] % self.c["ny"]
            self.bottom[s] += torch.bincount(col, minlength=self.c["ny"])
        if self.c["px"]:
            x1 = x1 % self.c["nx"]
        if self.c["py"]:
            y1 = y1 % self.c["ny"]
        new = [a[~dead] for a in (x1, y1, vx, vy, ids)]
        if s == 1 and self.c["recycle"]:
            new = [torch.cat(ab) for ab in zip(new, self.reborn(ids[dead]))]
        return new

    def reborn(self, ids):
        """Thermal ions in the bulk by Philox4x32-10 draws of (id, step)."""
        ids = ids.cpu().numpy().astype(np.uint64)
        m32 = np.uint64(0xFFFFFFFF)

        def philox(k):
            q = [ids.copy(), np.full_like(ids, self.n), np.full_like(ids, 1), np.full_like(ids, k)]
            k0, k1 = np.uint64(11), np.uint64(0)
            for _ in range(10):
                a, b = np.uint64(0xD2511F53) * q[0], np.uint64(0xCD9E8D57) * q[2]
                q = [(b >> np.uint64(32)) ^ q[1] ^ k0, b & m32, (a >> np.uint64(32)) ^ q[3] ^ k1, a & m32]
                k0, k1 = (k0 + np.uint64(0x9E3779B9)) & m32, (k1 + np.uint64(0xBB67AE85)) & m32
            return q

        r, q = philox(0), philox(1)
        u = lambda w: (w >> np.uint64(8)).astype(np.float64) * 2.0 ** -24   # noqa: E731
        rows = self.c["nx"] - self.c["depth"]
        x = ((r[0] * np.uint64(rows)) >> np.uint64(32)).astype(np.float64) + u(r[2])
        y = ((r[1] * np.uint64(self.c["ny"])) >> np.uint64(32)).astype(np.float64) + u(r[3])
        rad = np.sqrt(-2 * np.log(u(q[0]) + 2.0 ** -24)) * math.sqrt(self.c["tau"] / self.c["mass"])
        v = [rad * np.cos(2 * np.pi * u(q[1])), rad * np.sin(2 * np.pi * u(q[1]))]
        return [torch.from_numpy(a).to(self.d) for a in (x, y, *v, ids.astype(np.int64))]

    def go(self, seed, v_at_t0):
        p = []
        for s in (0, 1):
            a = _particles(self.c, seed, s)
            p.append(a + [torch.arange(a[0].numel(), device=self.d)])
        self.solve(self.deposit(p))
        for s, al in ((0, -1.0), (1, 1.0 / self.c["mass"])):
            if v_at_t0:
                e = self.gather(p[s][0], p[s][1])
                p[s][2], p[s][3] = p[s][2] - 0.05 * al * e[0], p[s][3] - 0.05 * al * e[1]
        for _ in range(self.c["steps"]):
            p = [self.move(s, p[s]) for s in (0, 1)]
            self.n += 1
            self.solve(self.deposit(p))
        return torch.stack(self.e)


def _conv64(x, w, b):
    """3x3 convolution in NHWC, w [out][3][3][in], as nine matrix products."""
    B, H, W, ci = x.shape
    xp = torch.nn.functional.pad(x, (0, 0, 1, 1, 1, 1))
    out = None
    for t in range(9):
        y = xp[:, t // 3:t // 3 + H, t % 3:t % 3 + W].reshape(-1, ci) @ w[:, t // 3, t % 3].T
        out = y if out is None else out + y
    return out.view(B, H, W, -1) + b


def _up64(x, w, b):
    """Transposed 2x2 stride-2 convolution in NHWC, w [2][2][in][out]."""
    B, H, W, ci = x.shape
    y = torch.einsum("bhwi,acio->bhawco", x, w)
    return y.reshape(B, 2 * H, 2 * W, -1) + b


def _unet64(flat, x):
    at, ws = 0, []
    for kind, ci, co in _layers():
        n = {"conv": co * 9 * ci, "up": 4 * ci * co, "head": ci}[kind]
        shape = {"conv": (co, 3, 3, ci), "up": (2, 2, ci, co), "head": (ci,)}[kind]
        ws.append((flat[at:at + n].view(shape), flat[at + n:at + n + co]))
        at += n + co
    skips, h = [], x
    for lv in range(4):
        for k in (0, 1):
            h = torch.relu(_conv64(h, *ws[2 * lv + k]))
        if lv < 3:
            skips.append(h)
            B, H, W, ch = h.shape
            h = h.view(B, H // 2, 2, W // 2, 2, ch).mean(dim=(2, 4))
    for q, lv in enumerate((2, 1, 0)):
        h = torch.cat([_up64(h, *ws[8 + 3 * q]), skips[lv]], dim=3)
        for k in (1, 2):
            h = torch.relu(_conv64(h, *ws[8 + 3 * q + k]))
    return h @ ws[-1][0] + ws[-1][1]


def exact(case, seed):
    kind = case["kind"]
    if kind in ("pic", "load"):
        return _Exact(case).go(seed, kind == "pic")
    if kind == "batch":
        return [_Exact(_member(case, k)).go(64 * int(seed) + k, True) for k in range(case["members"])]
    if kind == "deposit":
        c = case
        x, y = _deposit_inputs(c, seed)
        if c["px"]:
            x = x % c["nx"]
        if c["py"]:
            y = y % c["ny"]
        ok = (x >= 0) & (x < c["nx"]) & (y >= 0) & (y < c["ny"])
        x, y = x[ok], y[ok]
        n0, n1 = c["nx"] + (not c["px"]), c["ny"] + (not c["py"])
        rho = torch.zeros(n0 * n1, dtype=torch.float64, device=x.device)
        i, j = x.floor().long(), y.floor().long()
        fx, fy = x - i, y - j
        for a in (0, 1):
            for b in (0, 1):
                at = ((i + a) % n0) * n1 + (j + b) % n1
                rho.index_add_(0, at, 0.01 * (fx if a else 1 - fx) * (fy if b else 1 - fy))
        return rho.view(n0, n1)
    if kind == "unet":
        x, t = (a.double() for a in _net_inputs(case, seed))
        flat = torch.from_numpy(_params(seed)).to(x.device).double()
        if not case["grad"]:
            with torch.no_grad():
                return torch.cat([_unet64(flat, x[k:k + 1]) for k in range(case["batch"])])
        flat.requires_grad_(True)
        loss, n = 0.0, t.numel()
        for k in range(case["batch"]):   # sample by sample: the activations of one at a time
            part = ((_unet64(flat, x[k:k + 1]) - t[k:k + 1]) ** 2).sum() / n
            part.backward()
            loss += float(part.detach())
        return [None, flat.grad]         # (the loss of a 16-bit network is not the FP64 one's to 9 digits)
    x, dy, w, b = _layer_inputs(case, seed)
    op, ci, co = case["op"], case["cin"], case["cout"]
    xd, yd = x.double(), dy.double()
    if op == "conv":
        w64 = w.to(torch.bfloat16).double().view(co, 3, 3, ci)
        return [torch.relu(_conv64(xd, w64, b.double()))]
    if op == "wgrad":
        B, H, W, _ = x.shape
        xp = torch.nn.functional.pad(xd, (0, 0, 1, 1, 1, 1))
        cols = [yd.reshape(-1, co).T @ xp[:, t // 3:t // 3 + H, t % 3:t % 3 + W].reshape(-1, ci) for t in range(9)]
        return [torch.stack(cols, dim=1).reshape(-1)]
    w64 = w.double().view(2, 2, ci, co)
    B, H, W, _ = x.shape
    y6 = yd.view(B, H, 2, W, 2, co)
    if op == "upconv":
        return [_up64(xd, w64, b.double())]
    if op == "upback":
        return [torch.einsum("bhawco,acio->bhwi", y6, w64)]
    return [torch.einsum("bhwi,bhawco->acio", xd, y6).reshape(-1), yd.sum(dim=(0, 1, 2))]
