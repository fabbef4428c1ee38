"""The timed cases: what users of this package have it do, over the range of
sizes, storage forms and options in use.

Kinds of case:

* ``lattice``: one domain (``lbm.Lattice``). A pass advances it by ``steps``
  time steps (after re-setting it from a pinned host density with ``restart``),
  reads the observables record and the fields (rho, u_x, u_y).
* ``batch``: a sweep of channels (``lbm.Batch``). A pass advances all of them
  and reads every domain's observables and fields.
* ``train``: one training step of the warm-start U-Net (``surrogate.UNet``) as
  ``surrogate.train`` runs it.
* ``conv``: one 3x3 convolution layer of that network through the C ABI:
  forward, input gradient, weight and bias gradients.
"""
import ctypes
import math

import numpy as np
import torch

from paper_0708_4182_gb300 import lbm, surrogate
from paper_0708_4182_gb300 import workloads as wl

STORAGE = {"fp32": lbm.LBM_FP32, "fp32dev": lbm.LBM_FP32_DEV, "fp16dev": lbm.LBM_FP16_DEV, "bf16dev": lbm.LBM_BF16_DEV}
NODE_BYTES = {"fp32": 36, "fp32dev": 36, "fp16dev": 20, "bf16dev": 20}
FLOPS_PER_NODE_STEP = 250
MOST_NODE_STEPS = 16384 * 4096 * 10  # a drawn case does no more than the largest listed one
OBS = ("mass", "flux_Q", "mom_x", "mom_y", "max_u", "min_rho")


def lattice(name, nx, ny, storage, steps, **more):
    c = dict(kind="lattice", nx=nx, ny=ny, storage=storage, steps=steps, tau=1.0, level=8, amp=0, shape="slab",
             body=1e-6, obs_every=0, restart=False)
    c.update(more)
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # the paper's sessile droplet (contact angle against the electric force): the smallest domain
        lattice("droplet_128x64", 128, 64, "fp32", 1000, shape="droplets", body=0.0),
        # rough-wall channel run to steady flux: one convergence interval
        lattice("rough_1024x128", 1024, 128, "fp32dev", 1000, amp=8),
        # ragged domain at the paper's tau = 0.9, watched closely: few steps per call, fused observables
        lattice("ragged_301x67", 301, 67, "fp32", 20, amp=4, tau=0.9, obs_every=10),
        # the smallest call: one step at a time, the fields read after each (a movie, a coupled code)
        lattice("single_step_520x90", 520, 90, "fp32dev", 1, amp=6),
        # the precision study's crop in 16-bit storage
        lattice("crop_1024x256", 1024, 256, "fp16dev", 500, amp=6, shape="droplets"),
        # end to end: a host density is set, then every step's observables are recorded
        lattice("observed_4096x2048", 4096, 2048, "fp32dev", 10, amp=6, shape="droplets", obs_every=1, restart=True),
        # the benchmark channel, in its storage form
        lattice("droplet_row_16384x4096", 16384, 4096, "fp32dev", 10, amp=6, shape="droplets"),
        # large channel in 16-bit storage (twice the nodes in the same memory)
        lattice("large_8192x4096", 8192, 4096, "bf16dev", 20, amp=6, shape="droplets"),
        # the batched sweep: uneven channels, force levels and roughness
        dict(name="sweep_64_uneven", kind="batch", count=64, sizes="uneven", storage="fp32", steps=50, body=1e-6),
        # the warm-started sweep of equal channels: part of a convergence interval
        dict(name="sweep_64_256x64", kind="batch", count=64, sizes="256x64", storage="fp32dev", steps=250, body=1e-5),
        # one training step of the warm-start network at its batch and tile size
        dict(name="train_16x64x256", kind="train", batch=16, height=64, width=256),
        # one decoder layer of that network, forward and backward
        dict(name="conv_192_64_32x128", kind="conv", n=16, ci=192, co=64, h=32, w=128),
    ]


# ------------------------------------------------------------------ more cases of the same ranges

def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _draw_lattice(rng):
    storage = rng.choice(list(STORAGE))
    nx, ny = _log(rng, 64, 16384), _log(rng, 32, 4096)
    if "16" in storage:
        nx = max(64, nx // 8 * 8)  # 16-bit storage takes multiples of 8
    steps = min(_log(rng, 1, 1000), max(1, MOST_NODE_STEPS // (nx * ny)))
    return lattice(None, nx, ny, storage, steps, tau=rng.choice([1.0, 1.0, 1.0, 0.9]), level=rng.randint(0, 15),
                   amp=rng.randint(0, 8), shape=rng.choice(["slab", "droplets"]), body=rng.choice([1e-6, 1e-5]),
                   obs_every=rng.choice([0, 0, 0, 1, 10, 100]), restart=rng.random() < 0.15)


def _draw_batch(rng):
    sizes = rng.choice(["uneven", "256x64"])
    count = rng.randint(4, 64)
    nodes = count * (16384 if sizes == "256x64" else 185000)
    steps = min(_log(rng, 2, 1000), max(2, 500_000_000 // nodes))
    return dict(kind="batch", count=count, sizes=sizes, storage=rng.choice(["fp32", "fp32dev"] if sizes == "uneven" else list(STORAGE)),
                steps=steps, body=rng.choice([1e-6, 1e-5]))


def _draw_train(rng):
    return dict(kind="train", batch=rng.randint(2, 16), height=rng.choice([32, 64]), width=256)


def _draw_conv(rng):
    level, ci, co = rng.choice([(0, 32, 32), (1, 32, 64), (1, 64, 64), (2, 64, 128), (2, 128, 128), (3, 128, 256),
                                (3, 256, 256), (2, 384, 128), (1, 192, 64), (0, 96, 32)])
    return dict(kind="conv", n=rng.randint(1, 16), ci=ci, co=co, h=rng.choice([32, 64]) >> level, w=256 >> level)


def draw(rng):
    return rng.choice([_draw_lattice] * 6 + [_draw_batch] * 2 + [_draw_train] + [_draw_conv])(rng)


# ------------------------------------------------------------------ inputs

def _mask(nx, ny, amp, seed):
    """The rough-wall channel mask of ``workloads.channel_mask`` on the GPU."""
    amp = max(0, min(amp, (ny - 3) // 2))
    ys = torch.arange(ny, device="cuda")[:, None]
    solid = ((ys == 0) | (ys == ny - 1)).expand(ny, nx)
    if amp > 0:
        seeder = wl.SplitMix64(seed)
        b, t = (torch.as_tensor(wl.wall_profile(nx, amp, wl.SplitMix64(seeder.next()))).cuda()[None, :] for _ in range(2))
        solid = solid | ((ys >= 1) & (ys <= b)) | ((ys <= ny - 2) & (ys >= ny - 1 - t))
    return solid.to(torch.uint8).contiguous()


def _density(nx, ny, shape, amp, mask, seed):
    """Liquid slab up to the roughness crests, or a row of sessile droplets of
    radius 20 (as many as fit at pitch 128), tanh edges, 1e-3 perturbation."""
    d = torch.float64
    if shape == "slab":
        amp = max(0, min(amp, (ny - 3) // 2))
        fill = max(0.1, 1.0 - 2.0 * (amp + 1) / (ny - 2))
        dist = ((torch.arange(ny, device="cuda", dtype=d) - 0.5 * (ny - 1)).abs() - 0.5 * fill * (ny - 2))[:, None]
    else:
        pitch = 128 if nx >= 128 else nx
        x = torch.arange(nx, device="cuda", dtype=d) % pitch - 0.5 * pitch
        y = torch.arange(ny, device="cuda", dtype=d) - 0.5
        dist = torch.sqrt(x[None, :] ** 2 + y[:, None] ** 2) - min(20.0, 0.4 * pitch, 0.4 * ny)
    rho = 0.5 * (wl.RHO_L + wl.RHO_V) - 0.5 * (wl.RHO_L - wl.RHO_V) * torch.tanh(0.5 * dist)
    g = torch.Generator("cuda").manual_seed(seed)
    xi = torch.rand((ny, nx), generator=g, device="cuda", dtype=torch.float32)
    return torch.where(mask != 0, 0.0, rho * (1.0 + 1e-3 * (2.0 * xi.to(d) - 1.0)))


def _model(tau, level, body):
    return dict(wl.PAPER, tau=tau, f_elec=wl.f_level(level), body_fx=body, body_fy=0.0)


def _lattice_inputs(case, seed):
    nx, ny = case["nx"], case["ny"]
    mask = _mask(nx, ny, case["amp"], seed)
    rho = _density(nx, ny, case["shape"], case["amp"], mask, seed)
    return mask, (rho.float().double() if case["restart"] else rho), _model(case["tau"], case["level"], case["body"])


def _batch_inputs(case, seed):
    """(nx, ny, mask, rho, model) of every channel. The sizes belong to the
    case; roughness, force level and perturbation come from the seed."""
    shapes = wl.batched_channels(case["count"], 0) if case["sizes"] == "uneven" else None
    rng = wl.SplitMix64(seed)
    out = []
    for k in range(case["count"]):
        level, s = rng.randint(0, 15), rng.next() & 0x7FFFFFFF
        if shapes:
            nx, ny, amp = shapes[k]["nx"], shapes[k]["ny"], shapes[k]["amp"]
        else:
            nx, ny, amp = 256, 64, 0
        mask = _mask(nx, ny, amp, s)
        out.append((nx, ny, mask, _density(nx, ny, "slab", amp, mask, s), _model(1.0, level, case["body"])))
    return out


def _weights(seed):
    """FP32 weights and biases of the network (He initialisation)."""
    g = torch.Generator().manual_seed(seed)
    return {name: ((torch.randn((co, ci, k, k), generator=g) * (2.0 / (ci * k * k)) ** 0.5).numpy(),
                   (0.05 * torch.randn(co, generator=g)).numpy())
            for name, (co, ci, k) in surrogate.layer_shapes().items()}


def _train_inputs(case, seed):
    g = torch.Generator("cuda").manual_seed(seed)
    b, h, w = case["batch"], case["height"], case["width"]
    mask = (torch.rand((b, h, w), generator=g, device="cuda") < 0.15).float()
    level = torch.rand((b, 1, 1), generator=g, device="cuda").expand(b, h, w)
    fill = (0.5 + 0.5 * torch.rand((b, 1, 1), generator=g, device="cuda")).expand(b, h, w)
    planes = torch.stack([mask, level, fill], 1).contiguous()
    targets = torch.randn((b, 3, h, w), generator=g, device="cuda") * (mask[:, None] == 0)
    return planes, targets


def _conv_inputs(case, seed):
    g = torch.Generator("cuda").manual_seed(seed)
    n, ci, co, h, w = (case[k] for k in ("n", "ci", "co", "h", "w"))
    x = torch.relu(torch.randn((n, h, w, ci), generator=g, device="cuda")).to(torch.bfloat16)
    dy = torch.randn((n, h, w, co), generator=g, device="cuda").to(torch.bfloat16)
    wt = (torch.randn((co, ci, 3, 3), generator=g, device="cuda") * (2.0 / (9 * ci)) ** 0.5).to(torch.bfloat16).float()
    bias = 0.1 * torch.randn(co, generator=g, device="cuda")
    return x, dy, wt, bias


def _ptr(t):
    return ctypes.c_void_p(t.data_ptr())


LOSS_WEIGHTS = (1.0, 1.0, 0.25)


def prepare(case, seed):
    kind = case["kind"]
    if kind == "lattice":
        mask, rho, model = _lattice_inputs(case, seed)
        lat = lbm.Lattice(case["nx"], case["ny"], storage=STORAGE[case["storage"]], obs_every=case["obs_every"], **model)
        lat.set_geometry(mask)
        lat.set_rho(rho)
        host = rho.float().cpu().pin_memory().numpy() if case["restart"] else None
        return dict(case=case, lat=lat, host=host)
    if kind == "batch":
        doms = _batch_inputs(case, seed)
        b = lbm.Batch([dict(nx=nx, ny=ny, storage=STORAGE[case["storage"]], **m) for nx, ny, _, _, m in doms])
        for (_, _, mask, rho, _), d in zip(doms, b.domains):
            d.set_geometry(mask)
            d.set_rho(rho)
        if case["sizes"] == "uneven":
            b.set_tile_rows(64)  # the height the autotuner picks on the full sweep
        return dict(case=case, batch=b)
    if kind == "train":
        planes, targets = _train_inputs(case, seed)
        net = surrogate.UNet(batch=case["batch"], height=case["height"], width=case["width"])
        net.set_weights(_weights(seed))
        net.make_train_graph(LOSS_WEIGHTS, [1e-4])
        return dict(case=case, net=net, planes=planes, targets=targets)
    x, dy, wt, bias = _conv_inputs(case, seed)
    lib = surrogate.load_unet()
    co, ci = case["co"], case["ci"]
    stream = ctypes.c_void_p(torch.cuda.current_stream().cuda_stream)
    packs = []
    for transpose in (0, 1):
        p = torch.empty(int(lib.unet_conv_pack_elems(co, ci, transpose)), dtype=torch.bfloat16, device="cuda")
        if lib.unet_conv_pack(_ptr(wt), co, ci, transpose, _ptr(p), stream) != 0:
            raise RuntimeError("unet_conv_pack failed")
        packs.append(p)
    return dict(case=case, lib=lib, x=x, dy=dy, bias=bias, packs=packs, y=torch.empty_like(dy), dx=torch.empty_like(x),
                dw=torch.zeros((co, ci, 3, 3), device="cuda"), db=torch.zeros(co, device="cuda"))


# ------------------------------------------------------------------ one pass

def _record(o):
    return np.array([o[k] for k in OBS])


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "lattice":
        lat = state["lat"]
        if state["host"] is not None:
            lat.set_density_f32(state["host"])
        lat.step(case["steps"])
        f = lat.fields_device().float()
        # the record of the last observed step, or one of the state as it is after a long run
        out = dict(rho=f[0], u=f[1:])
        if case["obs_every"]:
            out["obs"] = _record(lat.obs_latest())
        elif case["steps"] >= 100:
            out["obs"] = _record(lat.observables())
        return out
    if kind == "batch":
        b = state["batch"]
        b.step(case["steps"])
        fields = [d.fields_device().float() for d in b.domains]
        return dict(obs=np.stack([_record(o) for o in b.observables()]), rho=torch.cat([f[0].reshape(-1) for f in fields]),
                    u=torch.cat([f[1:].reshape(-1) for f in fields]))
    if kind == "train":
        net = state["net"]
        net.replay_train_step(state["planes"], state["targets"])
        return dict(prediction=net.out, loss=net.loss_acc, gradients=net.flat["g"], weights=net.flat["w"])
    lib, n, ci, co, h, w = state["lib"], case["n"], case["ci"], case["co"], case["h"], case["w"]
    s = ctypes.c_void_p(torch.cuda.current_stream().cuda_stream)
    x, dy, y, dx, dw, db = (state[k] for k in ("x", "dy", "y", "dx", "dw", "db"))
    dw.zero_()
    db.zero_()
    if lib.unet_conv3x3(_ptr(x), ci, ci, _ptr(state["packs"][0]), _ptr(state["bias"]), _ptr(y), co, co, n, h, w, 1, s) or \
            lib.unet_conv3x3(_ptr(dy), co, co, _ptr(state["packs"][1]), None, _ptr(dx), ci, ci, n, h, w, 0, s) or \
            lib.unet_conv3x3_bwd_weight(_ptr(x), ci, ci, _ptr(dy), co, co, _ptr(dw), _ptr(db), n, h, w, s):
        raise RuntimeError("a convolution call failed")
    return dict(y=y, dx=dx, dw=dw, db=db)


# ------------------------------------------------------------------ what a pass cannot do without

def work(case):
    kind = case["kind"]
    if kind in ("lattice", "batch"):
        if kind == "lattice":
            nodes = case["nx"] * case["ny"]
        elif case["sizes"] == "uneven":
            nodes = sum(c["nx"] * c["ny"] for c in wl.batched_channels(case["count"], 0))
        else:
            nodes = case["count"] * 256 * 64
        # the state in and out once, the fields out once
        return {"bytes": nodes * (2 * NODE_BYTES[case["storage"]] + 12 + (4 if case.get("restart") else 0)),
                "flops": FLOPS_PER_NODE_STEP * nodes * case["steps"]}
    if kind == "train":
        px = case["batch"] * case["height"] * case["width"]
        flops, acts, params = 0, 0, 0
        for name, (co, ci, k) in surrogate.layer_shapes().items():
            p = px >> (0 if name == "head" else 2 * int(name[1]))
            flops += (2 if name == "e0a" else 3) * 2 * co * ci * k * k * p  # no input gradient of the first layer
            acts += 2 * co * p
            params += co * ci * k * k + co
        # planes and targets in, prediction out, weights and moments in and out, gradients out
        return {"bytes": 4 * px * 9 + params * 4 * 7, "flops": flops}
    n, ci, co, px = case["n"], case["ci"], case["co"], case["n"] * case["h"] * case["w"]
    return {"bytes": 2 * px * (ci + co) * 2 + 9 * ci * co * (2 + 2 + 4), "flops": 3 * 2 * 9 * ci * co * px}


# ------------------------------------------------------------------ the same in 64 bits

EX = (0, 1, 0, -1, 0, 1, -1, -1, 1)
EY = (0, 0, 1, 0, -1, 1, 1, -1, -1)
OPP = (0, 3, 4, 1, 2, 7, 8, 5, 6)
WT = (4 / 9,) + (1 / 9,) * 4 + (1 / 36,) * 4


def _at(a, dx, dy):
    """The array whose value at (x, y) is a(x + dx, y + dy), periodic."""
    return torch.roll(a, (-dy, -dx), (-2, -1)) if dx or dy else a


def _moments_and_force(f, solid, m):
    fluid = ~solid
    rho = f.sum(0)
    jx = (f[1] - f[3]) + (f[5] - f[7]) + (f[8] - f[6])
    jy = (f[2] - f[4]) + (f[5] - f[7]) + (f[6] - f[8])
    psi = torch.where(fluid, -m["rho0"] * torch.expm1(-rho / m["rho0"]), 0.0)
    s = solid.to(torch.float64)
    ax, ay, bx, by = (torch.zeros_like(rho) for _ in range(4))
    for a in range(1, 9):
        k = 1.0 if a <= 4 else 0.5
        p, q = _at(psi, EX[a], EY[a]), _at(s, EX[a], EY[a])
        if EX[a]:
            ax += k * EX[a] * p
            bx += k * EX[a] * q
        if EY[a]:
            ay += k * EY[a] * p
            by += k * EY[a] * q
    fx = -psi * (m["G"] * ax + m["G_wall"] * bx) + rho * m["body_fx"]
    fy = -psi * (m["G"] * ay + m["G_wall"] * by) + rho * m["body_fy"]
    wet = fluid & (rho >= m["rho_c"])
    fx += torch.where(wet, m["f_elec"] * (_at(s, 1, 0) - _at(s, -1, 0)), 0.0)
    fy += torch.where(wet, m["f_elec"] * (_at(s, 0, 1) - _at(s, 0, -1)), 0.0)
    return rho, jx, jy, fx, fy


def _evolve(mask, rho0, m, steps, obs_every=0):
    """Fields after ``steps`` steps from a fluid at rest, and the record of the
    last observed step (or of the end). [..., ny, nx] arrays, one domain or
    several of one size (then f_elec is an array too)."""
    solid = mask != 0
    one = torch.where(solid, 1.0, 0.0).double()
    f = torch.stack([w * torch.where(solid, 0.0, rho0) for w in WT])
    inside = [_at(solid, -EX[a], -EY[a]) for a in range(9)]  # the pull source is solid
    rec = None
    for t in range(steps + 1):
        rho, jx, jy, fx, fy = _moments_and_force(f, solid, m)
        safe = rho + one
        if t == steps or (obs_every and t % obs_every == 0):
            px, py = (torch.where(solid, 0.0, j + 0.5 * v) for j, v in ((jx, fx), (jy, fy)))
            ux, uy = px / safe, py / safe
            if t < steps or not obs_every:
                d = (-2, -1)
                rec = torch.stack([rho.sum(d), ux.sum(d) / mask.shape[-1], px.sum(d), py.sum(d),
                                   (ux * ux + uy * uy).amax(d).sqrt(), torch.where(solid, math.inf, rho).amin(d)], -1)
            if t == steps:
                return rho, torch.stack([ux, uy]), rec
        ux, uy = (jx + m["tau"] * fx) / safe, (jy + m["tau"] * fy) / safe
        om = 1.0 - 1.5 * (ux * ux + uy * uy)
        for a in range(9):
            c = EX[a] * ux + EY[a] * uy
            f[a] += (WT[a] * rho * (om + c * (3.0 + 4.5 * c)) - f[a]) / m["tau"]
        f = torch.stack([torch.where(solid, 0.0, torch.where(inside[a], f[OPP[a]], _at(f[a], -EX[a], -EY[a])))
                         for a in range(9)])


def _pad(x):
    x = torch.cat([x[..., -1:], x, x[..., :1]], -1)
    return torch.nn.functional.pad(x, (0, 0, 1, 1))


def _conv(x, w, b=None):
    """3x3 convolution (periodic in x, zeros in y) as one matrix product per tap."""
    n, _, h, wd = x.shape
    xp = _pad(x)
    y = sum(torch.einsum("oi,nihw->nohw", w[:, :, i, j], xp[:, :, i:i + h, j:j + wd]) for i in range(3) for j in range(3))
    return y if b is None else y + b[None, :, None, None]


def _network(p, x):
    def layer(name, v):
        return torch.relu(_conv(v, *p[name]))

    skips = []
    for l in range(4):
        x = layer(f"e{l}b", layer(f"e{l}a", x))
        if l < 3:
            skips.append(x)
            x = torch.nn.functional.avg_pool2d(x, 2)
    for l in (2, 1, 0):
        x = torch.cat([x.repeat_interleave(2, -1).repeat_interleave(2, -2), skips[l]], 1)
        x = layer(f"d{l}b", layer(f"d{l}a", x))
    w, b = p["head"]
    return torch.einsum("oi,nihw->nohw", w[:, :, 0, 0], x) + b[None, :, None, None]


def exact(case, seed):
    kind = case["kind"]
    if kind == "lattice":
        mask, rho, m = _lattice_inputs(case, seed)
        # about 120 array operations a step, over memory or 5 us each
        if case["steps"] * max(8e-4, 1e-9 * case["nx"] * case["ny"]) > 15.0:
            return None
        rho, u, rec = _evolve(mask, rho, m, case["steps"], case["obs_every"])
        out = dict(rho=rho, u=u)
        if case["obs_every"] or case["steps"] >= 100:
            out["obs"] = rec
        return out
    if kind == "batch":
        doms = _batch_inputs(case, seed)
        if case["sizes"] == "256x64":  # all domains at once
            m = dict(doms[0][4], f_elec=torch.tensor([d[4]["f_elec"] for d in doms], device="cuda", dtype=torch.float64)[:, None, None])
            rho, u, rec = _evolve(torch.stack([d[2] for d in doms]), torch.stack([d[3] for d in doms]), m, case["steps"])
            return dict(obs=rec, rho=rho.reshape(-1), u=u.transpose(0, 1).reshape(-1))
        if case["steps"] * case["count"] * 1.2e-3 > 15.0:
            return None
        got = [_evolve(mask, rho, m, case["steps"]) for _, _, mask, rho, m in doms]
        return dict(obs=torch.stack([g[2] for g in got]), rho=torch.cat([g[0].reshape(-1) for g in got]),
                    u=torch.cat([g[1].reshape(-1) for g in got]))
    if kind == "train":
        planes, targets = _train_inputs(case, seed)
        p = {k: [torch.as_tensor(v).double().cuda().requires_grad_(True) for v in wb] for k, wb in _weights(seed).items()}
        pred = _network(p, planes.double())
        wc = torch.tensor(LOSS_WEIGHTS, dtype=torch.float64, device="cuda")[None, :, None, None]
        loss = (wc * (pred - targets.double()) ** 2).sum() / pred.numel()
        loss.backward()
        grads = torch.cat([p[k][0].grad.reshape(-1) for k in p] + [p[k][1].grad for k in p])
        return dict(prediction=pred.detach(), loss=loss.detach().reshape(1), gradients=grads, weights=None)
    x, dy, wt, bias = _conv_inputs(case, seed)
    x, dy = (v.double().permute(0, 3, 1, 2).contiguous() for v in (x, dy))
    x.requires_grad_(True)
    w = wt.double().requires_grad_(True)
    z = _conv(x, w)
    y = torch.relu(z.detach() + bias.double()[None, :, None, None])
    z.backward(dy)
    nhwc = lambda v: v.permute(0, 2, 3, 1).contiguous()  # noqa: E731
    return dict(y=nhwc(y), dx=nhwc(x.grad), dw=w.grad, db=dy.sum((0, 2, 3)))
