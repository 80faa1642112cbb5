"""The work a user of this package has it do, as cases whose time and results can be compared.

A case is one of five kinds, each through the package's public entry points:

``solve``       one problem: steps of the two-phase GPE solver on device-resident fields (FP32), or a
                whole short run from host arrays to host arrays (``whole``)
``batch``       many uneven 2D problems advanced together, their states packed as network tensors
``controller``  one checked window of the learned surrogate: network calls, then the solver as referee
``forward``     the surrogate network on a batch of states
``train``       training steps of the surrogate network

``exact`` gives what a pass returns in 64-bit arithmetic, written here with plain torch from the
equations of the method (staggered grid, TVD-RK3 flow step, Cahn-Hilliard RK2 or RK4 step).
"""
from __future__ import annotations

import functools
import math
import os

import numpy as np
import torch
import torch.nn.functional as F

from paper_2011_00814_gb300 import gpe2p, inputs
from paper_2011_00814_gb300 import surrogate as S

WEIGHTS = os.path.join(os.path.dirname(S.__file__), "data", "unet_two_drops_256.npz")
CH = S.CHANNELS


# ---------------------------------------------------------------------------
# the cases
# ---------------------------------------------------------------------------

def _solve(name, problem, nx, ny, nz, precision, steps, **kw):
    c = dict(name=name, kind="solve", problem=problem, nx=nx, ny=ny, nz=nz, precision=precision, steps=steps,
             compensated=False, whole=False, packed=False, iso=9 if nz == 0 else 15, conservative=False)
    c.update(kw)
    return c


def listed():
    return [
        # the smallest problem, the 64 x 64 drop of the first validation, as a script runs it:
        # host arrays in, a few steps, host arrays out
        _solve("drop 64 FP64 whole", "drop", 64, 64, 0, 64, 20, whole=True),
        # the fine mesh of the capillary-wave validation (57,600 steps there): walls, FP64, latency
        _solve("wave 128x64 FP64", "wave", 128, 64, 0, 64, 50),
        # the solver's K = 64 steps between two snapshots of the surrogate's problem
        _solve("two drops 256 FP32", "two_drops", 256, 256, 0, 32, 64, packed=True),
        # the axisymmetric falling drop at the paper's resolution, FP32 with the compensated phi
        # accumulation that the default policy switches on
        _solve("falling 400x1200 FP32", "falling", 400, 1200, 0, 32, 20, compensated=True),
        # Rayleigh-Taylor on the paper's grid in FP64, the reference run of its validation
        _solve("rayleigh 256x1024 FP64", "rt", 256, 1024, 0, 64, 4),
        # the batched workload: 96 uneven drops and bubbles, sides 64 to 512
        dict(name="batch 96 FP32", kind="batch", n=96, sides="64,128,192,256,384,512", precision=32, steps=8),
        # the largest: the 3D buoyant bubble of the benchmark
        _solve("bubble 256x256x512 FP32", "bubble", 256, 256, 512, 32, 2),
        # a 3D box of odd sizes, D3Q19, compensated accumulation
        _solve("bubble 101x75x130 FP32", "bubble", 101, 75, 130, 32, 8, compensated=True, iso=19),
        # 3D in FP64, periodic, D3Q27, the conservative Cahn-Hilliard form
        _solve("box 64x48x80 FP64", "box", 64, 48, 80, 64, 2, iso=27, conservative=True),
        # the surrogate in use: four calls, the last one checked against the solver
        dict(name="controller 256", kind="controller", n=256, calls=4, layout=0),
        # the network on a batch of states, as evaluation over many problems runs it
        dict(name="forward 256 batch 8", kind="forward", n=256, w=256, batch=8, channels="32,64,128,256", trained=True),
        # training at the minibatch the surrogate was trained with
        dict(name="train 256 batch 8", kind="train", n=256, w=256, batch=8, channels="32,64,128,256", steps=4),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["solve2", "solve2", "solve2", "solve3", "solve3", "batch", "controller", "forward", "train"])
    if kind == "solve2":
        problem = rng.choice(["drop", "two_drops", "wave", "rt", "falling"])
        prec = rng.choice([32, 32, 64])
        nx, ny = _log(rng, 24, 640), _log(rng, 24, 1200)
        steps = max(2, min(64, int(4.0e6 / (nx * ny))))
        whole = rng.random() < 0.2 and prec == 64
        c = _solve("", problem, nx, ny, 0, prec, steps, compensated=prec == 32 and rng.random() < 0.5, whole=whole,
                   packed=problem == "two_drops" and prec == 32 and rng.random() < 0.5,
                   conservative=problem not in ("falling",) and rng.random() < 0.2)
    elif kind == "solve3":
        prec = rng.choice([32, 32, 32, 64])
        hi = 230 if prec == 32 else 80
        nx, ny, nz = _log(rng, 24, hi), _log(rng, 24, hi), _log(rng, 24, 1.5 * hi)
        c = _solve("", rng.choice(["bubble", "box"]), nx, ny, nz, prec, 2 if nx * ny * nz > 1000000 else 4,
                   compensated=prec == 32 and rng.random() < 0.4, iso=rng.choice([15, 15, 19, 27]),
                   conservative=rng.random() < 0.2)
    elif kind == "batch":
        sides = sorted({_log(rng, 40, 520) for _ in range(5)})
        c = dict(kind="batch", n=rng.randint(3, 60), sides=",".join(str(s) for s in sides),
                 precision=rng.choice([32, 32, 32, 64]), steps=rng.randint(2, 6))
        if c["precision"] == 64:
            c["n"] = min(c["n"], 10)
    elif kind == "controller":
        c = dict(kind="controller", n=256, calls=rng.choice([2, 3, 4, 8]), layout=rng.randint(1, 1000))
    else:
        levels = rng.choice([2, 3, 4])
        base = rng.choice([16, 32, 64]) if levels < 4 else rng.choice([16, 32])
        q = 1 << (levels - 1)
        c = dict(kind=kind, n=q * _log(rng, 24 / q, 288 / q), w=q * _log(rng, 24 / q, 288 / q), batch=rng.randint(1, 8),
                 channels=",".join(str(base << l) for l in range(levels)))
        if kind == "forward":
            c["trained"] = False
        else:
            c["steps"] = rng.randint(1, 3)
    c.pop("name", None)
    return c


# ---------------------------------------------------------------------------
# problems: parameters and seeded initial fields
# ---------------------------------------------------------------------------

def _params(case):
    """The parameters of a ``solve`` case: the repository's workload of that name on the case's grid."""
    p, nx, ny, nz = case["problem"], case["nx"], case["ny"], case["nz"]
    if p == "drop":
        prm, _ = inputs.static_drop(16)
    elif p == "two_drops":
        prm, _ = inputs.two_drops(7, n=16)
    elif p == "wave":
        prm, _ = inputs.capillary_wave(128, 1920, 0.03125, 4.0e4)
    elif p == "rt":
        prm, _ = inputs.rayleigh_taylor(8, 32, variant="paper")
        dx = 1.0 / 256.0
        prm.update(dx=dx, W=4.0 * dx, dt=1.0 / 51200.0)
    elif p == "falling":
        prm, _ = inputs.falling_drop(2)
        prm.update(dx=1.0 / 50.0, dt=1.0 / 4000.0, cs=4000.0 / 50.0 / math.sqrt(3.0))
    else:
        prm, _ = inputs.bubble3d(8, 8, 8, R=32.0)
        if p == "box":
            prm.update(bc=("periodic",) * 3, g=(0.0, 0.0, 0.0))
    prm = dict(prm, nx=nx, ny=ny, nz=nz or 1, precision=case["precision"], iso=case["iso"],
               ch_advection=int(case["conservative"]))
    if nz:
        prm["dt"] = 0.9 * prm["dt"]
    return prm


def _axes(prm, dev):
    """Cell-centre and low-face coordinates per axis, shaped to broadcast over (z, y, x) or (y, x)."""
    d, dx = prm["dim"], prm["dx"]
    cen, face = [], []
    for a, n in enumerate((prm["nx"], prm["ny"], prm["nz"])[:d]):
        shp = [1] * d
        shp[d - 1 - a] = n
        i = torch.arange(n, dtype=torch.float64, device=dev).reshape(shp)
        cen.append((i + 0.5) * dx)
        face.append(i * dx)
    return cen, face


def _fields(prm, problem, seed, dev="cuda"):
    """A state in mid-run: the workload's interface (moved, sharper than its equilibrium width, with
    noise) and a smooth flow and pressure.  Torch FP64 tensors on the GPU, rounded to the working
    precision."""
    g = torch.Generator(device="cpu").manual_seed(int(seed) * 7919 + 11)
    rnd = lambda lo, hi: lo + (hi - lo) * float(torch.rand((), generator=g, dtype=torch.float64))  # noqa: E731
    d, W = prm["dim"], prm["W"] * rnd(0.65, 0.8)
    ext = [n * prm["dx"] for n in (prm["nx"], prm["ny"], prm["nz"])[:d]]
    per = [b == "periodic" for b in prm["bc"][:d]]
    cen, face = _axes(prm, dev)
    short = min(ext)
    if problem in ("rt", "wave"):
        a, o = (1, 0) if problem == "rt" else (0, 1)
        h = ext[a] * rnd(0.42, 0.58) + 0.03 * short * torch.cos(2.0 * math.pi * cen[o] / ext[o] + rnd(0, 1))
        phi = torch.tanh(2.0 * (cen[a] - h) / W)
    elif problem == "two_drops":
        c1 = [e * rnd(0.2, 0.4) for e in ext]
        c2 = [e * rnd(0.6, 0.8) for e in ext]
        phi = None
        for c in (c1, c2):
            r = torch.sqrt(sum((x - q) ** 2 for x, q in zip(cen, c)))
            t = torch.tanh(2.0 * (short * rnd(0.1, 0.2) - r) / W)
            phi = t if phi is None else torch.maximum(phi, t)
    else:
        c = [e * rnd(0.4, 0.6) for e in ext]
        if prm.get("axisym"):
            c[0] = 0.0
        r = torch.sqrt(sum((x - q) ** 2 for x, q in zip(cen, c)))
        phi = torch.tanh(2.0 * (short * rnd(0.2, 0.3) - r) / W)
        if problem in ("bubble", "box"):
            phi = -phi
    gg = torch.Generator(device=dev).manual_seed(int(seed))
    phi = phi + 5e-3 * (torch.rand(phi.shape, generator=gg, dtype=torch.float64, device=dev) - 0.5)
    U = 0.01 * prm["cs"] * rnd(0.8, 1.2)
    k = [(2.0 if q else 1.0) * math.pi * (1 + (a == 0)) / e for a, (q, e) in enumerate(zip(per, ext))]
    ph = [rnd(0.0, 6.0) if q else 0.0 for q in per]
    cs = [torch.cos(k[a] * cen[a] + ph[a]) for a in range(d)]
    sn = [torch.sin(k[a] * face[a] + ph[a]) for a in range(d)]
    cz = cs[2] if d == 3 else 1.0
    f = {"phi": phi,
         "u": (U * sn[0] * cs[1] * cz).expand(phi.shape),
         "v": (-U * k[0] / k[1] * cs[0] * sn[1] * cz).expand(phi.shape),
         "p": (0.01 * prm["rhoL"] * prm["cs"] ** 2 * cs[0] * cs[1] * cz).expand(phi.shape)}
    if d == 3:
        f["w"] = (0.5 * U * cs[0] * cs[1] * sn[2]).expand(phi.shape)
    for a, nm in enumerate("uvw"[:d]):
        f[nm] = f[nm].clone()
        if not per[a]:
            f[nm].select(d - 1 - a, 0).zero_()
    if prm["precision"] == 32:
        f = {key: v.float().double() for key, v in f.items()}
    return {key: v.contiguous() for key, v in f.items()}


@functools.lru_cache(maxsize=4)
def _batch_params(n, sides, precision):
    prms, _ = inputs.batch_instances(n=n, seed=0, sides=tuple(int(s) for s in sides.split(",")), precision=precision)
    # sides that are not square, as ragged domains are
    for k, p in enumerate(prms):
        if k % 5 == 3:
            p["ny"] = max(16, p["ny"] * 3 // 4 + 1)
    return tuple(prms)


class _View:
    """Device memory of a handle as torch takes it; it keeps the handle's owner alive."""

    def __init__(self, owner, ptr, shape, strides, typ):
        self.owner = owner
        self.__cuda_array_interface__ = {"data": (ptr, False), "shape": shape, "strides": strides, "typestr": typ,
                                         "version": 3}


def _views(st):
    """The solver's device-resident fields as torch tensors (no copy)."""
    s, prm = st["s"], st["prm"]
    es = prm["precision"] // 8
    out = {}
    for nm in ("phi", "u", "v", "w", "p", "mu"):
        if nm == "w" and prm["dim"] == 2:
            continue
        ptr, pitch = s.field_ptr(nm)
        shape = inputs.shape_of(prm)
        strides = [es, pitch * es, pitch * prm["ny"] * es][:prm["dim"]][::-1]
        out[nm] = torch.as_tensor(_View(st, ptr, shape, tuple(strides), "<f%d" % es), device="cuda")
    return out


# ---------------------------------------------------------------------------
# prepare and run
# ---------------------------------------------------------------------------

def _drops_seed(case, seed):
    """Seeds of the two-drop problems that neither training, calibration nor evaluation uses."""
    return 60000 + (seed + 977 * case["layout"]) % 1000000


def _net_shape(case):
    return [int(c) for c in case["channels"].split(",")]


def _states(case, seed, count):
    """``count`` minibatches of packed states [B, H, W, 5] and the states some steps later."""
    H, W, B = case["n"], case["w"], case["batch"]
    g = torch.Generator(device="cpu").manual_seed(int(seed) * 104729 + 5)
    n = count * B
    r = torch.rand((n, 12), generator=g, dtype=torch.float64).cuda()
    at = lambda i: r[:, i].reshape(n, 1, 1)  # noqa: E731
    y = ((torch.arange(H, dtype=torch.float64, device="cuda") + 0.5) / H).reshape(1, H, 1)
    x = ((torch.arange(W, dtype=torch.float64, device="cuda") + 0.5) / W).reshape(1, 1, W)
    wide = 4.0 / max(H, W)

    def state(t):
        phi = None
        for c in (0, 3):
            dx = torch.remainder(x - at(c) - 0.01 * t + 0.5, 1.0) - 0.5
            dy = torch.remainder(y - at(c + 1) + 0.5, 1.0) - 0.5
            f = torch.tanh(2.0 * ((0.08 + 0.1 * at(c + 2)) * (1.0 - 0.01 * t) - torch.sqrt(dx * dx + dy * dy)) / wide)
            phi = f if phi is None else torch.maximum(phi, f)
        w = 2.0 * math.pi
        u = 4e-3 * (1.0 + 0.2 * t) * torch.sin(w * (x + at(6))) * torch.cos(w * (y + at(7))) * (1.2 + phi)
        v = -4e-3 * (1.0 - 0.1 * t) * torch.cos(w * (x + at(6))) * torch.sin(w * (y + at(7))) * (1.2 + phi)
        p = 3e-4 * (1.0 + phi + 0.3 * torch.cos(w * (2 * x + at(8) + 0.1 * t)) * torch.cos(w * (y + at(9))))
        rho = 0.5 * (1.0 + phi) + 0.5 * (1.0 - phi) * (0.05 + 0.4 * at(10))
        return torch.stack([phi, u, v, p, rho], dim=-1).float()

    shape = (count, B, H, W, 5)
    return state(0.0).reshape(shape).contiguous(), state(1.0).reshape(shape).contiguous()


def _stats(x, t):
    """Normalisation of the network for states x and their successors t."""
    m = x.double().reshape(-1, 5)
    dx = (t.double() - x.double()).reshape(-1, 5)
    sc = torch.clamp(m.std(dim=0), min=1e-6)
    osc = dx.square().mean(dim=0).sqrt()
    osc = torch.maximum(osc, 1e-3 * osc.max())
    return [v.float().cpu().numpy() for v in (m.mean(dim=0), sc, osc)]


def _surrogate(case, seed, stats):
    if case.get("trained"):
        return S.Surrogate.load(WEIGHTS, max_batch=case["batch"])
    ch = _net_shape(case)
    # the networks of this package are square; other shapes go through the network's own binding
    if case["n"] == case["w"]:
        sur = S.Surrogate(n=case["n"], levels=len(ch), channels=ch, max_batch=case["batch"], seed=seed)
        sur.set_stats(*stats)
        return sur
    net = gpe2p.Net(len(ch), ch, 5, 5, case["n"], case["w"], case["batch"], seed=seed)
    net.set_normalization(*stats, residual=True)
    return net


def prepare(case, seed):
    kind = case["kind"]
    st = {"case": case}
    if kind == "solve":
        prm = _params(case)
        f = {k: v.cpu().numpy() for k, v in _fields(prm, case["problem"], seed).items()}
        s = gpe2p.Solver(prm)
        s.set_phi_accumulation(gpe2p.PHI_ACC_COMPENSATED if case["compensated"] else gpe2p.PHI_ACC_FP32)
        if case["whole"]:
            st["f"] = f
        else:
            s.init_fields(f)
        if case["packed"]:
            st["x"] = torch.empty((prm["ny"], prm["nx"], 5), dtype=torch.float32, device="cuda")
        st.update(prm=prm, s=s)
    elif kind == "batch":
        prms = _batch_params(case["n"], case["sides"], case["precision"])
        b = gpe2p.Batch(prms)
        for k, p in enumerate(prms):
            f = _fields(p, "drop" if k % 2 == 0 else "bubble", seed * 131 + k)
            b.init_instance(k, {key: v.cpu().numpy() for key, v in f.items()})
        flat = torch.empty(sum(4 * p["nx"] * p["ny"] for p in prms), dtype=torch.float32, device="cuda")
        at, parts = 0, []
        for p in prms:
            m = 4 * p["nx"] * p["ny"]
            parts.append(flat[at:at + m].view(p["ny"], p["nx"], 4))
            at += m
        st.update(b=b, flat=flat, parts=parts)
    elif kind == "controller":
        sur = S.Surrogate.load(WEIGHTS, max_batch=1)
        prm, f = inputs.two_drops(_drops_seed(case, seed), n=case["n"])
        s = gpe2p.Solver(prm, stream=sur.stream)
        s.set_phi_accumulation(gpe2p.PHI_ACC_FP32)
        s.init_fields(f)
        x0 = torch.empty((case["n"], case["n"], 5), dtype=torch.float32, device="cuda")
        s.pack(x0)
        st.update(sur=sur, s=s, prm=prm, x0=x0, x=torch.empty_like(x0))
    else:
        count = case.get("steps", 1)
        x, t = _states(case, seed, count)
        sur = _surrogate(case, seed, _stats(x, t))
        st.update(sur=sur, net=getattr(sur, "net", sur), x=x, t=t, y=torch.empty_like(x[0]))
    torch.cuda.synchronize()
    return st


def run(st):
    case = st["case"]
    kind = case["kind"]
    if kind == "solve":
        s = st["s"]
        if case["whole"]:
            s.init_fields(st["f"])
            d = s.advance(case["steps"])
            return dict(s.read_fields(), kinetic=d["kinetic"], umax=d["umax"])
        if case["nz"] and not case["compensated"]:
            # asynchronous steps, as a program that overlaps its own work has them
            for _ in range(case["steps"]):
                s.step()
            return _views(st)
        d = s.advance(case["steps"])
        if case["packed"]:
            s.pack(st["x"])
            return st["x"]
        return dict(_views(st), kinetic=d["kinetic"], umax=d["umax"])
    if kind == "batch":
        b = st["b"]
        b.advance(case["steps"])
        for k, t in enumerate(st["parts"]):
            b.pack(k, t)
        return st["flat"]
    if kind == "controller":
        s = st["s"]
        s.unpack(st["x0"])
        # kept until the next pass: its tensors are read on the surrogate's stream
        st["c"] = S.Controller(st["sur"], s)
        stats = st["c"].run(case["calls"])
        s.pack(st["x"])
        return {"state": st["x"], "failures": stats.failures, "net_calls": stats.net_calls}
    if kind == "forward":
        st["net"].forward(st["x"][0], st["y"], case["batch"])
        return st["y"]
    loss = None
    for i in range(case["steps"]):
        # a small learning rate, as fine tuning ends with
        loss = st["net"].train_step(st["x"][i], st["t"][i], case["batch"], 2e-6, want_loss=i == case["steps"] - 1)
    return {"loss": loss, "params": st["net"].get_params()}


# ---------------------------------------------------------------------------
# work
# ---------------------------------------------------------------------------

# floating-point operations per cell of one flow stage, one Cahn-Hilliard stage and one mu sweep, each
# face and edge term of the stencils formed once
_FLOPS = {2: (100, 45, 20), 3: (190, 70, 30)}


def _solver_work(prm, steps):
    d = prm["dim"]
    cells = prm["nx"] * prm["ny"] * (prm["nz"] if d == 3 else 1)
    es = prm["precision"] // 8
    fl, ch, mu = _FLOPS[d]
    scheme = prm["ch_scheme"]
    # a step reads phi, p and the velocity and writes them and mu
    return {"bytes": steps * cells * es * ((d + 2) + (d + 3)), "flops": steps * cells * (3 * fl + scheme * (ch + mu))}


def _net_flops(case):
    ch = _net_shape(case)
    pix = case["n"] * case["w"] * case["batch"]
    L, fl = len(ch), 0.0
    for l in range(L):
        n = pix / 4 ** l
        fl += 18.0 * n * ((16 if l == 0 else ch[l - 1]) * ch[l] + ch[l] * ch[l])
        if l < L - 1:
            fl += 18.0 * n * (ch[l + 1] * ch[l] + 2 * ch[l] * ch[l] + ch[l] * ch[l])
    return fl + 2.0 * pix * 5 * ch[0]


def _net_params(ch):
    return sum(a * 9 * b + b for a, b in _convs(ch)) + 5 * ch[0] + 5


def _convs(ch):
    L = len(ch)
    c = []
    for l in range(L):
        c += [(16 if l == 0 else ch[l - 1], ch[l]), (ch[l], ch[l])]
    for l in range(L - 2, -1, -1):
        c += [(ch[l + 1], ch[l]), (2 * ch[l], ch[l]), (ch[l], ch[l])]
    return c


def work(case):
    kind = case["kind"]
    if kind == "solve":
        return _solver_work(_params(case), case["steps"])
    if kind == "batch":
        ws = [_solver_work(p, case["steps"]) for p in _batch_params(case["n"], case["sides"], case["precision"])]
        cells = sum(p["nx"] * p["ny"] for p in _batch_params(case["n"], case["sides"], case["precision"]))
        return {"bytes": sum(w["bytes"] for w in ws) + 16 * cells, "flops": sum(w["flops"] for w in ws)}
    if kind == "controller":
        net = dict(n=case["n"], w=case["n"], batch=1, channels=",".join(str(c) for c in CH))
        prm = dict(inputs.base_params(2, case["n"], case["n"]), precision=32)
        w = _solver_work(prm, 64 * (case["calls"] // 4))
        pix = case["n"] ** 2
        return {"bytes": w["bytes"] + case["calls"] * (2 * pix * 20 + 2 * _net_params(list(CH))),
                "flops": w["flops"] + case["calls"] * _net_flops(net)}
    pix = case["n"] * case["w"] * case["batch"]
    npar = _net_params(_net_shape(case))
    if kind == "forward":
        return {"bytes": 2 * pix * 20 + 2 * npar, "flops": _net_flops(case)}
    # weights, both Adam moments read and written; states and targets read; the weights returned
    return {"bytes": case["steps"] * (2 * pix * 20 + 24 * npar) + 4 * npar, "flops": 3.0 * case["steps"] * _net_flops(case)}


# ---------------------------------------------------------------------------
# the method in 64 bits
# ---------------------------------------------------------------------------

class _Exact:
    """The step of Sec. 3 in FP64 torch, one tensor operation per term."""

    def __init__(self, prm):
        self.p, self.d = prm, prm["dim"]
        self.n = [prm["nx"], prm["ny"], prm["nz"]][:self.d]
        self.bc = list(prm["bc"])[:self.d]
        self.axi = bool(prm.get("axisym"))
        iso = prm["iso"]
        self.w = {9: (0, 1 / 9, 1 / 36, 0), 15: (0, 1 / 9, 0, 1 / 72), 19: (0, 1 / 18, 1 / 36, 0),
                  27: (0, 2 / 27, 1 / 54, 1 / 216)}[iso]
        rng = range(-1, 2)
        self.e = [(x, y, z) for z in (rng if self.d == 3 else (0,)) for y in rng for x in rng
                  if (x, y, z) != (0, 0, 0) and self.w[x * x + y * y + z * z] != 0]
        if self.axi:
            i = torch.arange(self.n[0], dtype=torch.float64, device="cuda")
            self.r_cen, self.r_face = (i + 0.5) * prm["dx"], i * prm["dx"]

    def pad(self, f, comp=None, vec=None):
        """One ghost layer; comp: a face velocity component, vec: a cell vector component."""
        for a in range(self.d):
            ax = self.d - 1 - a
            n = self.n[a]
            lo, hi = f.narrow(ax, 0, 1), f.narrow(ax, n - 1, 1)
            if self.bc[a] == "periodic":
                lo, hi = hi, lo
            elif comp == a:
                lo = -f.narrow(ax, 1, 1) if n > 1 else torch.zeros_like(lo)
                hi = torch.zeros_like(hi)
            elif comp is not None and self.bc[a] == "noslip":
                lo, hi = (lo if (self.axi and a == 0) else -lo), -hi
            elif vec == a:
                lo, hi = -lo, -hi
            f = torch.cat([lo, f, hi], dim=ax)
        return f

    def at(self, f, *o):
        """The padded field at offset o = (x, y[, z])."""
        for a in range(self.d):
            f = f.narrow(self.d - 1 - a, 1 + (o[a] if a < len(o) else 0), self.n[a])
        return f

    def unit(self, a, s=1):
        return tuple(s if b == a else 0 for b in range(self.d))

    @staticmethod
    def add(*os):
        return tuple(sum(v) for v in zip(*os))

    def lap(self, f):
        c = self.at(f)
        s = sum(self.w[sum(abs(v) for v in e)] * (self.at(f, *e) - c) for e in self.e)
        return 6.0 / self.p["dx"] ** 2 * s

    def grad(self, f, a):
        s = sum(self.w[sum(abs(v) for v in e)] * e[a] * self.at(f, *e) for e in self.e if e[a])
        return 3.0 / self.p["dx"] * s

    def mu(self, phi):
        f = self.pad(phi)
        lap = self.lap(f)
        if self.axi:
            lap = lap + self.grad(f, 0) / self.r_cen
        a, kappa = 3.0 / (4.0 * self.p["W"]), 3.0 * self.p["W"] / 8.0
        return 4.0 * a * phi * (phi * phi - 1.0) - kappa * lap

    def flow_rates(self, q, mat):
        P, d, dx, at, add = self.p, self.d, self.p["dx"], self.at, self.add
        phi, mu, rho, eta, nu = mat
        p = self.pad(q[0])
        U = [self.pad(q[1 + a], comp=a) for a in range(d)]
        Z = (0,) * d
        un = [self.unit(a) for a in range(d)]
        mn = [self.unit(a, -1) for a in range(d)]

        def div(o):
            s = sum(at(U[a], *add(o, un[a])) - at(U[a], *o) for a in range(d)) / dx
            if self.axi:
                s = s + 0.5 * (at(U[0], *o) + at(U[0], *add(o, un[0]))) / (self.r_cen + o[0] * dx)
            return s

        D0 = div(Z)
        p0, nu0 = at(p), at(nu)
        diff = sum(0.5 * (nu0 + at(nu, *o)) * (at(p, *o) - p0) for o in un + mn) / dx ** 2
        if self.axi:
            diff = diff + nu0 * (at(p, 1, 0) - at(p, -1, 0)) / (2.0 * dx) / self.r_cen
        rates = [-at(rho) * P["cs"] ** 2 * D0 + diff]
        for c in range(d):
            m = mn[c]
            rb = 0.5 * (at(rho, *m) + at(rho))
            pp = p
            if P["p_average"]:
                for t in range(d):
                    if t != c:
                        ax = d - 1 - t
                        k = pp.shape[ax]
                        s = (pp.narrow(ax, 0, k - 2) + 4.0 * pp.narrow(ax, 1, k - 2) + pp.narrow(ax, 2, k - 2)) / 6.0
                        # back to a padded extent; the ghost layers along t are not read again
                        pp = torch.cat([s.narrow(ax, 0, 1), s, s.narrow(ax, k - 3, 1)], dim=ax)
            gradp = (at(pp) - at(pp, *m)) / dx
            f = U[c]
            f0 = at(f)
            visc = 2.0 * (at(eta) * (at(f, *un[c]) - f0) - at(eta, *m) * (f0 - at(f, *m))) / dx ** 2
            conv = f0 * (at(f, *un[c]) - at(f, *m)) / (2.0 * dx)
            for t in range(d):
                if t == c:
                    continue
                T = U[t]
                for s, o in ((1.0, un[t]), (-1.0, mn[t])):
                    eb = 0.25 * (at(eta) + at(eta, *m) + at(eta, *o) + at(eta, *add(m, o)))
                    edge = un[t] if s > 0 else Z
                    shear = s * (at(f, *o) - f0) + at(T, *edge) - at(T, *add(edge, m))
                    visc = visc + s * eb * shear / dx ** 2
                tb = 0.25 * (at(T) + at(T, *m) + at(T, *un[t]) + at(T, *add(un[t], m)))
                conv = conv + tb * (at(f, *un[t]) - at(f, *mn[t])) / (2.0 * dx)
            if P["bulk_visc"]:
                visc = visc + (at(eta) * D0 - at(eta, *m) * self._div_below(div, m)) / dx
            if self.axi:
                ef = 0.5 * (at(eta, *m) + at(eta))
                du = (at(f, 1, 0) - at(f, -1, 0)) / (2.0 * dx)
                if c == 0:
                    r = torch.clamp(self.r_face, min=dx)  # face 0 lies on the axis and is not updated
                    visc = visc + ef / r * (du - f0 / r)
                else:
                    visc = visc + ef / self.r_cen * du
            st = -P["sigma"] * 0.5 * (at(phi) + at(phi, *m)) * (at(mu) - at(mu, *m)) / dx
            L = -conv + (visc - gradp + st + (rb - P["rho_ref"]) * P["g"][c]) / rb
            if self.bc[c] != "periodic":
                L = L.clone()
                L.select(d - 1 - c, 0).zero_()
            rates.append(L)
        return rates

    @staticmethod
    def _div_below(div, m):
        return div(m)

    def step(self, q, phi, mu):
        P, d, dt = self.p, self.d, self.p["dt"]
        pf, pm = self.pad(phi), self.pad(mu)
        law = lambda L, G: 0.5 * (L + G) + 0.5 * (L - G) * pf  # noqa: E731
        rho, eta = law(P["rhoL"], P["rhoG"]), law(P["etaL"], P["etaG"])
        mat = (pf, pm, rho, eta, eta / rho)
        s = q
        for a, b in ((0.0, 1.0), (0.75, 0.25), (1.0 / 3.0, 2.0 / 3.0)):
            L = self.flow_rates(s, mat)
            s = [a * x0 + b * (x + dt * r) for x0, x, r in zip(q, s, L)]
        uh = []
        for a in range(d):
            f = 0.5 * (q[1 + a] + s[1 + a])
            uh.append(0.5 * (f + self.at(self.pad(f, comp=a), *self.unit(a))))
        uv = [self.pad(u, vec=a) for a, u in enumerate(uh)]

        def rate(ph, m):
            f, g = self.pad(ph), self.pad(m)
            lap = self.lap(g)
            if self.axi:
                lap = lap + self.grad(g, 0) / self.r_cen
            if P["ch_advection"]:
                adv = sum(self.grad(uv[a] * f, a) for a in range(d))
            else:
                adv = sum(uh[a] * self.grad(f, a) for a in range(d))
            return P["M"] * lap - adv

        if P["ch_scheme"] == 2:
            f1 = phi + dt * rate(phi, mu)
            out = 0.5 * phi + 0.5 * (f1 + dt * rate(f1, self.mu(f1)))
        else:
            k1 = dt * rate(phi, mu)
            f = phi + 0.5 * k1
            k2 = dt * rate(f, self.mu(f))
            f = phi + 0.5 * k2
            k3 = dt * rate(f, self.mu(f))
            f = phi + k3
            k4 = dt * rate(f, self.mu(f))
            out = phi + (k1 + 2.0 * k2 + 2.0 * k3 + k4) / 6.0
        return s, out, self.mu(out)

    def advance(self, f, steps):
        """(q, phi, mu) after the steps, from fields {phi, p, u, v[, w]}."""
        q = [f["p"]] + [f[n] for n in "uvw"[:self.d]]
        phi = f["phi"]
        mu = self.mu(phi)
        for _ in range(steps):
            q, phi, mu = self.step(q, phi, mu)
        return q, phi, mu

    def diag(self, q, phi):
        """Kinetic energy over the faces and the largest velocity component."""
        P, d = self.p, self.d
        rho = self.pad(0.5 * (P["rhoL"] + P["rhoG"]) + 0.5 * (P["rhoL"] - P["rhoG"]) * phi)
        ke = sum((0.5 * (self.at(rho, *self.unit(a, -1)) + self.at(rho)) * q[1 + a] ** 2).sum() for a in range(d))
        return float(0.5 * ke * P["dx"] ** d), float(max(q[1 + a].abs().max() for a in range(d)))


def _named(q, phi, mu, host=False):
    out = dict(zip(("p", "u", "v", "w"), q), phi=phi, mu=mu)
    return {k: v.cpu().numpy() for k, v in out.items()} if host else out


def _packed(prm, s):
    """phi, u, v, p and rho / rho_L as the last axis, the network's view of a state."""
    rho = 0.5 * (prm["rhoL"] + prm["rhoG"]) + 0.5 * (prm["rhoL"] - prm["rhoG"]) * s["phi"]
    return torch.stack([s["phi"], s["u"], s["v"], s["p"], rho / prm["rhoL"]], dim=-1)


def _exact_net(w, ch, x, mean, scale, oscale):
    """The U-Net in FP64: x [B, H, W, 5] -> x + oscale * head; w: the flat parameters."""
    L = len(ch)
    parts, at = [], 0
    for cin, cout in _convs(ch):
        k = w[at:at + cout * 9 * cin].reshape(cout, 3, 3, cin).permute(0, 3, 1, 2)
        at += cout * 9 * cin
        parts.append((k, w[at:at + cout]))
        at += cout
    hw = w[at:at + 5 * ch[0]].reshape(5, ch[0])
    hb = w[at + 5 * ch[0]:]

    def conv(f, i):
        k, b = parts[i]
        return F.silu(F.conv2d(F.pad(f, (1, 1, 1, 1), mode="circular"), k, b))

    h = ((x - mean) / scale).permute(0, 3, 1, 2)
    h = F.pad(h, (0, 0, 0, 0, 0, 11))
    skip, i = [], 0
    for l in range(L):
        if l:
            h = F.avg_pool2d(h, 2)
        h = conv(conv(h, i), i + 1)
        i += 2
        skip.append(h)
    for l in range(L - 2, -1, -1):
        h = conv(h.repeat_interleave(2, 2).repeat_interleave(2, 3), i)
        h = conv(conv(torch.cat([h, skip[l]], dim=1), i + 1), i + 2)
        i += 3
    y = torch.einsum("bchw,oc->bhwo", h, hw) + hb
    return x + oscale * y


def _f64(v):
    return torch.as_tensor(np.asarray(v, dtype=np.float64), device="cuda")


def _exact_train(case, seed):
    x, t = _states(case, seed, case["steps"])
    stats = _stats(x, t)
    sur = _surrogate(case, seed, stats)  # for its seeded starting weights
    net = getattr(sur, "net", sur)
    w = _f64(net.get_params()).requires_grad_(True)
    sur.close()
    mean, scale, oscale = (_f64(v) for v in stats)
    m, v, loss = torch.zeros_like(w), torch.zeros_like(w), None
    for i in range(case["steps"]):
        grad, loss = torch.zeros_like(w), 0.0
        for b in range(case["batch"]):
            y = _exact_net(w, _net_shape(case), x[i, b:b + 1].double(), mean, scale, oscale)
            part = ((y - t[i, b:b + 1].double()) / oscale).square().mean() / case["batch"]
            grad += torch.autograd.grad(part, w)[0]
            loss += float(part)
        m = 0.9 * m + 0.1 * grad
        v = 0.999 * v + 0.001 * grad * grad
        with torch.no_grad():
            w -= 2e-6 * (m / (1 - 0.9 ** (i + 1))) / ((v / (1 - 0.999 ** (i + 1))).sqrt() + 1e-8)
    return {"loss": loss, "params": w.detach().cpu().numpy()}


def _exact_controller(case, seed):
    sur = S.Surrogate.load(WEIGHTS, max_batch=1)
    w = _f64(sur.net.get_params())
    mean, scale, osc = (_f64(v) for v in (sur.in_mean, sur.in_scale, sur.out_scale))
    prm, f = inputs.two_drops(_drops_seed(case, seed), n=case["n"])
    ex = _Exact(prm)
    st = {k: _f64(v) for k, v in f.items()}
    st["mu"] = ex.mu(st["phi"])

    def solve(s, steps):
        q, phi, mu = ex.advance(s, steps)
        return _named(q, phi, mu)

    def call(s):
        y = _exact_net(w, list(CH), _packed(prm, s)[None], mean, scale, osc)[0]
        out = {k: y[..., c].contiguous() for c, k in enumerate(("phi", "u", "v", "p"))}
        out["mu"] = ex.mu(out["phi"])
        return out

    left, window, off, failures, calls, start = case["calls"], 0, 0, 0, 0, None
    with torch.no_grad():
        for _ in range(left):
            if window == 0:
                start = st
            window += 1
            last = window == 4
            if off:
                st = solve(st, sur.K)
                if last:
                    window, off = 0, off - 1
                continue
            y = call(st)
            calls += 1
            if not last:
                st = y
                continue
            window = 0
            st = solve(st, sur.K)
            e = float((y["phi"] - st["phi"]).norm() / st["phi"].norm())
            ph = ex.pad(st["phi"])
            g = sum((0.5 * (ex.at(ph, *ex.unit(a)) - ex.at(ph, *ex.unit(a, -1)))) ** 2 for a in range(2)).sqrt()
            band = st["phi"].abs() < 0.5
            disp = float(((y["phi"] - st["phi"]).abs() / g.clamp(min=1e-12))[band].max())
            if not (e <= sur.check_tol and disp <= sur.check_tol_disp):
                failures += 1
                st = solve(start, 4 * sur.K)
                off = 1
    sur.close()
    return {"state": _packed(prm, st), "failures": failures, "net_calls": calls}


def exact(case, seed):
    kind = case["kind"]
    if kind == "solve":
        prm = _params(case)
        ex = _Exact(prm)
        q, phi, mu = ex.advance(_fields(prm, case["problem"], seed), case["steps"])
        out = _named(q, phi, mu, host=case["whole"])
        if case["packed"]:
            return _packed(prm, out)
        if case["whole"] or not (case["nz"] and not case["compensated"]):
            out["kinetic"], out["umax"] = ex.diag(q, phi)
        return out
    if kind == "batch":
        flat = []
        for k, p in enumerate(_batch_params(case["n"], case["sides"], case["precision"])):
            q, phi, _ = _Exact(p).advance(_fields(p, "drop" if k % 2 == 0 else "bubble", seed * 131 + k), case["steps"])
            flat.append(torch.stack([phi, q[1], q[2], q[0]], dim=-1).reshape(-1))
        return torch.cat(flat)
    if kind == "controller":
        return _exact_controller(case, seed)
    if kind == "forward":
        x, t = _states(case, seed, 1)
        sur = _surrogate(case, seed, _stats(x, t))
        net = getattr(sur, "net", sur)
        w = _f64(net.get_params())
        stats = (sur.in_mean, sur.in_scale, sur.out_scale) if hasattr(sur, "net") else _stats(x, t)
        ch = list(CH) if case.get("trained") else _net_shape(case)
        sur.close()
        with torch.no_grad():
            return torch.cat([_exact_net(w, ch, x[0, b:b + 1].double(), *(_f64(v) for v in stats))
                              for b in range(case["batch"])])
    return _exact_train(case, seed)
