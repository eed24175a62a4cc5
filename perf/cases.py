"""Performance cases of the library: the work its users have it do, through
its public entry points (the Python binding of the C ABI), with sizes and
parameter sets of this repository's workloads, tests and benchmark.

kinds
  lb       a solver context on a stream of its own: `steps` time steps, then phi
           and u of every domain read into device memory (and, with `measure`,
           the tips, solid fraction and conserved sum).  The state goes on
           from pass to pass, as in a run that is looked at every `steps` steps.
  restart  fields written to the solver, `steps` steps from equilibrium, a
           measurement, the fields read back: one validation of the surrogate's
           controller, or a continuation from stored fields.
  layer    one 3x3 convolution layer: forward, data gradient, weight gradient.
  forward  the surrogate network on a batch of fields.
  train    forward and parameter gradients of the surrogate network on a batch.
"""
import math
import random

import numpy as np
import torch

from paper_1606_09432_gb300 import lbpf as L

# Parameter sets (physical units; lam 0: the lambda* rule).
SETS = {
    "plain2d": dict(dx=0.4, dt=0.008, W0=1.0, tau0=1.0, kappa=2.0, lam=0.0),
    "dendrite": dict(dx=0.01, dt=1.5e-5, W0=0.0125, tau0=1.5625e-4, kappa=1.0, lam=10.0),
    "multi": dict(dx=5e-3, dt=5e-6, W0=0.012, tau0=1e-4, kappa=0.7, lam=10.0),
}
PRECISIONS = {"fp64": L.LBPF_FP64, "fp32": L.LBPF_FP32, "fp16": L.LBPF_FP32_FP16DEV, "bf16": L.LBPF_FP32_BF16DEV,
              "fp16sr": L.LBPF_FP32_FP16DEV_SR}
LATTICES = {"d2q9": L.LBPF_D2Q9_D2Q5, "d3q15": L.LBPF_D3Q15_D3Q7, "d3q19": L.LBPF_D3Q19_D3Q7,
            "d3q27": L.LBPF_D3Q27_D3Q7}
FORMS = {"cubic100": L.LBPF_AS_CUBIC100, "angle": L.LBPF_AS_ANGLE, "y66": L.LBPF_AS_Y66, "hoyt110": L.LBPF_AS_HOYT110,
         "s111": L.LBPF_AS_S111}


def lb(name, lattice, precision, nx, ny, nz, steps, *, params, form, eps=0.05, gamma=0.0, q=4, delta=0.3, bc=0,
       grad="dd", crystals=1, domains=1, measure=False, corner=False, adv=0.0, kind="lb", stream=True):
    c = dict(kind=kind, lattice=lattice, precision=precision, nx=nx, ny=ny, nz=nz, steps=steps, params=params,
             form=form, eps=eps, gamma=gamma, q=q, delta=delta, bc=bc, grad=grad, crystals=crystals, domains=domains,
             measure=measure, corner=corner, adv=adv, stream=stream)
    return dict(c, name=name) if name else c


def listed():
    return [
        # the plain 2D method at its smallest in use: 100 steps between two looks at the crystal, all launch latency
        lb("plane-128-fp32", "d2q9", "fp32", 128, 128, 1, 100, params="plain2d", form="cubic100"),
        # the isotropy study of a sixfold crystal: 800 x 800 nodes, double precision, walls on all sides
        lb("sixfold-800-fp64", "d2q9", "fp64", 800, 800, 1, 20, params="dendrite", form="angle", q=6, bc=3),
        # 64 ragged 2D domains (sides 128..1024) with up to 12 crystals each in one context, read every 50 steps: the
        # batched configuration, and how training pairs of the surrogate are generated
        lb("batch-64-fp32", "d2q9", "fp32", 1024, 1024, 1, 50, params="multi", form="angle", crystals=12, domains=64,
           stream=False),
        # a point of the anisotropy sweep: 64^3 crop with BF16 deviations, measured every 12 steps
        lb("crop-64-bf16", "d3q15", "bf16", 64, 64, 64, 12, params="dendrite", form="hoyt110", eps=0.02, gamma=-0.02,
           delta=0.4, measure=True),
        # the 3D single crystal in full precision
        lb("crystal-256-fp32", "d3q15", "fp32", 256, 256, 256, 20, params="dendrite", form="cubic100"),
        # the D3Q19 lattice on a box whose sides fit no tile
        lb("ragged-d3q19-fp32", "d3q19", "fp32", 207, 174, 190, 20, params="dendrite", form="cubic100"),
        # the octant run with mirror walls, 351^3 nodes, seed in the corner, FP16 deviations, monitored
        lb("octant-351-fp16", "d3q15", "fp16", 351, 351, 351, 20, params="dendrite", form="hoyt110", eps=0.0,
           gamma=-0.02, delta=0.25, bc=7, corner=True, measure=True),
        # the benchmark's workload: 512^3, FP16 deviations
        lb("dendrite-512-fp16", "d3q15", "fp16", 512, 512, 512, 20, params="dendrite", form="hoyt110", eps=0.0,
           gamma=-0.02, delta=0.4),
        # one validation of the surrogate's controller on a 1024^2 domain of two crystals: write, 20 steps, measure, read
        lb("restart-1024-fp32", "d2q9", "fp32", 1024, 1024, 1, 20, params="multi", form="angle", crystals=2,
           measure=True, kind="restart", stream=False),
        # a wide layer of the surrogate, all three directions
        dict(kind="layer", name="layer-256-128ch", n=1, H=256, W=256, cin=128, cout=128),
        # a network jump on a 1024^2 domain
        dict(kind="forward", name="jump-1024", n=1, H=1024, W=1024, levels=3, base=16),
        # a training batch: 8 crops of 128^2
        dict(kind="train", name="train-8x128", n=8, H=128, W=128, levels=3, base=16),
    ]


def _log(rng, a, b):
    return int(round(math.exp(rng.uniform(math.log(a), math.log(b)))))


def draw(rng):
    kind = rng.choices(["2d", "3d", "batch", "restart", "layer", "forward", "train"], [4, 6, 1, 2, 2, 1, 2])[0]
    if kind == "layer":
        cin, cout = rng.choice([16, 32, 64, 96, 128, 192, 256, 384]), rng.choice([16, 32, 48, 64, 128, 256])
        while True:
            n, H, W = rng.choice([1, 1, 2, 8]), _log(rng, 8, 1024), _log(rng, 8, 1024)
            if rng.random() < 0.6:
                H, W = max(16, H // 16 * 16), max(8, W // 8 * 8)
            if n * H * W * max(cin, cout) <= 1 << 25 and n * H * W * cin * cout <= 1 << 31:
                return dict(kind="layer", n=n, H=H, W=W, cin=cin, cout=cout)
    if kind in ("forward", "train"):
        levels, base = rng.choice([(3, 16), (3, 16), (3, 16), (4, 32), (2, 32), (4, 16)])
        q = 8 << (levels - 1)
        while True:
            n = 1 if kind == "forward" else rng.choice([1, 2, 4, 8])
            H, W = (max(1, _log(rng, 64, 1024) // q) * q for _ in "HW")
            if n * H * W * base <= (1 << 24 if kind == "forward" else 1 << 22):
                return dict(kind=kind, n=n, H=H, W=W, levels=levels, base=base)
    steps = _log(rng, 8, 100)
    stream = rng.random() < 0.7
    if kind == "batch":
        return lb(None, "d2q9", rng.choice(["fp32", "fp16"]), _log(rng, 192, 768), _log(rng, 192, 768), 1,
                  min(steps, 40), params="multi", form="angle", crystals=rng.randint(1, 8), domains=rng.randint(2, 40),
                  stream=stream)
    measure, delta = rng.random() < 0.4, round(rng.uniform(0.25, 0.4), 3)
    if kind == "2d" or (kind == "restart" and rng.random() < 0.6):
        nx, ny = _log(rng, 48, 1200), _log(rng, 48, 1200)
        multi = rng.random() < 0.3
        form = "angle" if multi else rng.choice(["cubic100", "angle", "y66"])
        return lb(None, "d2q9", rng.choice(["fp32", "fp32", "fp64", "fp16", "bf16"]), nx, ny, 1, steps,
                  params="multi" if multi else rng.choice(["plain2d", "dendrite"]), form=form,
                  q=rng.choice([4, 6]), delta=delta, bc=0 if multi else rng.choice([0, 0, 0, 1, 2, 3]),
                  grad=rng.choice(["dd", "dd", "dd", "fd"]), crystals=rng.randint(2, 6) if multi else 1,
                  measure=measure, kind="restart" if kind == "restart" else "lb", stream=stream)
    precision = rng.choice(["fp32", "fp32", "fp16", "fp16", "bf16", "fp16sr", "fp64"])
    top = 64 if precision == "fp64" else 448
    while True:
        nx, ny, nz = (_log(rng, 24, top) for _ in range(3))
        if rng.random() < 0.5:
            nx = max(32, nx // 32 * 32)
        if nx * ny * nz <= 48_000_000:
            break
    steps = min(steps, 24)
    form, eps, gamma = rng.choice([("cubic100", 0.05, 0.0), ("hoyt110", 0.0, -0.02), ("hoyt110", 0.02, 0.02),
                                   ("s111", 0.0, 0.02)])
    walls = rng.random() < 0.25
    return lb(None, rng.choice(["d3q15", "d3q15", "d3q19", "d3q27"]), precision, nx, ny, nz, steps, params="dendrite",
              form=form, eps=eps, gamma=gamma, delta=delta, bc=7 if walls else 0, corner=walls,
              adv=0.02 if not walls and rng.random() < 0.15 else 0.0, measure=measure,
              kind="restart" if kind == "restart" else "lb", stream=stream)


# --- inputs ------------------------------------------------------------------

def _domains(case, seed):
    """Per domain: sizes, crystals (eps, phi0), undercooling and seeds (x, y, z, R, crystal)."""
    rng = random.Random(seed * 7919 + 17)
    out = []
    for k in range(case["domains"]):
        nx, ny, nz = case["nx"], case["ny"], case["nz"]
        if case["domains"] > 1:  # ragged batch: the same sides for every seed
            side = random.Random(1000 + k)
            nx, ny = (max(32, int(v * side.uniform(0.125, 1.0))) for v in (nx, ny))
        delta, nc = case["delta"], case["crystals"]
        if case["domains"] > 1:
            nc = random.Random(2000 + k).randint(1, nc)
        multi = nc > 1 or case["params"] == "multi"
        crystals, seeds = [], []
        for j in range(nc):
            crystals.append((rng.uniform(0.01, 0.07) if multi else case["eps"],
                             rng.uniform(0, math.pi / 2) if multi else 0.0))
            r = rng.uniform(4.0, 10.0) if multi else rng.uniform(6.0, 9.0)
            if case["corner"]:
                p = (0.0, 0.0, 0.0)
            elif multi:
                p = (rng.uniform(0, nx), rng.uniform(0, ny), 0.0)
            else:
                p = (nx // 2 + rng.uniform(-2, 2), ny // 2 + rng.uniform(-2, 2),
                     nz // 2 + rng.uniform(-2, 2) if nz > 1 else 0.0)
            seeds.append((*p, r, j))
        out.append(dict(nx=nx, ny=ny, nz=nz, crystals=crystals, delta=delta, seeds=seeds))
    return out


def _velocity(case):
    """v with v dt / dx = adv along x (and half of it along -y)."""
    p = SETS[case["params"]]
    v = case["adv"] * p["dx"] / p["dt"]
    return (v, -0.5 * v, 0.0)


def _profile(case, dom, dtype):
    """phi of the seeds (the max of their tanh profiles), u = -delta, and the dominant seed's crystal + 1."""
    p = SETS[case["params"]]
    dev = dict(device="cuda", dtype=torch.float64)
    best = idx = None
    for x0, y0, z0, r, j in dom["seeds"]:
        d2 = 0.0
        for axis, (n, c) in enumerate(((dom["nx"], x0), (dom["ny"], y0), (dom["nz"], z0))):
            d = torch.arange(n, **dev) - c
            if not case["bc"] >> axis & 1:
                d = torch.fmod(d, n)
                d = torch.where(d > 0.5 * n, d - n, torch.where(d < -0.5 * n, d + n, d))
            d2 = d2 + (d * d).reshape([-1 if a == 2 - axis else 1 for a in range(3)])
        v = torch.tanh((r - d2.sqrt()) * (p["dx"] / (math.sqrt(2.0) * p["W0"])))
        if best is None:
            best, idx = v, torch.full_like(v, j + 1, dtype=torch.int32)
        else:
            idx = torch.where(v > best, torch.full_like(idx, j + 1), idx)
            best = torch.maximum(best, v)
    return best.to(dtype).contiguous(), torch.full_like(best, -dom["delta"]).to(dtype).contiguous(), idx


def _layers(levels, base):
    ch = [base << k for k in range(levels)]
    out = [(16, ch[0]), (ch[0], ch[0])]
    for k in range(1, levels):
        out += [(ch[k - 1], ch[k]), (ch[k], ch[k])]
    for k in range(levels - 2, -1, -1):
        out += [(ch[k + 1] + ch[k], ch[k]), (ch[k], ch[k])]
    return out


def _weights(case, seed):
    """A network's flat parameters: He-uniform 3x3 weights, small biases and head."""
    rng = np.random.default_rng(seed * 31 + 5)
    out = []
    for cin, cout in _layers(case["levels"], case["base"]):
        out.append(rng.uniform(-1, 1, 9 * cin * cout) * math.sqrt(6.0 / (9 * cin)))
        out.append(rng.uniform(-0.05, 0.05, cout))
    out.append(rng.uniform(-1, 1, 2 * case["base"]) * math.sqrt(3.0 / case["base"]))
    out.append(rng.uniform(-0.05, 0.05, 2))
    return np.concatenate(out).astype(np.float32)


def _net_input(case, seed):
    """Network input of random growing crystals: phi a tanh profile, u diffusing around it, orientation and strength."""
    g = torch.Generator(device="cuda").manual_seed(seed + 3)
    n, H, W = case["n"], case["H"], case["W"]

    def uni(a, b, *shape):
        return a + (b - a) * torch.rand(*shape, generator=g, device="cuda")

    y = torch.arange(H, device="cuda").view(1, H, 1)
    x = torch.arange(W, device="cuda").view(1, 1, W)
    cy, cx, r = uni(0, H, n, 1, 1), uni(0, W, n, 1, 1), uni(0.1, 0.4, n, 1, 1) * min(H, W)
    dy, dx = (y - cy + H / 2) % H - H / 2, (x - cx + W / 2) % W - W / 2
    th = uni(0, math.pi / 2, n, 1, 1)
    d = torch.hypot(dy, dx) - r * (1 + 0.2 * torch.cos(4 * (torch.atan2(dy, dx) - th)))
    phi = torch.tanh(-d / 3.4)
    u = -uni(0.2, 0.6, n, 1, 1) * (1 - torch.exp(-d.clamp(min=0) / 12))
    X = torch.stack([phi, u, torch.cos(4 * th).expand_as(phi), torch.sin(4 * th).expand_as(phi),
                     uni(0.01, 0.07, n, 1, 1).expand_as(phi)], dim=-1)
    return X.float().contiguous()


def _loss_gradient(x):
    """Gradient of a squared error whose residual follows the interface and the cooled melt, as an early network's does."""
    phi, u = x[..., 0], x[..., 1]
    r = torch.stack([(1 - phi * phi) * (0.5 + u), 0.1 * (u - u.mean(dim=(1, 2), keepdim=True))], -1)
    return (r * (2.0 / r.numel())).contiguous()


def _layer_input(case, seed):
    g = torch.Generator(device="cuda").manual_seed(seed + 11)
    n, H, W, ci, co = (case[k] for k in ("n", "H", "W", "cin", "cout"))
    x = torch.randn(n, H, W, ci, generator=g, device="cuda").relu_()
    w = (torch.randn(9, co, ci, generator=g, device="cuda") * math.sqrt(2.0 / (9 * ci))).to(torch.bfloat16)
    b = torch.randn(co, generator=g, device="cuda") * 0.1
    dy = torch.randn(n, H, W, co, generator=g, device="cuda") * 0.1
    return x, w, b, dy


def prepare(case, seed):
    kind = case["kind"]
    if kind == "layer":
        x, w, b, dy = _layer_input(case, seed)
        return dict(kind=kind, x=x, w=w, b=b, dy=dy, wt=w.flip(0).transpose(1, 2).contiguous())
    if kind in ("forward", "train"):
        x = _net_input(case, seed)
        net = L.Net(case["H"], case["W"], batch=case["n"], levels=case["levels"], base=case["base"])
        net.set_params(_weights(case, seed))
        y = torch.empty(x.shape[:3] + (2,), device="cuda")
        return dict(kind=kind, net=net, x=x, y=y, dy=_loss_gradient(x) if kind == "train" else None)
    doms = _domains(case, seed)
    p = SETS[case["params"]]
    arr = [L.make_domain(d["nx"], d["ny"], d["nz"], delta=d["delta"], bc=case["bc"], adv=_velocity(case),
                         crystals=[L.make_crystal(FORMS[case["form"]], e, case["gamma"], case["q"], f)
                                   for e, f in d["crystals"]], **p) for d in doms]
    stream = torch.cuda.Stream() if case["stream"] else None
    grad = L.LBPF_GRAD_DD if case["grad"] == "dd" else L.LBPF_GRAD_FD
    s = L.Solver(arr, LATTICES[case["lattice"]], grad, PRECISIONS[case["precision"]],
                 stream=stream.cuda_stream if stream else None)
    dtype = torch.float64 if case["precision"] == "fp64" else torch.float32
    st = dict(kind=kind, s=s, stream=stream, steps=case["steps"], measure=case["measure"], doms=doms,
              out=torch.empty(sum(2 * d["nx"] * d["ny"] * d["nz"] for d in doms), dtype=dtype, device="cuda"))
    if kind == "restart":
        st["fields"] = _profile(case, doms[0], dtype)
    else:
        for k, d in enumerate(doms):
            s.seed(d["seeds"], domain=k)
    return st


def run(st):
    kind = st["kind"]
    if kind == "layer":
        x, dy = st["x"], st["dy"]
        y, dx = torch.empty_like(dy), torch.empty_like(x)
        dw = torch.zeros(st["w"].shape, device="cuda")
        L.nn_conv3x3(x, st["w"], st["b"], y, relu=True)
        L.nn_conv3x3(dy, st["wt"], None, dx)
        L.nn_conv3x3_wgrad(x, dy, dw)
        return dict(y=y, dx=dx, dw=dw)
    if kind == "forward":
        st["net"].forward(st["x"], st["y"])
        return st["y"]
    if kind == "train":
        st["net"].forward(st["x"], st["y"])
        return dict(y=st["y"], g=st["net"].backward(st["dy"]))
    s, doms, out = st["s"], st["doms"], st["out"]
    if kind == "restart":
        phi, u, idx = st["fields"]
        s.write_fields(phi, u, idx if len(doms[0]["crystals"]) > 1 else None)
    s.step(st["steps"])
    res = {}
    if st["measure"]:
        x, y, z = (int(v) for v in doms[0]["seeds"][0][:3])
        # the solid fraction is not returned: for a seed in a large box it is a sum of the rounding errors of 1 + phi
        res["tips"], _, res["conserved"] = s.measure(x, y, z)
    at = 0
    for k, d in enumerate(doms):
        n = 2 * d["nx"] * d["ny"] * d["nz"]
        L.lbpf_read_fields(s.ctx, k, L.LBPF_READ_PHI | L.LBPF_READ_U, out[at:at + n])
        at += n
    return dict(res, fields=out)


def work(case):
    kind = case["kind"]
    if kind == "layer":
        px = case["n"] * case["H"] * case["W"]
        ci, co = case["cin"], case["cout"]
        return {"bytes": px * (2 * ci + 2 * co) * 4 + 9 * ci * co * (2 + 2 + 4), "flops": 3 * 18 * px * ci * co}
    if kind in ("forward", "train"):
        px, lv = case["n"] * case["H"] * case["W"], case["levels"]
        level = [0, 0] + [k for k in range(1, lv) for _ in "ab"] + [k for k in range(lv - 2, -1, -1) for _ in "ab"]
        conv = sum(18 * (px >> 2 * k) * ci * co for k, (ci, co) in zip(level, _layers(lv, case["base"])))
        par = sum(9 * ci * co for ci, co in _layers(lv, case["base"]))
        return {"bytes": px * 7 * 4 + par * 4 + (px * 2 * 4 + par * 4 if kind == "train" else 0),
                "flops": conv * (3 if kind == "train" else 1)}
    qg, qu = {"d2q9": (9, 5), "d3q15": (15, 7), "d3q19": (19, 7), "d3q27": (27, 7)}[case["lattice"]]
    r, s = (8, 8) if case["precision"] == "fp64" else (4, 4) if case["precision"] == "fp32" else (4, 2)
    stored = qg + qu - (2 if s == 2 else 0)
    sites = sum(d["nx"] * d["ny"] * d["nz"] for d in _domains(case, 0))
    per_step = 2 * stored * s + 4 * r
    return {"bytes": sites * (case["steps"] * per_step + 2 * r + (2 * r if kind == "restart" else 0)),
            "flops": sites * case["steps"] * (14 * qg + 6 * qu + 100)}


# --- the same results in 64 bits, by plain torch ---------------------------

def _lattice(name):
    """(phi directions and weights, u directions and weights, e^2 of u); e^2 of phi is 1/3."""
    axes2 = [(1, 0, 0), (0, 1, 0), (-1, 0, 0), (0, -1, 0)]
    if name == "d2q9":
        dg = [(1, 1, 0), (-1, 1, 0), (-1, -1, 0), (1, -1, 0)]
        return ([(0, 0, 0)] + axes2 + dg, [4 / 9] + [1 / 9] * 4 + [1 / 36] * 4,
                [(0, 0, 0)] + axes2, [1 / 3] + [1 / 6] * 4, 1 / 3)
    axes = axes2 + [(0, 0, 1), (0, 0, -1)]
    every = [(x, y, z) for x in (-1, 0, 1) for y in (-1, 0, 1) for z in (-1, 0, 1)]
    edges = [e for e in every if sum(map(abs, e)) == 2]
    corners = [e for e in every if sum(map(abs, e)) == 3]
    w0, wa, we, wc = {"d3q15": (2 / 9, 1 / 9, 0, 1 / 72), "d3q19": (1 / 3, 1 / 18, 1 / 36, 0),
                      "d3q27": (8 / 27, 2 / 27, 1 / 54, 1 / 216)}[name]
    e, w = [(0, 0, 0)] + axes, [w0] + [wa] * 6
    if we:
        e, w = e + edges, w + [we] * 12
    if wc:
        e, w = e + corners, w + [wc] * 8
    return e, w, [(0, 0, 0)] + axes, [1 / 4] + [1 / 8] * 6, 1 / 4


def _at(f, e, bc):
    """f at x + e: periodic, or the mirror image beyond a wall."""
    for axis, k in enumerate(e):
        if not k:
            continue
        dim = 2 - axis
        if bc >> axis & 1:
            n = f.shape[dim]
            i = (torch.arange(n, device=f.device) + k).abs()
            f = f.index_select(dim, torch.where(i > n - 1, 2 * (n - 1) - i, i))
        else:
            f = torch.roll(f, -k, dim)
    return f


def _refill(pop, dirs, bc):
    """At walls: a population from beyond a wall is its mirror image's, axis by axis."""
    for axis in range(3):
        if not bc >> axis & 1:
            continue
        dim = 2 - axis
        for k, e in enumerate(dirs):
            if e[axis]:
                m = dirs.index(tuple(-v if a == axis else v for a, v in enumerate(e)))
                at = 0 if e[axis] > 0 else pop[k].shape[dim] - 1
                pop[k].select(dim, at).copy_(pop[m].select(dim, at))


def _grad(phi, case, dirs, w):
    G = [torch.zeros_like(phi) for _ in range(3)]
    if case["grad"] == "dd":
        for k, e in enumerate(dirs):
            first = next((v for v in e if v), 0)
            if first <= 0:
                continue
            d = (_at(phi, e, case["bc"]) - _at(phi, tuple(-v for v in e), case["bc"])) * (3.0 * w[k])
            for a in range(3):
                if e[a]:
                    G[a] += e[a] * d
    else:
        for a in range(2 if case["lattice"] == "d2q9" else 3):
            e = tuple(int(a == b) for b in range(3))
            G[a] = 0.5 * (_at(phi, e, case["bc"]) - _at(phi, tuple(-v for v in e), case["bc"]))
    return G


def _aniso(case, dom, G, idx):
    """a_s and N (lattice units) of the site's crystal; 1 and 0 where there is none or no gradient."""
    g2 = G[0] ** 2 + G[1] ** 2 + G[2] ** 2
    g = g2.clamp(min=1e-300).sqrt()
    on = g2 > 1e-20
    if idx is None:
        eps, phi0 = dom["crystals"][0]
    else:
        on = on & (idx > 0)
        tab = torch.tensor([(0.0, 0.0)] + dom["crystals"], dtype=torch.float64, device=g2.device)
        eps, phi0 = tab[idx.long(), 0], tab[idx.long(), 1]
    form, gam = case["form"], case["gamma"]
    if form == "angle":
        q = case["q"]
        t = q * (torch.atan2(-G[1], -G[0]) - phi0)
        a, ap = 1 + eps * torch.cos(t), -eps * q * torch.sin(t)
        N = [-a * ap * G[1], a * ap * G[0], torch.zeros_like(a)]
    else:
        m = [c / g for c in G]
        x2, y2, z2 = (c * c for c in m)
        if form == "cubic100":
            a = 1 - 3 * eps + 4 * eps * (x2 * x2 + y2 * y2 + z2 * z2)
            d = [16 * eps * s * c for s, c in zip((x2, y2, z2), m)]
        elif form == "y66":
            a = 1 + eps * (x2 ** 3 - 15 * x2 * x2 * y2 + 15 * x2 * y2 * y2 - y2 ** 3)
            d = [eps * m[0] * (6 * x2 * x2 - 60 * x2 * y2 + 30 * y2 * y2),
                 eps * m[1] * (-30 * x2 * x2 + 60 * x2 * y2 - 6 * y2 * y2), torch.zeros_like(a)]
        else:
            S, Q = x2 * y2 * z2, x2 * x2 + y2 * y2 + z2 * z2
            dS = [2 * m[0] * y2 * z2, 2 * m[1] * x2 * z2, 2 * m[2] * x2 * y2]
            if form == "hoyt110":
                a = 1 + eps * (Q - 0.6) + gam * (3 * Q + 66 * S - 17 / 7)
                d = [(4 * eps + 12 * gam) * s * c + 66 * gam * t for s, c, t in zip((x2, y2, z2), m, dS)]
            else:
                a = 1 + 66 * gam * S
                d = [66 * gam * t for t in dS]
        md = m[0] * d[0] + m[1] * d[1] + m[2] * d[2]
        N = [g * a * (dc - c * md) for dc, c in zip(d, m)]
    zero = torch.zeros_like(g2)
    return torch.where(on, a, torch.ones_like(g2)), [torch.where(on, c, zero) for c in N]


def _lb_exact(case, dom):
    p, bc = SETS[case["params"]], case["bc"]
    eg, wg, eu, wu, e2u = _lattice(case["lattice"])
    D = p["W0"] ** 2 / p["tau0"] * p["dt"] / p["dx"] ** 2
    qphi = p["dt"] / p["tau0"]
    lam = p["lam"] if p["lam"] > 0 else p["kappa"] * p["tau0"] / (0.6267 * p["W0"] ** 2)
    ieta_u = 1.0 / (p["kappa"] * p["dt"] / (e2u * p["dx"] ** 2) + 0.5)
    adv = [v * p["dt"] / (p["dx"] * e2u) for v in _velocity(case)]
    ea = [sum(c * v for c, v in zip(e, adv)) for e in eu]
    phi, u, idx = _profile(case, dom, torch.float64)
    xi = 1e-7 * p["dx"]
    G = _grad(phi, case, eg, wg)
    if len(dom["crystals"]) == 1:
        idx = None
    elif case["kind"] == "lb":  # a seeded start keeps the index inside and near the seeds
        idx = torch.where((phi > 0) | (G[0] ** 2 + G[1] ** 2 + G[2] ** 2 > xi * xi), idx, torch.zeros_like(idx))
    a, N = _aniso(case, dom, G, idx)
    g = [w * (phi - 3 * D * sum(c * n for c, n in zip(e, N) if c)) if any(e) else w * phi for e, w in zip(eg, wg)]
    f = [w * u * (1 + t) for w, t in zip(wu, ea)]
    for _ in range(case["steps"]):
        G = _grad(phi, case, eg, wg)
        if idx is not None:
            take, new = (idx == 0) & (G[0] ** 2 + G[1] ** 2 + G[2] ** 2 > xi * xi), idx
            for e in eg[1:]:
                new = torch.where(take & (new == 0), _at(idx, e, bc), new)
            idx = new
        a, N = _aniso(case, dom, G, idx)
        a2 = a * a
        ieta = 1 / (3 * D * a2 + 0.5)
        source = qphi * (phi - lam * u * (1 - phi * phi)) * (1 - phi * phi)
        for k, e in enumerate(eg):
            eq = phi if not any(e) else phi - 3 * D * sum(c * n for c, n in zip(e, N) if c)
            back = tuple(-v for v in e)
            post = (g[k] - (g[k] - wg[k] * eq) * ieta + wg[k] * source) / a2
            g[k] = _at(post, back, bc) - _at((1 - a2) / a2, back, bc) * g[k]
        del G, a, N, a2, ieta, source, post
        _refill(g, eg, bc)
        new = sum(g)
        half = 0.5 * (new - phi)
        for k, e in enumerate(eu):
            f[k] = _at(f[k] - (f[k] - wu[k] * (1 + ea[k]) * u) * ieta_u + wu[k] * half, tuple(-v for v in e), bc)
        _refill(f, eu, bc)
        phi, u = new, sum(f)
    return phi, u


def _conv(x, w, b=None, relu=False):
    """Periodic 3x3 convolution, NHWC; w (9, cout, cin)."""
    y = 0.0
    for t in range(9):
        y = y + torch.roll(x, (1 - t // 3, 1 - t % 3), (1, 2)) @ w[t].T
    y = y if b is None else y + b
    return y.relu() if relu else y


def _net_exact(case, p, X):
    lv, base, at, k = case["levels"], case["base"], 0, []
    for cin, cout in _layers(lv, base):
        n = 9 * cin * cout
        k.append((p[at:at + n].view(9, cout, cin), p[at + n:at + n + cout]))
        at += n + cout
    hw, hb = p[at:at + 2 * base].view(2, base), p[at + 2 * base:]
    h = torch.cat([X, X.new_zeros(X.shape[:3] + (11,))], -1)
    k, skip = iter(k), []
    for l in range(lv):
        if l:
            n, H, W, c = h.shape
            h = h.view(n, H // 2, 2, W // 2, 2, c).mean((2, 4))
        h = _conv(h, *next(k), relu=True)
        h = _conv(h, *next(k), relu=True)
        skip.append(h)
    for l in range(lv - 2, -1, -1):
        h = torch.cat([h.repeat_interleave(2, 1).repeat_interleave(2, 2), skip[l]], -1)
        h = _conv(h, *next(k), relu=True)
        h = _conv(h, *next(k), relu=True)
    y = h @ hw.T + hb
    return torch.stack([y[..., 0] * (1 - X[..., 0] ** 2), y[..., 1]], -1)


def exact(case, seed):
    kind = case["kind"]
    if kind == "layer":
        x, w, b, dy = (t.double() for t in _layer_input(case, seed))
        xx = [torch.roll(x, (1 - t // 3, 1 - t % 3), (1, 2)).reshape(-1, case["cin"]) for t in range(9)]
        dw = torch.stack([dy.reshape(-1, case["cout"]).T @ v for v in xx])
        del xx
        return dict(y=_conv(x, w, b, True), dx=_conv(dy, w.flip(0).transpose(1, 2)), dw=dw)
    if kind in ("forward", "train"):
        X = _net_input(case, seed)
        p = torch.from_numpy(_weights(case, seed)).cuda().double()
        if kind == "forward":
            return _net_exact(case, p, X.double())
        p.requires_grad_(True)
        y = _net_exact(case, p, X.double())
        y.backward(_loss_gradient(X).double())
        return dict(y=y.detach(), g=p.grad)
    out, res = [], {}
    for dom in _domains(case, seed):
        phi, u = _lb_exact(case, dom)
        out += [phi.reshape(-1), u.reshape(-1)]
    if case["measure"]:
        res = dict(tips=None, conserved=None)
        if not case["bc"]:
            res["conserved"] = float((u - phi / 2).sum())
    return dict(res, fields=torch.cat(out))
