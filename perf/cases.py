"""What a user of this framework has it do, as cases whose speed and outputs can be measured.

A case is a dict of plain values; `prepare` makes what the user's program has in hand (the model
with its parameters, points, targets, a volume, a camera), `run` makes one pass through the public
entry points (`SRN`, `TiledVolume`, `APMGSRNFunction`), `work` states what that pass cannot do
without and `exact` is the same in 64-bit torch, without the package.

`op` is the entry point a case goes through:
  query        SRN.forward at points in memory
  grad         SRN.backward at points and targets in memory: L_rec, and with `density` L_den
  autograd     APMGSRNFunction forward and backward with an upstream gradient
  train        sample_points, sample_target and backward: an iteration of a user's own optimiser
  train_step   SRN.train_step on a stream of its own (the library's Adam, replayed as a graph)
  render       SRN.render of a whole frame
  progressive  SRN.render_progressive: one pass of an interactive viewer and its preview
  decode       SRN.decode of the whole lattice
"""
import math

import numpy as np
import torch

#: (n_grids, res, channels): the 16 -> 64 -> 64 -> 1 model of the small configuration, the other
#: widths and an odd resolution of the parity tests, and the paper-scale model.
SHAPES = [(8, 16, 2), (16, 9, 1), (16, 16, 2), (32, 20, 2), (64, 32, 2)]
ADAM = {"beta1": 0.9, "beta2": 0.99, "eps": 1e-8}
CHUNK = 1 << 16   # points at a time in the 64-bit evaluation


def _case(name, op, prec, shape, **more):
    m, r, c = shape
    return {"name": name, "op": op, "prec": prec, "grids": m, "res": r, "channels": c, "zoom": 0.0, **more}


def listed():
    small, mid, k32, paper = SHAPES[0], SHAPES[3], SHAPES[2], SHAPES[4]
    return [
        # A probe of a few points, as an interactive tool asks for: latency and launches.
        _case("query-few", "query", "fp32", small, bricks=1, points=1000, sorted=False),
        # Values of a trained model at points of the caller's own, in no order, an odd number of them.
        _case("query-bf16", "query", "bf16", paper, bricks=1, points=1_000_003, sorted=False, zoom=0.4),
        # The same in full precision through a small decomposition with uneven shares.
        _case("query-fp32", "query", "fp32", mid, bricks=4, points=200_003, sorted=False, zoom=0.4),
        # The small training configuration: a 64^3 volume, 16384 points, every step a graph replay.
        _case("step-small", "train_step", "fp32", small, bricks=1, points=16384, vox=64, density=True),
        # The paper-scale model's gradients on a sampler-ordered batch, in each precision.
        _case("grad-fp32", "grad", "fp32", paper, bricks=1, points=1 << 18, sorted=True, density=True),
        _case("grad-bf16", "grad", "bf16", paper, bricks=1, points=1 << 18, sorted=True, density=True),
        # A loss of the user's own through torch.autograd, on points in no order.
        _case("autograd-bf16", "autograd", "bf16", mid, bricks=1, points=100_003, sorted=False, through_g=False),
        # The benchmark's iteration: 8 uneven bricks of a 1024^3 volume, density loss, BF16.
        _case("train-bricks", "train", "bf16", paper, bricks=8, points=2_653_469, vox=1024, density=True),
        # The larger single-model batch, transforms fixed (their early stop has fired).
        _case("step-bf16", "train_step", "bf16", paper, bricks=1, points=1 << 20, vox=512, density=False),
        # A frame through the 8-brick model.
        _case("frame", "render", "bf16", paper, bricks=8, width=1024, height=1024, samples=512, ortho=False,
              batch=1 << 22),
        # An interactive viewer's pass: the first level of a VGA view, with its preview.
        _case("preview", "progressive", "bf16", k32, bricks=1, width=640, height=480, samples=256, ortho=True,
              first=4800, count=14400, batch=1 << 21),
        # Decompression of a whole (odd) lattice through the 8-brick model.
        _case("decode", "decode", "bf16", paper, bricks=8, vox=319, batch=1 << 22, zoom=0.4),
    ]


def draw(rng):
    def spread(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    op = rng.choice(["query", "query", "grad", "grad", "autograd", "train", "train_step", "render", "progressive",
                     "decode"])
    prec = rng.choice(["bf16", "bf16", "fp32"])
    shape = rng.choice(SHAPES + SHAPES[4:])
    c = {"op": op, "prec": prec, "grids": shape[0], "res": shape[1], "channels": shape[2],
         "zoom": rng.choice([0.0, 0.0, 0.4]), "bricks": rng.choice([1, 1, 2, 4, 8])}
    if op == "query":
        c |= {"points": spread(500, 2_000_000), "sorted": rng.random() < 0.3}
    elif op == "grad":
        c |= {"points": spread(4096, 1_000_000), "sorted": rng.random() < 0.8, "density": rng.random() < 0.7}
    elif op == "autograd":
        c |= {"points": spread(2000, 300_000), "sorted": rng.random() < 0.3, "through_g": rng.random() < 0.3}
    elif op in ("train", "train_step"):
        c |= {"points": spread(8192, 1_500_000), "vox": rng.choice([64, 127, 256, 512]), "density": op == "train"}
    elif op in ("render", "progressive"):
        w = spread(96, 800)
        c |= {"width": w, "height": max(64, int(w * rng.uniform(0.5, 1.2))), "samples": spread(32, 512),
              "ortho": rng.random() < 0.5, "batch": 1 << rng.randint(18, 22)}
        if op == "progressive":
            n = c["width"] * c["height"]
            c["first"] = rng.choice([0, n // 64, n // 16])
            c["count"] = min(n - c["first"], spread(256, 30_000))
    else:
        c |= {"vox": spread(33, 300), "batch": 1 << rng.randint(18, 22)}
    return c


# ----------------------------------------------------------------- inputs, from the seed alone
def _shape(c):
    return c["grids"], c["res"], c["channels"], c["grids"] * c["channels"]


def _grid(c):
    """The bricks of a decomposition as I x J x K."""
    return {1: (1, 1, 1), 2: (2, 1, 1), 4: (2, 2, 1), 8: (2, 2, 2)}[c["bricks"]]


def _boxes(c, ghost=2):
    """Voxel boxes (lo xyz, hi xyz) of the bricks with ghost cells, x fastest."""
    v, g, out = c.get("vox", 1024), _grid(c), []
    for k in range(g[2]):
        for j in range(g[1]):
            for i in range(g[0]):
                w = [v // n for n in g]
                lo = [max(0, a * x - ghost) for a, x in zip((i, j, k), w)]
                hi = [v - 1 if a == n - 1 else min(v - 1, a * x + x - 1 + ghost) for a, x, n in zip((i, j, k), w, g)]
                out.append(lo + hi)
    return np.array(out, dtype=np.int64)


def _offsets(c, seed):
    """Uneven shares of the batch, U[2^16, 2^19] against one another as in the benchmark."""
    share = np.random.default_rng(seed).uniform(2.0 ** 16, 2.0 ** 19, c["bricks"])
    cut = np.floor(np.cumsum(share) / share.sum() * c["points"]).astype(np.int64)
    cut[-1] = c["points"]
    return [0] + [int(v) for v in cut]


def _params(c, gen):
    """Per brick: features and decoder of a trained size, transforms near the identity; `zoom`
    shrinks and moves the grids' supports as training does."""
    m, r, ch, k = _shape(c)
    b = c["bricks"]

    def uni(shape, a):
        return (torch.rand(shape, device="cuda", generator=gen) * 2 - 1) * a

    p = {"F": uni((b, m, r, r, r, ch), 0.5), "W1": uni((b, 64, k), math.sqrt(6 / k)),
         "W2": uni((b, 64, 64), math.sqrt(6 / 64)), "w3": uni((b, 64), math.sqrt(6 / 64))}
    g = torch.randn((b, m, 3, 4), device="cuda", generator=gen) * 0.05
    for d in range(3):
        g[..., d, d] += 1
    if c["zoom"]:
        g[..., :3] *= 1 + c["zoom"] * torch.rand((b, m, 1, 1), device="cuda", generator=gen)
        g[..., 3] += uni((b, m, 3), 0.3)
    p["G"] = g
    return p


def _bin_code(x):
    """Morton code of a point's bin of 32^3, as a sampler-ordered batch is sorted by."""
    q = ((x.double() + 1) * 16).floor().clamp(0, 31).long()
    code = torch.zeros(len(x), dtype=torch.int64, device=x.device)
    for bit in range(5):
        for a in range(3):
            code |= ((q[:, a] >> bit) & 1) << (3 * bit + a)
    return code


def _points(c, off, gen):
    x = torch.rand((c["points"], 3), device="cuda", generator=gen) * 2 - 1
    if c["sorted"]:
        for a, b in zip(off, off[1:]):
            x[a:b] = x[a:b][torch.argsort(_bin_code(x[a:b]), stable=True)]
    return x


def _targets(x, gen):
    """A field with structure at several scales, and the noise of measured data."""
    ph = torch.rand((8, 3), device="cuda", generator=gen) * 6.28
    v = torch.full((len(x),), 0.5, device="cuda")
    for j in range(8):
        k = 1.5 ** j
        v += 0.25 / (j + 1) * torch.cos(k * x + ph[j]).prod(1)
    return v + 0.02 * torch.randn(len(x), device="cuda", generator=gen)


def _volume(c, gen):
    """[z][y][x] float32 sum of separable waves of wave numbers 1 to 64, near [0, 1]."""
    v, n = c["vox"], 24
    k = 64.0 ** torch.rand((3, n, 1), device="cuda", generator=gen)
    ph = torch.rand((3, n, 1), device="cuda", generator=gen) * 6.28
    ax = torch.linspace(0, 3.14159, v, device="cuda")
    amp = (k.pow(2).sum(0).sqrt() ** (-5 / 6)) * 0.3
    wz, wy, wx = (torch.cos(k[d] * ax + ph[d]) for d in range(3))
    vol = torch.empty((v, v, v), device="cuda")
    for z in range(v):
        vol[z] = (wy * amp * wz[:, z:z + 1]).T @ wx
    return vol.add_(0.5)


def _camera(c, seed):
    r = np.random.default_rng(seed)
    th, phi = r.uniform(0, 2 * math.pi), r.uniform(-0.6, 0.6)
    eye = 3 * np.array([math.cos(phi) * math.sin(th), math.sin(phi), math.cos(phi) * math.cos(th)])
    fwd = -eye / 3
    right = np.cross(fwd, [0.0, 1.0, 0.0])
    right /= np.linalg.norm(right)
    f32 = {"eye": eye, "forward": fwd, "right": right, "up": np.cross(right, fwd),
           "scale": math.sqrt(3) if c["ortho"] else math.tan(math.radians(22.5))}
    return {k: np.float32(v) for k, v in f32.items()} | {"ortho": c["ortho"]}


def _lut(seed):
    """A piecewise-linear transfer function of 8 random knots."""
    r = np.random.default_rng(seed + 1)
    pos = np.concatenate([[0.0], np.sort(r.random(6)), [1.0]])
    val = r.random((8, 4)) * [1, 1, 1, 0.01]
    return np.stack([np.interp(np.arange(256) / 255, pos, val[:, k]) for k in range(4)], 1).astype(np.float32)


def _inputs(c, seed):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    s = {"p": _params(c, gen)}
    if "points" in c:
        s["off"] = _offsets(c, seed)
    if c["op"] in ("query", "grad", "autograd"):
        s["xyz"] = _points(c, s["off"], gen)
        if c["op"] == "grad":
            s["target"] = _targets(s["xyz"], gen)
        if c["op"] == "autograd":
            s["up"] = torch.randn(c["points"], device="cuda", generator=gen) / c["points"]
    elif c["op"] in ("train", "train_step"):
        s["vol"] = _volume(c, gen)
    elif c["op"] in ("render", "progressive"):
        s["cam"], s["lut"] = _camera(c, seed), torch.as_tensor(_lut(seed), device="cuda")
    return s


# The learning rates of a late training phase: after two cuts of the plateau schedule and a finer one.
LATE_LR = 1e-5


def prepare(c, seed):
    from paper_2308_02494_gb300.model import SRN, TiledVolume
    from paper_2308_02494_gb300.synth import ModelShape

    m, r, ch, _ = _shape(c)
    s = _inputs(c, seed)
    p = s.pop("p")
    s["op"], s["c"], s["seed"], s["boxes"], s["grid"] = c["op"], c, seed, _boxes(c), _grid(c)
    lr = {"lr_feat": LATE_LR, "lr_xform": LATE_LR} if c["op"] == "train_step" else {}
    net = SRN(ModelShape(m, r, ch), n_bricks=c["bricks"], precision=c["prec"],
              max_points=c.get("points") or c["batch"], **lr)
    lay = net.lay
    for k, v in p.items():
        off, size = getattr(lay, "off_" + k), getattr(lay, "size_" + k)
        flat = v.reshape(c["bricks"], -1)
        for b in range(c["bricks"]):
            net.params[off + b * size: off + b * size + flat.shape[1]] = flat[b]
    net.sync_shadow()
    s["net"] = net
    if c["op"] == "autograd":
        s["w"] = net.params.detach().requires_grad_()
    elif c["op"] in ("train", "train_step"):
        s["vol"] = TiledVolume(s["vol"])
        s["xyz"] = torch.empty((c["points"], 3), device="cuda")
        s["target"] = torch.empty(c["points"], device="cuda")
        if c["op"] == "train_step":
            torch.cuda.synchronize()
            s["stream"] = torch.cuda.Stream()
    elif c["op"] in ("render", "progressive"):
        s["rgba"] = torch.zeros((c["height"], c["width"], 4), device="cuda")
        if c["op"] == "progressive":
            s["preview"] = torch.zeros_like(s["rgba"])
            if c["first"]:
                _pass(s, 0, c["first"], None)
    elif c["op"] == "decode":
        s["out"] = torch.empty((c["vox"],) * 3, device="cuda")
    elif c["op"] == "query":
        s["out"] = torch.empty(c["points"], device="cuda")
    torch.cuda.synchronize()
    return s


def _pass(s, first, count, preview):
    c = s["c"]
    return s["net"].render_progressive(s["cam"], s["lut"], 0.0, 1.0, c["width"], c["height"], c["samples"], s["grid"],
                                       s["boxes"], c.get("vox", 1024), first, count, s["rgba"], preview)


def _parts(flat, lay):
    """The flat gradient (or parameter) buffer by tensor, all bricks of each together."""
    n = {"F": lay.off_W1, "W1": lay.off_W2, "W2": lay.off_w3, "w3": lay.off_G, "G": lay.n_params}
    return {k: flat[getattr(lay, "off_" + k):end] for k, end in n.items()}


def run(s):
    op, c, net = s["op"], s["c"], s["net"]
    if op == "query":
        return net.forward(s["xyz"], s["off"], out=s["out"])
    if op == "grad":
        losses = net.backward(s["xyz"], s["target"], s["off"], density=c["density"])
        return {"losses": losses, "grads": _parts(net.grads, net.lay)}
    if op == "autograd":
        from paper_2308_02494_gb300.model import APMGSRNFunction
        f = APMGSRNFunction.apply(s["xyz"], s["w"], net, s["off"], c["through_g"])
        (g,) = torch.autograd.grad(f, s["w"], s["up"])
        return {"f": f.detach(), "grads": _parts(g, net.lay)}
    if op == "train":
        # (the sampler leaves the points of a bin in any order, so the points themselves are
        # not among the outputs)
        net.sample_points(s["seed"], 0, s["off"], s["xyz"])
        net.sample_target(s["vol"], s["boxes"], s["xyz"], s["off"], s["target"])
        losses = net.backward(s["xyz"], s["target"], s["off"], density=c["density"])
        return {"losses": losses, "grads": _parts(net.grads, net.lay)}
    if op == "train_step":
        losses = net.train_step(s["seed"], s["vol"], s["boxes"], s["off"], c["density"], s["xyz"], s["target"],
                                stream=s["stream"])
        return {"losses": losses, "grads": _parts(net.grads, net.lay), "params": _parts(net.params, net.lay),
                "m": net.adam_m, "v": net.adam_v}
    if op == "render":
        return net.render(s["cam"], s["lut"], 0.0, 1.0, c["width"], c["height"], c["samples"], s["grid"], s["boxes"],
                          c.get("vox", 1024), rgba=s["rgba"])
    if op == "progressive":
        return {"rgba": _pass(s, c["first"], c["count"], s["preview"]), "preview": s["preview"]}
    return net.decode(s["grid"], s["boxes"], c["vox"], out=s["out"])


# ----------------------------------------------------------------- what a pass cannot do without
def work(c):
    m, r, ch, k = _shape(c)
    nodes, dec = m * r ** 3 * ch * c["bricks"], (64 * k + 64 * 64 + 64)
    par = (nodes + c["bricks"] * (dec + 12 * m))
    stored = (2 if c["prec"] == "bf16" else 4) * nodes + 4 * c["bricks"] * (dec + 12 * m)
    fwd = m * (18 + 12 + 14 * ch) + 2 * dec              # Eq. 1, cell and weights, Eq. 2, decoder
    bwd = m * (12 + 16 * ch) + 4 * dec                   # adjoint of Eq. 2, decoder gradients
    den = m * 2 * (18 + 20) + m * 32 if c.get("density") else 0
    op = c["op"]
    if op in ("render", "progressive"):
        n = c["count"] if op == "progressive" else c["width"] * c["height"]
        seen = 32 * c["width"] * c["height"] if op == "progressive" else 16 * n
        return {"bytes": stored + seen, "flops": n * c["samples"] * (fwd + 20) / 2}   # about half the rays' span hits
    if op == "decode":
        return {"bytes": stored + 4 * c["vox"] ** 3, "flops": c["vox"] ** 3 * fwd}
    n = c["points"]
    if op == "query":
        return {"bytes": stored + 16 * n, "flops": n * fwd}
    b = {"bytes": stored + 4 * par + 16 * n, "flops": n * (fwd + bwd + den)}
    if op in ("train", "train_step"):
        b["bytes"] += 32 * n
    if op == "train_step":
        b["bytes"] += 24 * par + (2 * nodes if c["prec"] == "bf16" else 0)
        b["flops"] += 12 * par
    return b


# ----------------------------------------------------------------- the same in 64 bits
def _corners(w):
    for k in range(8):
        sel = [w[..., a] if (k >> a) & 1 else 1 - w[..., a] for a in range(3)]
        yield k, sel


def _encode64(P, x, r):
    """Features [n, M, C] of the points, and per corner (node index, weight), the mask and the
    weights' parts; P holds one brick's tensors in 64 bits."""
    u = torch.einsum("mde,ne->nmd", P["G"][:, :, :3], x) + P["G"][:, :, 3]
    ins = (u.abs() <= 1).all(-1)
    t = (u.clamp(-1, 1) + 1) / 2 * (r - 1)
    c = t.floor().clamp(max=r - 2)
    w = t - c
    c = c.long()
    m = u.shape[1]
    base = (c[..., 2] * r + c[..., 1]) * r + c[..., 0] + torch.arange(m, device=x.device) * r ** 3
    F = P["F"].reshape(m * r ** 3, -1)
    y = 0
    for k, (a, b, d) in _corners(w):
        node = base + (k & 1) + ((k >> 1) & 1) * r + (k >> 2) * r * r
        y = y + (a * b * d * ins)[..., None] * F[node]
    return y, (u, ins, base, w)


def _mlp64(P, y):
    z1 = y @ P["W1"].T
    h1 = z1.relu()
    z2 = h1 @ P["W2"].T
    return z1, h1, z2, z2.relu() @ P["w3"]


def _query64(P, x, r):
    out = [torch.zeros(0, dtype=torch.float64, device=x.device)]
    for i in range(0, len(x), CHUNK):
        y, _ = _encode64(P, x[i:i + CHUNK].double(), r)
        out.append(_mlp64(P, y.flatten(1))[3])
    return torch.cat(out)


def _grads64(P, x, target, r, c, up=None, density=False, through_g=False):
    """One brick's losses [4] and gradients; `up`: an upstream dL/df in the target's place."""
    n, g = len(x), {k: torch.zeros_like(v) for k, v in P.items()}
    dF = g["F"].view(-1, c["channels"])
    fs = []
    for i in range(0, n, CHUNK):
        q = x[i:i + CHUNK].double()
        y, (u, ins, base, w) = _encode64(P, q, r)
        y = y.reshape(len(q), -1)
        z1, h1, z2, f = _mlp64(P, y)
        fs.append(f)
        d = up[i:i + CHUNK].double() if up is not None else 2 / n * (f - target[i:i + CHUNK].double())
        g["w3"] += z2.relu().T @ d
        d2 = d[:, None] * P["w3"] * (z2 > 0)
        g["W2"] += d2.T @ h1
        d1 = (d2 @ P["W2"]) * (z1 > 0)
        g["W1"] += d1.T @ y
        dy = (d1 @ P["W1"]).view(len(q), -1, c["channels"])
        du = [0, 0, 0]
        for k, s in _corners(w):
            node = base + (k & 1) + ((k >> 1) & 1) * r + (k >> 2) * r * r
            dF.index_add_(0, node.reshape(-1), ((s[0] * s[1] * s[2] * ins)[..., None] * dy).reshape(-1, dF.shape[1]))
            if through_g:
                e = (dy * P["F"].reshape(dF.shape)[node]).sum(-1) * ins * (r - 1) / 2
                for a in range(3):
                    du[a] = du[a] + (1 if (k >> a) & 1 else -1) * s[(a + 1) % 3] * s[(a + 2) % 3] * e
        if through_g:
            du = torch.stack(du, -1)
            g["G"][:, :, :3] += torch.einsum("nmd,ne->mde", du, q)
            g["G"][:, :, 3] += du.sum(0)
    f = torch.cat(fs)
    los = [0.0, 0.0, 0.0, float(n)]
    if up is None:
        h = (f - target.double()) ** 2
        los[0] = float(h.mean())
        if density:
            los[1], los[2], g["G"] = _density64(P["G"], x, h)
    return f, torch.tensor(los, dtype=torch.float64, device=x.device), g


def _density64(G, x, h, eps=1e-8):
    """L_den (Eq. 7-9, p = 10, the target density held constant), the sum of rho, and dL_den/dG."""
    G = G.clone().requires_grad_()
    det = torch.linalg.det(G[:, :, :3])

    def rho_of(q):
        u = torch.einsum("mde,ne->nmd", G[:, :, :3], q) + G[:, :, 3]
        return (torch.exp(-((u * u) ** 10).sum(-1)) * det).sum(-1)

    with torch.no_grad():
        rho = torch.cat([rho_of(q.double()) for q in x.split(CHUNK)])
    tot = rho.sum().requires_grad_()
    rho.requires_grad_()
    lr = torch.log(rho / tot + eps)
    ls = (h.mean() / (h + eps) * lr).detach()
    loss = (ls.exp() * (ls - lr)).mean()
    d_rho, d_tot = torch.autograd.grad(loss, (rho, tot))
    dG = torch.zeros_like(G)
    for i in range(0, len(x), CHUNK):
        part = (rho_of(x[i:i + CHUNK].double()) * (d_rho[i:i + CHUNK] + d_tot)).sum()
        dG += torch.autograd.grad(part, G, retain_graph=True)[0]
    return float(loss), float(tot), dG


def _philox(n, brick, step, seed):
    """The sampler's draws: Philox4x32-10 with counter (n, brick, step, 0) and the seed as key."""
    mask = 0xFFFFFFFF

    def mul(a, b):   # high and low words of a constant's product with words b
        lo, hi = a * (b & 0xFFFF), a * (b >> 16)
        mid = (lo >> 16) + (hi & 0xFFFF)
        return (hi >> 16) + (mid >> 16), ((mid & 0xFFFF) << 16) | (lo & 0xFFFF)

    z = torch.zeros(n, dtype=torch.int64, device="cuda")
    c = [torch.arange(n, device="cuda"), z + brick, z + step, z]
    k0, k1 = seed & mask, (seed >> 32) & mask
    for r in range(10):
        if r:
            k0, k1 = (k0 + 0x9E3779B9) & mask, (k1 + 0xBB67AE85) & mask
        h0, l0 = mul(0xD2511F53, c[0])
        h1, l1 = mul(0xCD9E8D57, c[2])
        c = [h1 ^ c[1] ^ k0, l1, h0 ^ c[3] ^ k1, l0]
    return torch.stack([2.0 * (v >> 8).double() * 2.0 ** -24 - 1 for v in c[:3]], 1)


def _lookup64(vol, box, x):
    """The volume at brick-local points: trilinear, corner-aligned to the brick's box."""
    lo = torch.tensor(box[:3], dtype=torch.float64, device="cuda")
    hi = torch.tensor(box[3:], dtype=torch.float64, device="cuda")
    t = lo + (x + 1) / 2 * (hi - lo)
    c = torch.minimum(t.floor(), hi - 1)
    w, c, out = t - c, c.long(), 0
    for k, (a, b, d) in _corners(w):
        out = out + a * b * d * vol[c[:, 2] + (k >> 2), c[:, 1] + ((k >> 1) & 1), c[:, 0] + (k & 1)]
    return out


def _render64(c, s, brick, pixels):
    """RGBA of the given flat pixels: slab test, midpoint samples, brick hash, transfer function."""
    cam, w, h, n = s["cam"], c["width"], c["height"], c["samples"]
    t64 = {k: torch.tensor(np.asarray(cam[k], dtype=np.float64), device="cuda") for k in ("eye", "forward", "right", "up")}
    px, py = (pixels % w).double(), (pixels // w).double()
    sc = float(cam["scale"])
    off = ((2 * (px + 0.5) / w - 1) * sc * w / h)[:, None] * t64["right"] + \
        ((1 - 2 * (py + 0.5) / h) * sc)[:, None] * t64["up"]
    if cam["ortho"]:
        org, d = t64["eye"] + off, t64["forward"].expand_as(off)
    else:
        d = t64["forward"] + off
        org, d = t64["eye"].expand_as(off), d / d.norm(dim=1, keepdim=True)
    ta, tb = (-1 - org) / d, (1 - org) / d
    t0 = torch.minimum(ta, tb).max(1).values.clamp(min=0)
    t1 = torch.maximum(ta, tb).min(1).values
    dt = ((t1 - t0) / n).clamp(min=0)
    vox, grid = c.get("vox", 1024), torch.tensor(_grid(c), device="cuda")
    box = torch.tensor(_boxes(c), dtype=torch.float64, device="cuda")
    p = org[:, None] + (t0[:, None] + (torch.arange(n, device="cuda") + 0.5) * dt[:, None])[..., None] * d[:, None]
    cell = torch.minimum((grid * (p + 1) / 2).floor().long().clamp(min=0), grid - 1)
    b = cell[..., 0] + grid[0] * (cell[..., 1] + grid[1] * cell[..., 2])
    loc = ((p + 1) / 2 * (vox - 1) - box[b, :3]) / (box[b, 3:] - box[b, :3]) * 2 - 1
    f = torch.zeros(b.shape, dtype=torch.float64, device="cuda")
    for k in range(c["bricks"]):
        sel = (b == k) & (t1 > t0)[:, None]
        f[sel] = _query64(brick(k), loc[sel], c["res"])
    pos = f.clamp(0, 1) * 255
    i0 = pos.floor().clamp(max=254).long()
    lut = s["lut"].double()
    rgba = torch.lerp(lut[i0], lut[i0 + 1], (pos - i0)[..., None])
    alpha = 1 - torch.exp(-rgba[..., 3] * dt[:, None] / (2 / 512))
    keep = torch.cumprod(1 - alpha, 1)
    before = torch.cat([torch.ones_like(keep[:, :1]), keep[:, :-1]], 1)
    return torch.cat([((before * alpha)[..., None] * rgba[..., :3]).sum(1), 1 - keep[:, -1:]], 1)


def _pixel_order(c):
    """The progressive order: a level's pixels that no coarser level holds, row by row."""
    w, h, out, step = c["width"], c["height"], [torch.zeros(1, dtype=torch.int64)], 1
    while step < max(w, h):
        step *= 2
    y, x = torch.meshgrid(torch.arange(h), torch.arange(w), indexing="ij")
    while step > 1:
        f, step = step, step // 2
        sel = (y % step == 0) & (x % step == 0) & ~((y % f == 0) & (x % f == 0))
        out.append((y * w + x)[sel])
    return torch.cat(out)


def exact(c, seed):
    op = c["op"]
    samples = c["samples"] * (c["first"] + c["count"] if op == "progressive" else c["width"] * c["height"]) \
        if op in ("render", "progressive") else c["vox"] ** 3 if op == "decode" else c["points"]
    if samples * c["grids"] > 6e9:
        return None   # over about 20 seconds
    s = _inputs(c, seed)
    r = c["res"]

    def brick(b):
        return {k: v[b].double() for k, v in s["p"].items()}

    if op == "query":
        return torch.cat([_query64(brick(b), s["xyz"][i:j], r) for b, (i, j) in enumerate(zip(s["off"], s["off"][1:]))])
    if op == "render":
        pix = torch.arange(c["width"] * c["height"], device="cuda")
        rows = [_render64(c, s, brick, q) for q in pix.split(max(1, (1 << 22) // c["samples"]))]
        return torch.cat(rows).view(c["height"], c["width"], 4)
    if op == "progressive":
        pix = _pixel_order(c)[:c["first"] + c["count"]].cuda()
        img = torch.zeros((c["width"] * c["height"], 4), dtype=torch.float64, device="cuda")
        for q in pix.split(max(1, (1 << 22) // c["samples"])):
            img[q] = _render64(c, s, brick, q)
        return {"rgba": img.view(c["height"], c["width"], 4), "preview": None}
    if op == "decode":
        v, grid, box = c["vox"], _grid(c), _boxes(c)
        own = [torch.clamp(n * torch.arange(v, device="cuda") // (v - 1), max=n - 1) for n in grid]
        out = torch.empty((v, v, v), dtype=torch.float64, device="cuda")
        for b in range(c["bricks"]):
            at = (b % grid[0], b // grid[0] % grid[1], b // (grid[0] * grid[1]))
            ax = [torch.nonzero(own[a] == at[a])[:, 0] for a in range(3)]
            loc = [(ax[a].double() - box[b][a]) / float(box[b][3 + a] - box[b][a]) * 2 - 1 for a in range(3)]
            P = brick(b)
            for z in range(len(ax[2])):
                x = torch.stack(torch.meshgrid(loc[2][z:z + 1], loc[1], loc[0], indexing="ij")[::-1], -1).view(-1, 3)
                out[ax[2][z], ax[1][0]:ax[1][-1] + 1, ax[0][0]:ax[0][-1] + 1] = _query64(P, x, r).view(len(ax[1]), -1)
        return out
    losses, f, parts = [], [], {k: [] for k in ("F", "W1", "W2", "w3", "G")}
    for b, (i, j) in enumerate(zip(s["off"], s["off"][1:])):
        P = brick(b)
        if "xyz" in s:
            x = s["xyz"][i:j]
            t = s["target"][i:j] if "target" in s else None
        else:
            x = _philox(j - i, b, 0, seed)
            t = _lookup64(s["vol"], _boxes(c)[b], x)
        fb, los, g = _grads64(P, x, t, r, c, up=s["up"][i:j] if "up" in s else None, density=bool(c.get("density")),
                              through_g=bool(c.get("through_g")))
        losses.append(los)
        f.append(fb)
        for k in parts:
            v = g[k].reshape(-1)
            parts[k].append(torch.cat([v, v.new_zeros(-len(v) % 64)]))   # every tensor fills whole 64s
    grads = {k: torch.cat(v) for k, v in parts.items()}
    if op == "autograd":
        return {"f": torch.cat(f), "grads": grads}
    out = {"losses": torch.stack(losses), "grads": grads}
    if op == "train_step":
        out |= _adam64(c, s["p"], grads)
    return out


def _adam64(c, p, grads):
    """The first Adam step of fresh moments; BF16 gradients have no value to hold their squares to."""
    new, ms, vs = {}, [], []
    for k, g in grads.items():
        if k == "G" and not c["density"]:
            g = torch.zeros_like(g)
        flat = p[k].double().reshape(c["bricks"], -1)
        flat = torch.nn.functional.pad(flat, (0, -flat.shape[1] % 64)).reshape(-1)
        new[k] = flat - LATE_LR * g / (g.abs() + ADAM["eps"])
        ms.append((1 - ADAM["beta1"]) * g)
        vs.append((1 - ADAM["beta2"]) * g * g)
    return {"params": new, "m": torch.cat(ms), "v": torch.cat(vs) if c["prec"] == "fp32" else None}
