"""The workloads whose speed counts: what a user of the package has it do, through its public entry
points (paper_2212_08058_gb300.sfseg), over the range of sizes, radii, types and directions that it
serves.

    listed()             the named workloads
    draw(rng)            one more workload from the ranges that the named ones stand for
    prepare(case, seed)  the inputs and handles a program holds before the call
    run(state)           one pass, and its outputs
    work(case)           the bytes and operations that a pass cannot do without
    exact(case, seed)    the same outputs in 64-bit arithmetic, from plain torch

Shapes are T x H x W; a voxel-iteration of Eq. 7 filters three signals with 2r + 1 taps along each
axis and cannot do without reading the iterate and f and writing the iterate.
"""
import math

import torch

from paper_2212_08058_gb300 import sfseg

ALPHA, P = 1.0, 0.1                      # the package's defaults (Sec. 5.1.1)
CHECK_VOXELS = 1 << 28                   # exact() gives up above this many voxel-passes of a network


# ------------------------------------------------------------------------------------ workloads
def _iterate(T, H, W, radius, iters, C=1, dtype="float32", iters_bf16=0, init="uniform", residual=False):
    return {"kind": "iterate", "T": T, "H": H, "W": W, "rt": radius[0], "rh": radius[1], "rw": radius[2],
            "iters": iters, "C": C, "dtype": dtype, "iters_bf16": iters_bf16, "init": init, "residual": residual}


def listed():
    r133, r277 = (1, 3, 3), (2, 7, 7)
    return [
        # The smallest call: one short clip of a few frames, the 3 x 7 x 7 neighbourhood; latency and
        # launches count.
        dict(_iterate(8, 64, 64, r133, 20), name="iterate 8x64x64"),
        # The plain method on one 480p clip, with the Eq. 3 check that ends it.
        dict(_iterate(64, 480, 854, r277, 50, residual=True), name="solve 480p"),
        # SFSeg++ on the same clip: eight soft-mask channels in bf16, bf16 storage of the iterate with
        # the last iterations in float32.
        dict(_iterate(64, 480, 854, r277, 50, C=8, dtype="bfloat16", iters_bf16=40, init="smap"),
             name="solve 480p c8 bf16"),
        # The largest clip, a chunk of the iterations between two residual checks.
        dict(_iterate(120, 1080, 1920, r277, 10, C=8, dtype="bfloat16"), name="iterate 1080p c8"),
        # A neighbourhood of the user's own choice on a half-size clip.
        dict(_iterate(32, 240, 427, (1, 6, 6), 20), name="iterate radius 1,6,6"),
        # Learning the channel weights: 30 recorded iterations, the soft-IoU loss, the reverse pass.
        {"name": "learn 240x427", "kind": "learn", "T": 32, "H": 240, "W": 427, "rt": 1, "rh": 3, "rw": 3,
         "iters": 30, "every": 5, "C": 8},
        # Alg. 1 end to end on a clip of ordinary length: continuous iterations, then soft-binarisation.
        {"name": "segment 480p", "kind": "segment", "T": 50, "H": 480, "W": 854, "rt": 2, "rh": 7, "rw": 7,
         "iters": 60, "cont": 50, "C": 3},
        # The online form: one pushed frame, ten iterations on the window of 13 frames.
        {"name": "online 480p", "kind": "online", "T": 13, "H": 480, "W": 854, "rt": 2, "rh": 7, "rw": 7,
         "iters": 10, "C": 1},
        # The exact (Eq. 1) operator, the diagnostic of the first-order expansion.
        {"name": "exact 240x427", "kind": "exact", "T": 32, "H": 240, "W": 427, "rt": 2, "rh": 7, "rw": 7,
         "iters": 5, "C": 1},
        # One hidden layer of the warm-start network, forward and backward.
        {"name": "net layer", "kind": "layer", "T": 32, "H": 256, "W": 512, "layer": 1},
        # One training step of the network on a training volume.
        {"name": "net train", "kind": "train", "T": 16, "H": 128, "W": 128, "C": 8},
        # The network's start vector for 1080p frames.
        {"name": "net forward 1080p", "kind": "forward", "T": 24, "H": 1080, "W": 1920, "C": 8},
    ]


RADII = [(1, 3, 3), (2, 7, 7), (1, 3, 3), (2, 7, 7), (1, 2, 2), (1, 4, 4), (2, 5, 5), (1, 7, 7), (2, 3, 3), (1, 5, 5),
         (1, 1, 1), (0, 1, 1), (1, 6, 6), (2, 4, 4), (2, 2, 5), (3, 5, 5), (1, 8, 8), (4, 3, 2)]
OWN_RADII = RADII[:10]                   # those the exact operator takes


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _volume(rng, most, lo=2, hi_h=1080, hi_w=1920):
    while True:
        T, H, W = _log(rng, lo, 120), _log(rng, 48, hi_h), _log(rng, 48, hi_w)
        if T * H * W <= most:
            return T, H, W


def draw(rng):
    kind = rng.choice(["iterate"] * 5 + ["learn"] * 2 + ["segment", "online", "exact", "layer", "train", "forward"])
    if kind == "iterate":
        T, H, W = _volume(rng, 30_000_000)
        iters = _log(rng, 5, 50)
        C = rng.choice([1, 1, 2, 3, 8])
        lowp = rng.random() < 0.25
        return _iterate(T, H, W, rng.choice(RADII), iters, C, rng.choice(["float32", "float32", "bfloat16"]),
                        max(iters - 4, 0) if lowp else 0, rng.choice(["uniform", "smap"]), rng.random() < 0.3)
    if kind == "learn":
        T, H, W = _volume(rng, 4_000_000)
        r = rng.choice(RADII[:10] + [(1, 6, 6), (1, 1, 1)])
        return {"kind": kind, "T": T, "H": H, "W": W, "rt": r[0], "rh": r[1], "rw": r[2], "iters": _log(rng, 6, 30),
                "every": rng.choice([1, 3, 5, 10]), "C": rng.choice([2, 3, 5, 8])}
    if kind == "segment":
        T, H, W = _volume(rng, 20_000_000)
        r = rng.choice(RADII)
        cont = _log(rng, 5, 50)
        return {"kind": kind, "T": T, "H": H, "W": W, "rt": r[0], "rh": r[1], "rw": r[2],
                "iters": cont + rng.randint(1, 10), "cont": cont, "C": rng.choice([1, 3, 8])}
    if kind == "online":
        r = rng.choice(RADII[:10])
        return {"kind": kind, "T": rng.randint(3, 25), "H": _log(rng, 48, 720), "W": _log(rng, 48, 1280), "rt": r[0],
                "rh": r[1], "rw": r[2], "iters": rng.randint(2, 20), "C": rng.choice([1, 3])}
    if kind == "exact":
        T, H, W = _volume(rng, 4_000_000)
        r = rng.choice(OWN_RADII)
        return {"kind": kind, "T": T, "H": H, "W": W, "rt": r[0], "rh": r[1], "rw": r[2], "iters": rng.randint(1, 5),
                "C": rng.choice([1, 3])}
    if kind == "train":
        T, H, W = _volume(rng, 600_000, 4, 200, 300)
        return {"kind": kind, "T": T, "H": H, "W": W, "C": rng.choice([3, 8])}
    T, H, W = _volume(rng, 5_000_000, 3)
    if kind == "layer":
        return {"kind": kind, "T": T, "H": H, "W": W, "layer": rng.choice([1, 2])}
    return {"kind": kind, "T": T, "H": H, "W": W, "C": rng.choice([3, 8])}


# --------------------------------------------------------------------------------------- inputs
def _radius(case):
    return (case["rt"], case["rh"], case["rw"])


def _scene(T, H, W, g):
    """A soft mask [T, H, W]: three blobs of amplitude 0.9 / 0.6 / 0.4 on straight lines, the
    brightest in front."""
    dev = "cuda"
    hh = torch.arange(H, device=dev, dtype=torch.float32)[:, None]
    ww = torch.arange(W, device=dev, dtype=torch.float32)[None, :]
    tt = torch.linspace(0.0, 1.0, T, device=dev)[:, None, None]
    m = torch.zeros((T, H, W), device=dev)
    for amp in (0.4, 0.6, 0.9):
        a, b, c, d, s = torch.rand(5, generator=g, device=dev).tolist()
        sg = (0.06 + 0.08 * s) * H + 2.0
        y = (a + (b - a) * tt) * (H - 1)
        x = (c + (d - c) * tt) * (W - 1)
        blob = ((hh - y).square_() + (ww - x).square_()).mul_(-0.5 / (sg * sg)).exp_().mul_(amp)
        m = torch.where(blob > 0.5 * amp, blob, torch.maximum(m, blob))
    return m


def _features(C, T, H, W, seed, dtype):
    """[C, T, H, W] soft masks in [0, 1] of one scene and the Eq. 9 weights (None for one channel).
    One channel: the mask plus U(0, 0.15).  Several: each channel is another method's estimate, the
    mask moved by up to 4 pixels plus N(0, s^2), s from 0.05 to 0.3, a tenth of its frames lost."""
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    m = _scene(T, H, W, g)
    if C == 1:
        V = m.add_(torch.rand(m.shape, generator=g, device="cuda").mul_(0.15)).clamp_(0.0, 1.0)
        return V[None].to(dtype), None, None
    V = torch.empty((C, T, H, W), device="cuda", dtype=dtype)
    moves = torch.randint(-4, 5, (C, 2), generator=g, device="cuda").tolist()
    for c in range(C):
        s = 0.05 + 0.25 * c / (C - 1)
        n = torch.randn(m.shape, generator=g, device="cuda").mul_(s)
        n.add_(torch.roll(m, (moves[c][0], moves[c][1]), (1, 2))).clamp_(0.0, 1.0)
        n[torch.randperm(T, generator=g, device="cuda")[: int(round(0.1 * T))]] = 0.0
        V[c] = n
    w = -torch.log(torch.rand(C, generator=g, device="cuda"))       # a Dirichlet(1) draw
    w = (w / w.sum()).float().cpu().numpy()
    return V, w, m


def _net_weights(net, seed):
    """The network's own start weights with small biases, as a network in training has."""
    p = net.get_params()
    g = torch.Generator()
    g.manual_seed(seed)
    for _, b in net.unflatten(p):
        b[:] = (0.1 * torch.rand(b.shape, generator=g)).numpy()
    net.set_params(p)
    return p


def _layer_inputs(case, seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    shape = (case["T"], case["H"], case["W"], 32)
    x = torch.randn(shape, generator=g, device="cuda").clamp_(min=0.0).to(torch.bfloat16)     # a ReLU's output
    dz = torch.randn(shape, generator=g, device="cuda").mul_(1e-2).to(torch.bfloat16)
    return x, dz


def prepare(case, seed):
    kind = case["kind"]
    s = {"case": case}
    if kind == "layer":
        s["net"] = sfseg.WarmStartNet(9, seed=seed)
        _net_weights(s["net"], seed)
        s["x"], s["dz"] = _layer_inputs(case, seed)
        return s
    C, T, H, W = case["C"], case["T"], case["H"], case["W"]
    dtype = torch.bfloat16 if kind in ("train", "forward") else getattr(torch, case.get("dtype", "float32"))
    s["V"], s["w"], mask = _features(C, T, H, W, seed, dtype)
    if kind in ("train", "forward"):
        g = torch.Generator(device="cuda")
        g.manual_seed(seed + 1)
        if mask is None:
            mask = s["V"][0].float()
        mask = mask / mask.max()
        s["net"] = sfseg.WarmStartNet(C + 1, seed=seed)
        _net_weights(s["net"], seed)
        s["coarse"] = (mask + 0.05 * torch.rand(mask.shape, generator=g, device="cuda")).contiguous()
        s["target"] = mask.contiguous()
        return s
    if kind == "online":
        s["h"] = sfseg.OnlineStream(C, T, H, W, alpha=ALPHA, p=P)
        s["frames"] = [s["V"][:, t].contiguous() for t in range(T)]
        for f in s["frames"][:-1]:
            s["h"].push(f, s["w"], 0.0, radius=_radius(case), iters=case["iters"])
        return s
    s["h"] = sfseg.PowerIteration(C, T, H, W, alpha=ALPHA, p=P)
    if kind == "learn":
        s["mask"] = mask
    return s


# ----------------------------------------------------------------------------------------- pass
def run(s):
    case = s["case"]
    kind = case["kind"]
    if kind == "layer":
        y = s["net"].layer_forward(case["layer"], s["x"])
        dx, dW, db = s["net"].layer_backward(case["layer"], s["x"], s["dz"])
        return {"y": y, "dx": dx, "dW": dW, "db": db}
    if kind == "train":
        loss, grads = s["net"].backward(s["V"], s["target"], want_grads=True, extra=s["coarse"])
        s["net"].adamw(lr=1e-3, weight_decay=1e-4)
        return {"loss": loss, "grads": grads}
    if kind == "forward":
        return s["net"].forward(s["V"], s["coarse"])
    r, h = _radius(case), s["h"]
    if kind == "online":
        return h.push(s["frames"][-1], s["w"], 0.0, radius=r, iters=case["iters"])
    if kind == "exact":
        h.set_features(s["V"], s["w"], 0.0)
        return h.power_iterate_exact(r, iters=case["iters"])
    if kind == "segment":
        # The hard mask beside it is this output compared with 1/2: a voxel within a rounding of 1/2
        # has no value of its own to be compared with, so the soft segmentation stands for both.
        return h.segment(s["V"], s["w"], 0.0, radius=r, n_iter=case["iters"], n_cont=case["cont"])[0]
    if kind == "learn":
        x = h.power_iterate(s["V"], s["w"], 0.0, r, iters=case["iters"], record_every=case["every"])
        loss, g = h.soft_iou_loss(x, s["mask"])
        gw, gb = h.backward(g, r)
        return {"x": x, "loss": loss, "gw": gw, "gb": gb}
    x = h.power_iterate(s["V"], s["w"], 0.0, radius=r, iters=case["iters"], iters_bf16=case["iters_bf16"],
                        init=case["init"])
    if case["residual"]:
        rho, res = h.rayleigh(x, r)
        return {"x": x, "rho": rho, "residual": res}
    return x


def work(case):
    kind = case["kind"]
    N = case["T"] * case["H"] * case["W"]
    if kind == "layer":                  # forward, data gradient and weight gradient of 32 -> 32 channels
        return {"bytes": N * 32 * 2 * 4 + 2 * 27 * 1024 * 4, "flops": 3 * 2 * 27 * 32 * 32 * N}
    if kind in ("train", "forward"):
        c = case["C"] + 1
        taps = 27 * (32 * c + 2 * 32 * 32 + 32)
        if kind == "forward":            # channels and coarse start in, start vector out
            return {"bytes": N * (2 * case["C"] + 4 + 4), "flops": 2 * taps * N}
        return {"bytes": N * (2 * case["C"] + 4 + 4) + 4 * 4 * taps, "flops": (3 * 2 * taps - 2 * 27 * 32 * c) * N}
    C, it = case["C"], case["iters"]
    fma = 3 * sum(2 * r + 1 for r in _radius(case))
    el = 2 if case.get("dtype") == "bfloat16" else 4
    if kind == "online":
        return {"bytes": N // case["T"] * (4 * C + 4) + 12 * N * it, "flops": 2 * fma * N * it}
    if kind == "exact":
        # per step and pair of neighbours, whatever the method: read x and f, write x; the three
        # filtered signals of one separable term group
        return {"bytes": N * (4 * C + 12 * it), "flops": 2 * fma * N * it}
    if kind == "learn":
        # per step: the forward, and the filtering of x and of the gradient on the way back
        return {"bytes": N * (4 * C * 2 + 12 * it + 36 * it), "flops": 2 * fma * N * it * 3}
    if kind == "segment":
        return {"bytes": N * (4 * C + 12 * it), "flops": 2 * fma * N * it}
    b = case["iters_bf16"]
    extra = 1 if case["residual"] else 0
    return {"bytes": N * (el * C + 4 + 6 * b + 12 * (it - b + extra)), "flops": 2 * fma * N * (it + extra)}


# ------------------------------------------------------------------------------ 64-bit reference
def _taps(radius):
    s = max(radius) / 2.0 or 1.0         # the package's default width
    return [[math.exp(-d * d / (2.0 * s * s)) for d in range(r + 1)] for r in radius]


def _filter(z, taps):
    """The separable Gaussian of the last three axes, zero outside the volume."""
    for axis, g in enumerate(taps):
        y = z * g[0]
        n = z.shape[axis]
        for d in range(1, min(len(g), n)):
            y.narrow(axis, d, n - d).add_(z.narrow(axis, 0, n - d), alpha=g[d])
            y.narrow(axis, 0, n - d).add_(z.narrow(axis, d, n - d), alpha=g[d])
        z = y
    return z


class _Filter(torch.autograd.Function):
    """_filter, its own transpose."""

    @staticmethod
    def forward(ctx, z, radius):
        ctx.radius = radius
        return _filter(z, _taps(radius))

    @staticmethod
    def backward(ctx, g):
        return _filter(g, _taps(ctx.radius)), None


def _combine(V, w):
    if w is None:
        return V[0].double()
    z = torch.zeros(V.shape[1:], device=V.device, dtype=torch.float64)
    for c in range(V.shape[0]):
        z.add_(V[c].double(), alpha=float(w[c]))
    return torch.sigmoid_(z)


def _apply(f, u, x, radius):
    """A x of Eq. 7: u [(1/alpha - f^2) G(ux) - G(f^2 ux) + 2 f G(f ux)]."""
    t = _taps(radius)
    v = u * x
    y = _filter(v, t).mul_(1.0 / ALPHA - f * f)
    v = v.mul_(f)
    y.add_(_filter(v, t).mul_(f), alpha=2.0)
    y.sub_(_filter(v.mul_(f), t))
    return y.mul_(u)


def _power(f, u, x, radius, iters):
    x = x / x.norm()
    for _ in range(iters):
        x = _apply(f, u, x, radius)
        x.div_(x.norm())
    return x


def _unary(f):
    return f.pow(P)


def _apply_exact(f, u, x, radius):
    """(1/alpha) M x with M_ij = u_i u_j exp(-alpha (f_i - f_j)^2) G_ij, neighbour by neighbour."""
    t = _taps(radius)
    v = u * x
    y = torch.zeros_like(v)
    T, H, W = v.shape
    for a in range(-radius[0], radius[0] + 1):
        for b in range(-radius[1], radius[1] + 1):
            for c in range(-radius[2], radius[2] + 1):
                if abs(a) >= T or abs(b) >= H or abs(c) >= W:
                    continue
                i = tuple(slice(max(0, -d), n - max(0, d)) for d, n in ((a, T), (b, H), (c, W)))
                j = tuple(slice(max(0, d), n - max(0, -d)) for d, n in ((a, T), (b, H), (c, W)))
                k = (f[i] - f[j]).square_().mul_(-ALPHA).exp_().mul_(v[j])
                y[i].add_(k, alpha=t[0][abs(a)] * t[1][abs(b)] * t[2][abs(c)])
    return y.mul_(u).mul_(1.0 / ALPHA)


def _shift(x, tap):
    """x[v + tap offset] of a channels-last [T, H, W, C] volume, zero outside; tap = 9 dt + 3 dh + dw."""
    p = torch.nn.functional.pad(x, (0, 0, 1, 1, 1, 1, 1, 1))
    T, H, W, _ = x.shape
    a, b, c = tap // 9, tap // 3 % 3, tap % 3
    return p[a:a + T, b:b + H, c:c + W].reshape(T * H * W, -1)


def _conv(x, w, b):
    """The 3x3x3 cross-correlation, w [out, 27, in]."""
    y = 0.0 if b is None else b
    for tap in range(27):
        y = y + _shift(x, tap) @ w[:, tap].T
    return y.reshape(*x.shape[:3], -1)


def _conv_grads(x, dz, w):
    """(gradient at the input, at the weights [out, 27, in], at the bias)."""
    d2 = dz.reshape(-1, dz.shape[-1])
    dw = torch.stack([d2.T @ _shift(x, tap) for tap in range(27)], 1)
    dx = _conv(dz, w.flip(1).permute(2, 1, 0), None)
    return dx, dw, d2.sum(0)


def _net64(net_params, c_in):
    """[(w [out, 27, in], b)] in 64 bits, the weights as the bf16 copies that the layers multiply."""
    out, o = [], 0
    p = torch.from_numpy(net_params).cuda()
    for co, ci in ((32, c_in), (32, 32), (32, 32), (1, 32)):
        w = p[o:o + co * 27 * ci].to(torch.bfloat16).double().reshape(co, 27, ci)
        o += co * 27 * ci
        out.append((w, p[o:o + co].double()))
        o += co
    return out


def exact(case, seed):
    kind = case["kind"]
    N = case["T"] * case["H"] * case["W"]
    if kind == "layer":
        net = sfseg.WarmStartNet(9, seed=seed)
        layers = _net64(_net_weights(net, seed), 9)
        net.close()
        x, dz = (t.double() for t in _layer_inputs(case, seed))
        w, b = layers[case["layer"]]
        dx, dw, db = _conv_grads(x, dz, w)
        return {"y": _conv(x, w, b).relu_(), "dx": dx * (x > 0), "dW": dw.reshape(32, 3, 3, 3, 32), "db": db}
    if kind in ("train", "forward"):
        if N * 27 > CHECK_VOXELS:
            return None                  # over a minute in 64 bits
        s = prepare(case, seed)
        layers = _net64(_net_weights(s["net"], seed), case["C"] + 1)
        s["net"].close()
        x = torch.cat([s["V"].double(), s["coarse"].to(torch.bfloat16).double()[None]]).permute(1, 2, 3, 0)
        acts = [x.contiguous()]
        for w, b in layers[:3]:
            acts.append(_conv(acts[-1], w, b).relu_())
        z = _conv(acts[-1], *layers[3])
        x0 = torch.nn.functional.softplus(z, threshold=40.0)
        if kind == "forward":
            return x0[..., 0]
        t = s["target"].double()[..., None]
        nx, nt, xt = x0.norm(), t.norm(), (x0 * t).sum()
        loss = 1.0 - xt / (nx * nt)
        d = -(t / (nx * nt) - x0 * (xt / (nx * nt) / (nx * nx))) * torch.sigmoid(z)
        grads = []
        for k in (3, 2, 1, 0):
            dx, dw, db = _conv_grads(acts[k], d, layers[k][0])
            grads = [dw.reshape(-1), db] + grads
            d = dx * (acts[k] > 0)
        return {"loss": float(loss), "grads": torch.cat(grads)}
    C, T, H, W, r = case["C"], case["T"], case["H"], case["W"], _radius(case)
    V, w, mask = _features(C, T, H, W, seed, getattr(torch, case.get("dtype", "float32")))
    f = _combine(V, w)
    u = _unary(f)
    ones = torch.ones_like(f)
    if kind == "online":
        fw, x = torch.zeros_like(f), torch.zeros_like(f)
        for t in range(T):
            fw = torch.cat([fw[1:], f[t:t + 1]])
            x = torch.cat([x[1:], x[-1:] if t else ones[:1]])
            x = _power(fw, _unary(fw), x, r, case["iters"])
        return x[-1]
    if kind == "exact":
        x = ones / ones.norm()
        for _ in range(case["iters"]):
            x = _apply_exact(f, u, x, r)
            x.div_(x.norm())
        return x
    if kind == "segment":
        x = _power(f, u, ones, r, case["cont"])
        for _ in range(case["iters"] - case["cont"]):
            y = _apply(f, u, x, r)
            x = torch.sigmoid_(y.div_(y.max()).sub_(0.5).mul_(10.0))
        return x
    if kind == "learn":
        wt = torch.tensor(w, device="cuda", dtype=torch.float64, requires_grad=True)
        b = torch.zeros((), device="cuda", dtype=torch.float64, requires_grad=True)
        f = torch.sigmoid(sum(wt[c] * V[c].double() for c in range(C)) + b)
        u = f.pow(P)
        x = ones / ones.norm()
        for _ in range(case["iters"]):
            v = u * x
            z = f * v
            y = u * ((1.0 / ALPHA - f * f) * _Filter.apply(v, r) - _Filter.apply(f * z, r) + 2.0 * f * _Filter.apply(z, r))
            x = y / y.norm()
        m = mask.double()
        xh = x / x.max()
        loss = 1.0 - (xh * m).sum() / (xh + m - xh * m).sum()
        gw, gb = torch.autograd.grad(loss, (wt, b))
        return {"x": x.detach(), "loss": float(loss.detach()), "gw": gw, "gb": float(gb)}
    x = _power(f, u, f if case["init"] == "smap" else ones, r, case["iters"])
    if case["residual"]:
        y = _apply(f, u, x, r)
        rho = float((x * y).sum() / (x * x).sum())
        return {"x": x, "rho": rho, "residual": float((y - rho * x).norm() / x.norm()) / rho}
    return x
