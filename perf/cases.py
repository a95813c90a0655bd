"""Performance cases of the registration library: the calls its users make, over the sizes,
dimensions, similarities, spacings and layers they make them with.

Every case goes through the package's public entry points (`airgb`, `registration`). Volumes are
(Z, Y, X) or (Y, X), x fastest, as the package takes them; a case holds its sizes as nz, ny, nx
(nz = 1 in 2D). `exact` evaluates the method's definitions in 64 bits with plain torch.
"""
import math

import torch
import torch.nn.functional as tnf

from paper_1806_09907_gb300 import airgb, registration

LAMBDA = 0.1
EPS = 1e-5
LR, BETA1, BETA2, ADAM_EPS = 0.01, 0.9, 0.999, 1e-8
STEP0 = 20  # Adam steps taken before the measured one: the middle of an optimisation

# (cin, cout, stride) of the initialisation network's layers
LAYERS = ((2, 16, 2), (16, 32, 2), (32, 48, 2), (48, 64, 2), (112, 48, 1), (48, 48, 1), (48, 16, 1))


def _case(kind, name=None, **kw):
    d = {"kind": kind, **kw}
    if name is not None:
        d["name"] = name
    return d


def listed():
    return [
        # One evaluation of J and its gradient of a 2D image pair, called from Python as an
        # optimiser of the user's own calls it: the smallest call, where launches count.
        _case("objective", "objective_2d_mse_128", nz=1, ny=128, nx=128, spacing=8, sim="mse",
              window=7, scene="blobs", sigma=2.0),
        # One graph-replayed iteration (objective through autograd, Adam step) on 128^3, the
        # plain optimiser's inner loop.
        _case("iteration", "iteration_3d_mse_128", nz=128, ny=128, nx=128, spacing=8, sim="mse",
              window=7, scene="blobs", sigma=1.0),
        # The evaluation of a ragged volume at a control spacing without a fused kernel, with the
        # global correlation: the library composes its step kernels.
        _case("objective", "objective_3d_ncc_odd", nz=97, ny=141, nx=173, spacing=5, sim="ncc",
              window=7, scene="ct", sigma=2.0),
        # The evaluation a CT-sized registration spends its time in: local correlation over 7^3.
        _case("objective", "objective_ct_lcc", nz=160, ny=256, nx=256, spacing=6, sim="lcc",
              window=7, scene="ct", sigma=3.0),
        # One iteration on the middle level of the same registration's pyramid.
        _case("iteration", "iteration_half_ct_lcc", nz=80, ny=128, nx=128, spacing=6, sim="lcc",
              window=7, scene="ct", sigma=1.5),
        # The diffeomorphic model on the same CT volume: six squarings forward and adjoint.
        _case("diffeo", "diffeo_ct_lcc", nz=160, ny=256, nx=256, spacing=6, sim="lcc", window=7,
              scene="ct", sigma=2.0, steps=6),
        # One iteration of many pairs of uneven sizes, 2D and 3D together, in one launch.
        _case("batch", "batch_16_uneven", n2d=8, n3d=8, lo2=96, hi2=512, lo3=64, hi3=192,
              spacing=8),
        # The network's first layer in a training step: two input channels at full resolution.
        _case("conv", "conv_2_16_train", layer=0, batch=16, nz=128, ny=128, nx=128, train=True),
        # Its second layer, forward and both adjoints: the largest activations with a gradient.
        _case("conv", "conv_16_32_train", layer=1, batch=16, nz=64, ny=64, nx=64, train=True),
        # The decoder's widest layer for a single pair: inference, few output tiles.
        _case("conv", "conv_112_48_infer", layer=4, batch=1, nz=16, ny=16, nx=16, train=False),
        # Training pairs rendered and warped into the network's input.
        _case("pairs", "pairs_16_128", batch=16, nz=128, ny=128, nx=128, blobs=60),
        # What happens between two pyramid levels: both images' next level and the refinement
        # of the coefficients onto it.
        _case("level", "level_half_ct", nz=160, ny=256, nx=256, spacing=6, factor=2),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _volume(rng, most, lo=24, hi=256):
    while True:
        n = [_log_int(rng, lo, hi) for _ in range(3)]
        if n[0] * n[1] * n[2] <= most:
            return dict(nz=n[0], ny=n[1], nx=n[2])


def draw(rng):
    kind = rng.choice(["objective", "objective", "iteration", "diffeo", "batch", "conv", "conv",
                       "pairs", "level"])
    sim = rng.choice(["mse", "ncc", "lcc"])
    window = rng.choice([3, 5, 7, 7])
    spacing = rng.choice([4, 6, 8, 8, 3, 5, 10])
    scene = rng.choice(["blobs", "ct"])
    sigma = round(rng.uniform(0.5, 3.0), 2)
    if kind in ("objective", "iteration"):
        if rng.random() < 0.35:
            size = dict(nz=1, ny=_log_int(rng, 64, 1024), nx=_log_int(rng, 64, 1024))
        else:
            size = _volume(rng, 10_000_000)
        return _case(kind, **size, spacing=spacing, sim=sim, window=window, scene=scene,
                     sigma=sigma)
    if kind == "diffeo":
        return _case(kind, **_volume(rng, 4_000_000, lo=32), spacing=spacing, sim=sim,
                     window=window, scene=scene, sigma=sigma, steps=rng.randint(4, 7))
    if kind == "batch":
        return _case(kind, n2d=rng.randint(1, 8), n3d=rng.randint(1, 8),
                     lo2=rng.randint(64, 128), hi2=rng.randint(200, 512),
                     lo3=rng.randint(32, 72), hi3=rng.randint(80, 192),
                     spacing=rng.choice([4, 6, 8]))
    if kind == "conv":
        layer = rng.randrange(len(LAYERS))
        train = rng.random() < 0.6
        top = (128, 64, 32, 16, 16, 16, 16)[layer]
        n = [_log_int(rng, max(4, top // 3), top) for _ in range(3)]
        return _case(kind, layer=layer, batch=rng.randint(2, 16) if train else 1, nz=n[0],
                     ny=n[1], nx=n[2], train=train)
    if kind == "pairs":
        n = [4 * rng.randint(12, 32) for _ in range(3)]
        return _case(kind, batch=rng.randint(1, 16), nz=n[0], ny=n[1], nx=n[2],
                     blobs=rng.randint(20, 60))
    return _case("level", **_volume(rng, 10_000_000, lo=32), spacing=spacing,
                 factor=rng.choice([2, 4]))


# ------------------------------------------------------------------ inputs --

def _shape(case):
    return (case["ny"], case["nx"]) if case["nz"] == 1 else (case["nz"], case["ny"], case["nx"])


def _lattice(shape, spacing):
    return (len(shape),) + tuple((n - 1) // spacing + 4 for n in shape)


def _gen(seed, stream=0):
    return torch.Generator(device="cuda").manual_seed(int(seed) * 64 + stream)


def _uniform(g, n, lo, hi):
    return torch.rand(n, generator=g, device="cuda", dtype=torch.float64) * (hi - lo) + lo


def _points(shape):
    """Voxel coordinates, x first, broadcastable, fp32."""
    d = len(shape)
    return [torch.arange(n, device="cuda", dtype=torch.float32).view(
        [n if a == k else 1 for a in range(d)]) for k, n in reversed(list(enumerate(shape)))]


def _smooth_field(shape, rms, g):
    """Displacement of `rms` voxels made of a few cosine waves of at least 32 voxels."""
    d, xs, out = len(shape), _points(shape), []
    for _ in range(d):
        acc = torch.zeros(shape, device="cuda")
        par = _uniform(g, (4, d + 3), -1.0, 1.0).cpu().tolist()
        for p in par:
            norm = math.sqrt(sum(v * v for v in p[:d])) + 1e-9
            wl = 32.0 + (p[d] + 1.0) * max(shape)
            arg = math.pi * p[d + 1]
            for k in range(d):
                arg = arg + (2.0 * math.pi / wl * p[k] / norm) * xs[k]
            acc += p[d + 2] * torch.cos(arg)
        out.append(acc * (rms / float(acc.square().mean().sqrt().clamp_min(1e-6))))
    return out


def _blob_image(shape, pos, table):
    img = torch.zeros(shape, device="cuda")
    for row in table:
        r2 = sum((pos[k] - row[k]) ** 2 for k in range(len(shape)))
        img += row[-1] * torch.exp(-r2 / (2.0 * row[-2] * row[-2]))
    return img


def _ct_image(shape, pos, items):
    img = torch.full(shape, -1000.0, device="cuda")
    for c, ax, hu in items:
        q = sum(((pos[k] - c[k]) / ax[k]) ** 2 for k in range(len(shape)))
        img = torch.where(q <= 1.0, hu, img)
    return img


def _pair(shape, scene, seed):
    """Fixed and moving image: Gaussian blobs, or ellipsoids in HU with noise, and the same scene
    seen through a smooth displacement of 2 or 3 voxels."""
    g, d = _gen(seed, 1), len(shape)
    ext = [n - 1.0 for n in reversed(shape)]
    xs = [x.expand(shape) for x in _points(shape)]
    field = _smooth_field(shape, 2.0 if scene == "blobs" else 3.0, g)
    moved = [x + u for x, u in zip(xs, field)]
    if scene == "blobs":
        n, lo, hi = (20, 4.0, 16.0) if d == 2 else (60, 3.0, 12.0)
        u = _uniform(g, (n, d + 2), 0.0, 1.0).cpu().tolist()
        table = [[r[k] * ext[k] for k in range(d)] + [lo + (hi - lo) * r[d], r[d + 1]] for r in u]
        return _blob_image(shape, xs, table), _blob_image(shape, moved, table)
    u = _uniform(g, (31, 2 * d + 1), 0.0, 1.0).cpu().tolist()
    items = [([0.5 * e for e in ext], [0.44 * e + 1.0 for e in ext], 40.0 * u[0][-1])]
    for r in u[1:]:
        items.append(([(0.2 + 0.6 * r[k]) * ext[k] for k in range(d)],
                      [(0.02 + 0.14 * r[d + k]) * min(ext) + 1.0 for k in range(d)],
                      2500.0 * r[-1] - 1000.0))
    noise = [20.0 * torch.randn(shape, generator=g, device="cuda") for _ in range(2)]
    return _ct_image(shape, xs, items) + noise[0], _ct_image(shape, moved, items) + noise[1]


def _moments(shape, lattice, sim, scene, seed):
    """Adam's moments in the middle of a run (normalised units): a running gradient and its
    square, of the size the first iterations of such a pair have."""
    g = _gen(seed, 2)
    size = 3e-2 if sim == "lcc" or scene == "ct" else 1e-2
    size *= 64.0 / math.prod(lattice[1:]) ** 0.5
    m = size * torch.randn(lattice, generator=g, device="cuda")
    v = size * size * (0.5 + torch.rand(lattice, generator=g, device="cuda"))
    return m, v * (1.0 - BETA2 ** STEP0)


def _objective_inputs(case, seed):
    shape = _shape(case)
    F, M = _pair(shape, case["scene"], seed)
    lat = _lattice(shape, case["spacing"])
    c = case["sigma"] * torch.randn(lat, generator=_gen(seed, 3), device="cuda")
    m, v = _moments(shape, lat, case["sim"], case["scene"], seed)
    return shape, F, M, c, m, v


def _batch_shapes(case):
    def between(lo, hi, n):
        return [round(lo + (hi - lo) * (k / max(n - 1, 1))) for k in range(n)]
    return [(n, n) for n in between(case["lo2"], case["hi2"], case["n2d"])] + \
        [(n, n, n) for n in between(case["lo3"], case["hi3"], case["n3d"])]


def _batch_inputs(case, seed):
    out = []
    for k, shape in enumerate(_batch_shapes(case)):
        sub = dict(nz=shape[0] if len(shape) == 3 else 1, ny=shape[-2], nx=shape[-1],
                   spacing=case["spacing"], sim="mse", scene="blobs", sigma=1.0)
        out.append(_objective_inputs(sub, seed * 64 + k))
    return out


def _conv_inputs(case, seed):
    cin, cout, stride = LAYERS[case["layer"]]
    n = (case["nz"], case["ny"], case["nx"])
    o = tuple((k - 1) // stride + 1 for k in n)
    g = _gen(seed, 4)
    x = torch.randn((case["batch"],) + n + (cin,), generator=g, device="cuda")
    # the first layer reads images in [0, 1], the others the ReLU outputs of the layer before
    x = (x.sigmoid() if cin == 2 else x.relu()).to(torch.bfloat16)
    w = torch.randn((cout, 27, cin), generator=g, device="cuda") * math.sqrt(2.0 / (27 * cin))
    b = 0.1 * torch.randn(cout, generator=g, device="cuda")
    gy = None
    if case["train"]:
        gy = (1e-3 * torch.randn((case["batch"],) + o + (cout,), generator=g, device="cuda"))
        gy = gy.to(torch.bfloat16)
    return x, w, b, gy


def _pairs_inputs(case, seed):
    g, shape, n = _gen(seed, 5), _shape(case), case["batch"]
    scale = torch.tensor([s - 1.0 for s in reversed(shape)] + [9.0, 1.0], device="cuda")
    shift = torch.tensor([0.0, 0.0, 0.0, 3.0, 0.0], device="cuda")
    table = torch.rand((n, case["blobs"], 5), generator=g, device="cuda") * scale + shift
    ctrl = 4.0 * torch.randn((n,) + _lattice(shape, 8), generator=g, device="cuda")
    return shape, table, ctrl


def _level_inputs(case, seed):
    shape = _shape(case)
    F, M = _pair(shape, "ct", seed)
    coarse = tuple((n - 1) // 2 + 1 for n in shape)
    c = 2.0 * torch.randn(_lattice(coarse, case["spacing"]), generator=_gen(seed, 6),
                          device="cuda")
    return shape, coarse, F, M, c


# --------------------------------------------------------------- the calls --

def prepare(case, seed):
    kind = case["kind"]
    if kind == "objective":
        shape, F, M, c, _, _ = _objective_inputs(case, seed)
        ob = airgb.Objective(shape, case["spacing"], case["sim"], LAMBDA, EPS, case["window"])
        return dict(kind=kind, ob=ob, F=F, M=M, c=c)
    if kind == "diffeo":
        shape, F, M, c, _, _ = _objective_inputs(case, seed)
        ev = registration.Evaluator(shape, case["spacing"], case["sim"], LAMBDA, EPS,
                                    case["window"], diffeo_steps=case["steps"])
        return dict(kind=kind, ev=ev, F=F, M=M, c=c, grad=torch.empty_like(c),
                    value=torch.empty(4, dtype=torch.float64, device="cuda"))
    if kind == "iteration":
        shape, F, M, c, m, v = _objective_inputs(case, seed)
        c.requires_grad_(True)
        ev = registration.Evaluator(shape, case["spacing"], case["sim"], LAMBDA, EPS,
                                    case["window"])
        opt = registration.BsplineAdam([c], shape, case["spacing"], lr=LR)
        opt.init_state()
        opt.state[c]["exp_avg"].copy_(m)
        opt.state[c]["exp_avg_sq"].copy_(v)
        opt.state[c]["step"].fill_(STEP0)
        return dict(kind=kind, it=registration.GraphedIteration(c, ev, F, M, opt), ev=ev, c=c,
                    st=opt.state[c], F=F, M=M)
    if kind == "batch":
        ins = _batch_inputs(case, seed)
        b = airgb.Batch([(i[1], i[2]) for i in ins], case["spacing"], LAMBDA, history=1)
        for k, (_, _, _, c, m, v) in enumerate(ins):
            b.ctrl[k].copy_(c)
            b.m[k].copy_(m)
            b.v[k].copy_(v)
        return dict(kind=kind, b=b)
    if kind == "conv":
        x, w, b, gy = _conv_inputs(case, seed)
        cin, cout, stride = LAYERS[case["layer"]]
        cv = airgb.make_conv(case["batch"], tuple(x.shape[1:4]), cin, cout, stride)
        pf, pd = airgb.al_conv3d_pack(cv, w, True, case["train"] and cin % 16 == 0)
        new = lambda n: torch.empty(max(n, 256), dtype=torch.uint8, device="cuda")
        s = dict(kind=kind, cv=cv, x=x, b=b, gy=gy, pf=pf, pd=pd, relu=case["layer"] != 6,
                 fws=new(airgb.conv_forward_workspace_bytes(cv)),
                 y=torch.empty((case["batch"],) + airgb.conv_output_size(cv) + (cout,),
                               dtype=torch.float32 if case["layer"] == 6 else torch.bfloat16,
                               device="cuda"))
        if case["train"]:
            s.update(wws=new(airgb.conv_wgrad_workspace_bytes(cv)), gw=torch.empty_like(w),
                     gb=torch.empty_like(b), gx=torch.empty_like(x) if pd is not None else None)
        return s
    if kind == "pairs":
        shape, table, ctrl = _pairs_inputs(case, seed)
        M = torch.empty((case["batch"],) + shape, device="cuda")
        return dict(kind=kind, shape=shape, table=table, ctrl=ctrl, M=M,
                    x=torch.empty(M.shape + (2,), dtype=torch.bfloat16, device="cuda"))
    shape, coarse, F, M, c = _level_inputs(case, seed)
    return dict(kind=kind, shape=shape, coarse=coarse, F=F, M=M, c=c, factor=case["factor"],
                spacing=case["spacing"])


def run(s):
    kind = s["kind"]
    if kind == "objective":
        value, grad = s["ob"](s["F"], s["M"], s["c"])
        return {"value": value, "grad": grad}
    if kind == "diffeo":
        s["ev"].evaluate(s["F"], s["M"], s["c"], s["value"], s["grad"])
        return {"value": s["value"], "grad": s["grad"]}
    if kind == "iteration":
        s["it"]()
        return {"value": s["ev"].last_value, "grad": s["c"].grad, "ctrl": s["c"],
                "m": s["st"]["exp_avg"], "v": s["st"]["exp_avg_sq"]}
    if kind == "batch":
        b = s["b"]
        b.step(STEP0 + 1, 0, LR)
        return {"ctrl": b.ctrl, "m": b.m, "v": b.v, "values": b.values}
    if kind == "conv":
        out = {"y": airgb.al_conv3d_forward(s["cv"], s["x"], s["pf"], s["b"], relu=s["relu"],
                                            out_f32=s["y"].dtype == torch.float32, out=s["y"],
                                            workspace=s["fws"])}
        if s["gy"] is not None:
            out["gw"], out["gb"] = airgb.al_conv3d_backward_weight(
                s["cv"], s["x"], s["gy"], s["gw"], s["gb"], s["wws"])
            if s["pd"] is not None:
                out["gx"] = airgb.al_conv3d_backward_data(s["cv"], s["gy"], s["pd"],
                                                          relu_input=s["x"], grad_in=s["gx"])
        return out
    if kind == "pairs":
        airgb.al_render_blobs(s["shape"], s["table"], out=s["M"])
        airgb.al_initnet_pair_input(s["shape"], 8, s["M"], s["ctrl"], out=s["x"])
        return {"M": s["M"], "x": s["x"]}
    F = airgb.al_pyramid_level(s["F"], s["factor"])
    M = airgb.al_pyramid_level(s["M"], s["factor"])
    return {"F": F, "M": M, "ctrl": airgb.al_bspline_refine(s["coarse"], s["shape"], s["spacing"],
                                                            s["c"])}


# -------------------------------------------------------------------- work --

def _objective_work(shape, spacing, sim, extra=0.0):
    d, nv, npar = len(shape), math.prod(shape), math.prod(_lattice(shape, spacing))
    per = ({"mse": 150, "ncc": 160, "lcc": 287} if d == 3 else
           {"mse": 60, "ncc": 70, "lcc": 150})[sim]
    return {"bytes": 8.0 * nv + 8.0 * npar, "flops": (per + extra) * nv}


def work(case):
    kind = case["kind"]
    shape = _shape(case) if "nx" in case else None
    if kind == "objective":
        return _objective_work(shape, case["spacing"], case["sim"])
    if kind == "diffeo":
        # per squaring: 3 interpolations, their derivatives and the transposed interpolation
        return _objective_work(shape, case["spacing"], case["sim"], 190.0 * case["steps"])
    if kind == "iteration":
        w = _objective_work(shape, case["spacing"], case["sim"])
        w["bytes"] += 24.0 * math.prod(_lattice(shape, case["spacing"]))
        return w
    if kind == "batch":
        ws = [_objective_work(s, case["spacing"], "mse") for s in _batch_shapes(case)]
        par = sum(math.prod(_lattice(s, case["spacing"])) for s in _batch_shapes(case))
        return {"bytes": sum(w["bytes"] for w in ws) + 24.0 * par,
                "flops": sum(w["flops"] for w in ws)}
    if kind == "conv":
        cin, cout, stride = LAYERS[case["layer"]]
        n = (case["nz"], case["ny"], case["nx"])
        vi = case["batch"] * math.prod(n)
        vo = case["batch"] * math.prod((k - 1) // stride + 1 for k in n)
        size = 4 if case["layer"] == 6 else 2
        macs, wb = 27.0 * cin * cout * vo, 27 * cin * cout
        if not case["train"]:
            return {"bytes": 2.0 * vi * cin + size * vo * cout + 2.0 * wb, "flops": 2.0 * macs}
        dgrad = cin % 16 == 0
        return {"bytes": 2.0 * vi * cin * (2 if dgrad else 1) + (size + 2.0) * vo * cout
                + (4.0 if dgrad else 2.0) * wb + 4.0 * wb,
                "flops": 2.0 * macs * (3 if dgrad else 2)}
    nv = math.prod(shape)
    if kind == "pairs":
        par = math.prod(_lattice(shape, 8))
        return {"bytes": case["batch"] * (8.0 * nv + 4.0 * par + 20.0 * case["blobs"]),
                "flops": case["batch"] * nv * (83.0 + 2.0 * case["blobs"])}
    f = case["factor"]
    small = math.prod((n - 1) // f + 1 for n in shape)
    coarse = tuple((n - 1) // 2 + 1 for n in shape)
    return {"bytes": 8.0 * nv + 8.0 * small + 4.0 * math.prod(_lattice(coarse, case["spacing"]))
            + 4.0 * math.prod(_lattice(shape, case["spacing"])),
            "flops": 2.0 * 2 * (2 * (3 * f // 2) + 1) * nv / f}


# ------------------------------------------------------------------- exact --

def _kernel(r):
    r = r.abs()
    return torch.where(r < 1, 2.0 / 3.0 - r * r + 0.5 * r ** 3,
                       torch.where(r < 2, (2.0 - r) ** 3 / 6.0, torch.zeros_like(r)))


def _displacement64(shape, spacing, c):
    """u = sum_j c_j k(x - (j - 1) spacing), per axis, 64 bits."""
    u = c
    for a, n in enumerate(shape):
        x = torch.arange(n, device="cuda", dtype=torch.float64)
        p = (torch.arange((n - 1) // spacing + 4, device="cuda", dtype=torch.float64) - 1) * spacing
        B = _kernel((x[:, None] - p[None, :]) / spacing)
        u = torch.movedim(torch.tensordot(u, B, dims=([a + 1], [1])), -1, a + 1)
    return u


def _sample64(shape, u):
    """Linear interpolation cells at x + u: per axis (x first) cell, offset, inside."""
    out = []
    d = len(shape)
    for k, x in enumerate(_points(shape)):
        n = shape[d - 1 - k]
        y = x.double() + u[k]
        inside = (y >= 0) & (y <= n - 1)
        y = torch.where(torch.isfinite(y), y, torch.zeros_like(y))
        cell = y.detach().floor().clamp(0, n - 2).long()
        out.append((cell, y, inside, n))
    return out


def _interpolate64(img, shape, axes):
    """The interpolant of img (..., *shape) at the positions of `axes` (cell, y)."""
    d, flat, total = len(shape), img.reshape(img.shape[:-len(shape)] + (-1,)), 0.0
    strides = [1, shape[-1], shape[-1] * shape[-2]][:d]
    for corner in range(2 ** d):
        w, idx = 1.0, 0
        for k, (cell, y, _, _) in enumerate(axes):
            f = y - cell
            hi = (corner >> k) & 1
            w = w * (f if hi else 1.0 - f)
            idx = idx + (cell + hi) * strides[k]
        total = total + w * flat[..., idx]
    return total


def _box64(t, r):
    """Window sums of width 2r + 1 along every axis, zero outside."""
    for a in range(t.dim()):
        pad = [0, 0] * t.dim()
        pad[2 * (t.dim() - 1 - a)] = pad[2 * (t.dim() - 1 - a) + 1] = r
        p = tnf.pad(t, pad)
        t = sum(p.narrow(a, k, t.shape[a]) for k in range(2 * r + 1))
    return t


def _similarity64(sim, F, W, mask, window):
    n = float(mask.sum())
    if n == 0:
        return (W * 0).sum()
    if sim == "mse":
        return (mask * (W - F) ** 2).sum() / n
    if sim == "ncc":
        a, b = mask * (F - (mask * F).sum() / n), mask * (W - (mask * W).sum() / n)
        return 1.0 - (a * b).sum() / torch.sqrt((a * a).sum() * (b * b).sum() + EPS)
    r, cnt = window // 2, float(window ** F.dim())
    sf, sw = _box64(F, r), _box64(W, r)
    cov = _box64(F * W, r) - sf * sw / cnt
    vf, vw = _box64(F * F, r) - sf * sf / cnt, _box64(W * W, r) - sw * sw / cnt
    return 1.0 - (mask * cov / torch.sqrt(vf * vw + EPS)).sum() / n


def _objective64(case, shape, F, M, c, steps=None):
    """{J, S, R, n_mask} and dJ/dc in 64 bits, the gradient by autograd."""
    with torch.enable_grad():
        c = c.detach().double().requires_grad_(True)
        F, M = F.double(), M.double()
        u = _displacement64(shape, case["spacing"], c)
        if steps is not None:
            u = u * 2.0 ** -steps
            for _ in range(steps):
                axes = [(cell, y.clamp(0, n - 1), inside, n)
                        for cell, y, inside, n in _sample64(shape, u)]
                u = u + _interpolate64(u, shape, axes)
        axes = _sample64(shape, u)
        mask = math.prod([a[2].double() for a in axes])
        axes = [(cell, torch.where(inside, y, y.detach().clamp(0, n - 1)), inside, n)
                for cell, y, inside, n in axes]
        W = mask * _interpolate64(M, shape, axes)
        S = _similarity64(case["sim"], F, W, mask, case.get("window", 7))
        R = sum(u.diff(dim=a).square().sum() for a in range(1, u.dim())) / math.prod(shape)
        J = S + LAMBDA * R
        (g,) = torch.autograd.grad(J, c)
    return torch.stack([J.detach(), S.detach(), R.detach(), mask.sum()]), g


def _adam64(shape, c, g, m, v):
    """One Adam step after STEP0, in the coordinates in which an image spans [-1, 1]."""
    half = torch.tensor([(n - 1) / 2.0 for n in reversed(shape)], device="cuda",
                        dtype=torch.float64).view((-1,) + (1,) * len(shape))
    g, t = g * half, STEP0 + 1
    m = BETA1 * m.double() + (1 - BETA1) * g
    v = BETA2 * v.double() + (1 - BETA2) * g * g
    step = LR * (m / (1 - BETA1 ** t)) / (torch.sqrt(v / (1 - BETA2 ** t)) + ADAM_EPS)
    return c.double() - step * half, m, v


def _taps(x, stride, o):
    """The 27 shifted views of channels-last x, zero padded, at the output grid."""
    p = tnf.pad(x, (0, 0, 1, 1, 1, 1, 1, 1))
    for t in range(27):
        a = (t // 9, t // 3 % 3, t % 3)
        yield t, tuple(slice(a[k], a[k] + (o[k] - 1) * stride + 1, stride) for k in range(3)), p


def _conv64(case, x, w, b, gy):
    cin, cout, stride = LAYERS[case["layer"]]
    o = tuple((n - 1) // stride + 1 for n in x.shape[1:4])
    x, w = x.double(), w.to(torch.bfloat16).double()
    y = b.double().expand((x.shape[0],) + o + (cout,)).clone()
    for t, at, p in _taps(x, stride, o):
        y += p[(slice(None),) + at] @ w[:, t].T
    out = {"y": y if case["layer"] == 6 else y.relu()}
    if gy is None:
        return out
    g2 = gy.double().reshape(-1, cout)
    gw = torch.zeros_like(w)
    gp = torch.zeros_like(tnf.pad(x, (0, 0, 1, 1, 1, 1, 1, 1)))
    for t, at, p in _taps(x, stride, o):
        gw[:, t] = g2.T @ p[(slice(None),) + at].reshape(-1, cin)
        if cin % 16 == 0:
            gp[(slice(None),) + at] += gy.double() @ w[:, t]
    out.update(gw=gw, gb=g2.sum(0))
    if cin % 16 == 0:
        out["gx"] = gp[:, 1:-1, 1:-1, 1:-1] * (x > 0)
    return out


def _level64(img, f):
    s, r = f / 2.0, int(3 * f / 2.0)
    k = torch.exp(-torch.arange(-r, r + 1, device="cuda", dtype=torch.float64) ** 2 / (2 * s * s))
    k, img = k / k.sum(), img.double()
    for a, n in enumerate(img.shape):
        at = torch.arange(0, n, f, device="cuda")
        img = sum(k[t + r] * img.index_select(a, (at + t).clamp(0, n - 1))
                  for t in range(-r, r + 1))
    return img


def _refine64(c, fine):
    """Two-scale relation of the cubic B-spline, times 2 for the finer voxels."""
    c = c.double()
    for a, n in enumerate(fine[1:]):
        i = torch.arange(n, device="cuda")[:, None] - 1
        j = torch.arange(c.shape[a + 1], device="cuda")[None, :] - 1
        k = i - 2 * j
        w = torch.tensor([1, 4, 6, 4, 1], device="cuda", dtype=torch.float64) / 8.0
        T = torch.where(k.abs() <= 2, w[(k + 2).clamp(0, 4)], torch.zeros((), device="cuda",
                                                                       dtype=torch.float64))
        c = torch.movedim(torch.tensordot(c, T, dims=([a + 1], [1])), -1, a + 1)
    return 2.0 * c


@torch.no_grad()
def exact(case, seed):
    kind = case["kind"]
    if kind in ("objective", "diffeo"):
        shape, F, M, c, _, _ = _objective_inputs(case, seed)
        value, g = _objective64(case, shape, F, M, c, case.get("steps"))
        return {"value": value, "grad": g}
    if kind == "iteration":
        shape, F, M, c, m, v = _objective_inputs(case, seed)
        value, g = _objective64(case, shape, F, M, c)
        c, m, v = _adam64(shape, c, g, m, v)
        return {"value": value, "grad": g, "ctrl": c, "m": m, "v": v}
    if kind == "batch":
        out = {"ctrl": [], "m": [], "v": [], "values": []}
        for shape, F, M, c, m, v in _batch_inputs(case, seed):
            value, g = _objective64(dict(spacing=case["spacing"], sim="mse"), shape, F, M, c)
            for name, t in zip(("ctrl", "m", "v"), _adam64(shape, c, g, m, v)):
                out[name].append(t)
            out["values"].append(value[None])
        return out
    if kind == "conv":
        return _conv64(case, *_conv_inputs(case, seed))
    if kind == "pairs":
        shape, table, ctrl = _pairs_inputs(case, seed)
        Ms, xs, d = [], [], 3
        pos = [p.double() for p in _points(shape)]
        for tab, c in zip(table.double(), ctrl.double()):
            # the blob separates over the axes: one product per blob and axis
            e = [torch.exp(-(pos[k].reshape(1, -1) - tab[:, k:k + 1]) ** 2
                           / (2 * tab[:, 3:4] ** 2)) for k in range(d)]
            M = torch.einsum("b,bz,by,bx->zyx", tab[:, 4], e[2], e[1], e[0])
            axes = _sample64(shape, _displacement64(shape, 8, c))
            mask = math.prod([a[2].double() for a in axes])
            axes = [(cell, y.clamp(0, n - 1), i, n) for cell, y, i, n in axes]
            Ms.append(M)
            xs.append(torch.stack([mask * _interpolate64(M, shape, axes), M], -1))
        return {"M": torch.stack(Ms), "x": torch.stack(xs)}
    shape, _, F, M, c = _level_inputs(case, seed)
    return {"F": _level64(F, case["factor"]), "M": _level64(M, case["factor"]),
            "ctrl": _refine64(c, _lattice(shape, case["spacing"]))}
