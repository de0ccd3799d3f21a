"""What a user of this framework has it do, as cases that can be timed and checked.

Every case goes through the package's public entry points.  The inputs are made on the GPU from a seed and follow the
workloads of this repository: a small ball of Gaussians, and a synthetic thorax whose measured projections are the
closed-form line integrals of its ellipsoids.  ``exact`` restates each path in float64 with plain torch.
"""
import math

import numpy as np
import torch

import paper_2506_22280_gb300 as pkg
from paper_2506_22280_gb300 import digs as D

CUTOFF = 3.5
N_PROJ = 680  # projections of a whole scan
BODY = (120.0, 85.0, 120.0)
LUNGS = (((55.0, 0.0, 20.0), (40.0, 55.0, 80.0)), ((-55.0, 0.0, 20.0), (40.0, 55.0, 80.0)))
TUMOUR = ((-55.0, 0.0, 30.0), (7.5, 7.5, 7.5))
CNN_EDGES, CNN_CHANNELS = (128, 64, 32, 16, 8), (1, 32, 64, 128, 128)

# learning rates and schedule of a run that is nearly over: (mu0, log-scale, quaternion, density, phi, w)
LR0, LR1, TOTAL_ITERS, AT_ITER = (0.02, 0.005, 0.002, 0.01, 0.02, 0.01), 0.01, 6000, 5900
MOMENT = 1e-6


def _projector_case(name, kind, n, views, nu, nv, pitch, R, **more):
    c = {"name": name, "kind": kind, "n": n, "views": views, "nu": nu, "nv": nv, "pitch": pitch, "R": R,
         "spacing": 16.0, "tile": 16, "lanes": 16, "model": "exact", "sorted": True, "scans": 1, "off_u": 0.0}
    c.update(more)
    return c


def listed():
    return [
        # the smallest call: project a small test cloud (2,000 Gaussians, 16 views of 64 x 64)
        _projector_case("tiny_forward", "forward", 2000, 16, 64, 64, 1.6, 2, spacing=10.0),
        # one eager optimisation step on that cloud: launches and host work are most of it
        _projector_case("tiny_step", "step", 2000, 16, 64, 64, 1.6, 2, spacing=10.0),
        # the optimisation loop of a reconstruction before a batch size is tuned: 16 projections per eager step
        _projector_case("thorax_step_16", "step", 100_000, 16, 256, 256, 1.6, 3),
        # the same loop at the tuned batch size, each step replayed from its captured graph
        _projector_case("thorax_step_128", "replay", 100_000, 128, 256, 256, 1.6, 3),
        # scoring a scan of 680 projections: the forward and loss of its last, shorter chunk (680 = 5 x 128 + 40)
        _projector_case("scan_loss_40", "loss", 100_000, 40, 256, 256, 1.6, 3),
        # differentiable rendering inside a user's own torch program: odd sizes, shifted detector, cloud in no
        # particular order, the 2D-Gaussian projection model
        _projector_case("render_ragged", "render", 33_331, 7, 203, 151, 2.1, 2, model="ewa", sorted=False,
                        off_u=11.5),
        # differentiable rendering at the largest scale: 500k Gaussians, 512 x 512 detector, fine lattice, four ranks
        _projector_case("scale_render", "render", 500_000, 8, 512, 512, 0.8, 4, spacing=8.0),
        # four scans of 30k, 60k, 120k and 200k Gaussians reconstructed together, 64 projections per captured step
        _projector_case("batch_step_64", "replay", 410_000, 64, 256, 256, 1.6, 3, scans=4),
        # one training step of the weight predictor at its batch size (BF16 operands on the tensor cores)
        {"name": "cnn_train_256", "kind": "cnn_train", "batch": 256, "R": 3},
        # the trained predictor proposes the weights of a whole scan of 256 x 256 projections
        {"name": "cnn_predict_680", "kind": "cnn_predict", "batch": 680, "edge": 256, "R": 3},
        # the predictor's forward and backward in FP32, the default mode of those two calls
        {"name": "cnn_fp32_64", "kind": "cnn_fp32", "batch": 64, "R": 3},
        # judging a reconstruction at one time point: attenuation volume and displacement field on a 2 mm grid
        {"name": "volume_128", "kind": "volume", "n": 100_000, "R": 3, "spacing": 16.0, "sorted": True,
         "gx": 128, "gy": 128, "gz": 128},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["forward", "step", "step", "replay", "loss", "render", "render", "replay", "cnn_train",
                       "cnn_predict", "cnn_fp32", "volume"])
    if kind == "cnn_train":
        return {"kind": kind, "batch": _log_int(rng, 16, 300), "R": rng.randint(1, 4)}
    if kind == "cnn_predict":
        return {"kind": kind, "batch": _log_int(rng, 1, 900), "edge": rng.choice([128, 256]), "R": rng.randint(1, 4)}
    if kind == "cnn_fp32":
        return {"kind": kind, "batch": _log_int(rng, 2, 80), "R": rng.randint(1, 4)}
    if kind == "volume":
        return {"kind": kind, "n": _log_int(rng, 2000, 130_000), "R": rng.randint(1, 4),
                "spacing": rng.choice([8.0, 12.0, 16.0]), "sorted": rng.random() < 0.7, "gx": rng.randint(40, 140),
                "gy": rng.randint(40, 140), "gz": rng.randint(40, 140)}
    n = _log_int(rng, 600, 500_000)
    body = n >= 10_000
    nu, nv = (rng.randint(100, 512), rng.randint(100, 512)) if body else (rng.randint(40, 128), rng.randint(40, 128))
    scans = rng.randint(2, 6) if kind == "replay" and body and rng.random() < 0.5 else 1
    c = {"kind": kind, "n": n, "views": _log_int(rng, 1, 128), "nu": nu, "nv": nv,
         "pitch": round((410.0 if body else 110.0) / max(nu, nv) * rng.uniform(0.7, 1.1), 3), "R": rng.randint(1, 4),
         "spacing": rng.choice([8.0, 12.0, 16.0]) if body else 10.0, "tile": rng.choice([8, 16, 16, 16, 32]),
         "lanes": rng.choice([16, 16, 16, 32]),
         "model": rng.choice(["exact", "exact", "exact" if kind in ("step", "replay") else "ewa", "parallel"]),
         "sorted": rng.random() < 0.7, "scans": scans, "off_u": rng.choice([0.0, 0.0, 7.25])}
    while c["views"] > 1 and (_pairs(c) > 2.5e9 or c["views"] * n > 9_000_000):
        c["views"] = c["views"] // 2 + c["views"] % 2 if c["views"] > 2 else 1
    return c


# ---- what a pass cannot do without ------------------------------------------------------------------
def _is_body(c):
    return c["n"] >= 10_000


def _pairs(c):
    """About how many (pixel, Gaussian) pairs lie within the cutoff over all views of a case."""
    s2 = 9.0 * math.exp(0.0625) if _is_body(c) else 4.0 * math.exp(0.16)
    area = math.pi * CUTOFF ** 2 * s2 * (1.0 if c["model"] == "parallel" else 2.25) / c["pitch"] ** 2
    return c["n"] / c["scans"] * c["views"] * min(area, c["nu"] * c["nv"])


def _cnn_work(B, train, operand_bytes):
    flops = 0.0
    act = B * 128 * 128 * 4
    for l in range(4):
        m, k, n = B * CNN_EDGES[l + 1] ** 2, 9 * CNN_CHANNELS[l], CNN_CHANNELS[l + 1]
        flops += 2.0 * m * k * n * ((3 if l else 2) if train else 1)
        act += m * n * operand_bytes * (3 if train else 0)
    flops += 2.0 * B * 8194 * 128 * (3 if train else 1)
    return {"bytes": act + (1.3e6 * 4) * (5 if train else 1), "flops": flops}


def work(case):
    k = case["kind"]
    if k == "cnn_train":
        return _cnn_work(case["batch"], True, 2)
    if k == "cnn_fp32":
        return _cnn_work(case["batch"], True, 4)
    if k == "cnn_predict":
        w = _cnn_work(case["batch"], False, 2)
        return {"bytes": w["bytes"] + case["batch"] * (case["edge"] ** 2 - 128 ** 2) * 4.0, "flops": w["flops"]}
    if k == "volume":
        vox, r = case["gx"] * case["gy"] * case["gz"], case["R"]
        h = [_grid(case)["spacing"][a] for a in range(3)]
        pairs = case["n"] * 4.0 / 3.0 * math.pi * CUTOFF ** 3 * (27.0 if _is_body(case) else 8.0) / (h[0] * h[1] * h[2])
        return {"bytes": vox * 16.0 + case["n"] * 44.0, "flops": pairs * 24.0 + vox * 64 * 6.0 * r}
    n, r, px = case["n"], case["R"], case["views"] * case["nu"] * case["nv"]
    pairs = _pairs(case)
    nphi = 3 * r * _lattice(case)["nx"] ** 3 * case["scans"]
    if k in ("forward", "loss"):
        return {"bytes": n * 44.0 + nphi * 4.0 + px * (4.0 if k == "forward" else 8.0), "flops": pairs * 20.0}
    state = 28.0 if k in ("step", "replay") else 8.0  # parameters, gradients and Adam's moments, or the first two
    return {"bytes": (n * 11 + nphi) * state + px * 8.0, "flops": pairs * 68.0}


# ---- inputs -----------------------------------------------------------------------------------------
def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed))


def _randn(g, *shape):
    return torch.randn(*shape, generator=g, device="cuda")


def _rand(g, *shape):
    return torch.rand(*shape, generator=g, device="cuda")


def _lattice(c):
    if _is_body(c):
        nodes = int(math.ceil(256.0 / c["spacing"])) + 3
        origin = -128.0 - c["spacing"]
    else:
        nodes, origin = 8, -35.0
    return {"nx": nodes, "ny": nodes, "nz": nodes, "R": c["R"], "origin": (origin,) * 3,
            "spacing": (c["spacing"] if _is_body(c) else 10.0,) * 3}


def _inside(x, ell):
    c, s = ell
    return sum(((x[:, a] - c[a]) / s[a]) ** 2 for a in range(3)) <= 1.0


def _cloud(c, n, g):
    """(mu0, scale, quat, rho) of one scan in the state that its optimisation starts from."""
    semi = BODY if _is_body(c) else (32.0, 32.0, 32.0)
    d = _randn(g, n, 3)
    x = d / d.norm(dim=1, keepdim=True) * _rand(g, n, 1) ** (1.0 / 3.0) * torch.tensor(semi, device="cuda")
    if _is_body(c):
        mu = torch.where(_inside(x, ((0.0, 0.0, 0.0), BODY)), 0.02, 0.0)
        for ell in LUNGS:
            mu = torch.where(_inside(x, ell), 0.004, mu)
        mu = torch.where(_inside(x, TUMOUR), 0.02, mu)
        nbar = n / (4.0 / 3.0 * math.pi * BODY[0] * BODY[1] * BODY[2])
        scale = 3.0 * torch.exp(0.25 * _randn(g, n, 3))
        rho = mu / (nbar * (2 * math.pi) ** 1.5 * (2.5 * math.exp(0.03125)) ** 3) * (0.5 + _rand(g, n))
        x = x + _randn(g, n, 3)
    else:
        scale = 2.0 * torch.exp(0.4 * _randn(g, n, 3))
        rho = 0.005 + 0.025 * _rand(g, n)
    quat = _randn(g, n, 4)
    quat = quat / quat.norm(dim=1, keepdim=True)
    if c["sorted"]:  # lattice-cell order, as the workloads of this repository store their clouds
        lat = _lattice(c)
        cell = torch.floor((x - lat["origin"][0]) / lat["spacing"][0]).long() + 64
        order = torch.argsort((cell[:, 2] * 1024 + cell[:, 1]) * 1024 + cell[:, 0], stable=True)
        x, scale, quat, rho = x[order], scale[order], quat[order], rho[order]
    return [t.contiguous() for t in (x, scale, quat, rho)]


def _scan_sizes(c):
    """Uneven scans: 30 : 60 : 120 : 200 for four, a like progression otherwise."""
    s = c["scans"]
    if s == 1:
        return [c["n"]]
    share = [3.0, 6.0, 12.0, 20.0] if s == 4 else [1.0 + 0.8 * k for k in range(s)]
    sizes = [int(c["n"] * x / sum(share)) for x in share]
    sizes[-1] = c["n"] - sum(sizes[:-1])
    return sizes


def _views(c, seed):
    """Views of the batch (evenly spread over the scan, starting anywhere) and their projection numbers."""
    rows = 16 if not _is_body(c) and c["views"] <= 16 else N_PROJ
    start = int(np.random.default_rng(seed).integers(rows))
    per = -(-c["views"] // c["scans"])
    out, ids = [], []
    for v in range(c["views"]):
        s, j = v // per, v % per
        p = (start + 37 * s + j * max(1, rows // per)) % rows
        a = 2 * math.pi * p / rows
        cs, sn = math.cos(a), math.sin(a)
        out.append({"src": (1000.0 * cs, 1000.0 * sn, 0.0), "det_c": (-500.0 * cs, -500.0 * sn, 0.0),
                    "e_u": (-sn, cs, 0.0), "e_v": (0.0, 0.0, 1.0), "du": c["pitch"], "dv": c["pitch"],
                    "off_u": c["off_u"], "off_v": 0.0, "nu": c["nu"], "nv": c["nv"],
                    "parallel": c["model"] == "parallel", "scan": s})
        ids.append(rows * s + p)
    return out, ids, rows


def _motion(c, rows, g):
    """Control points and the weights of every time point, as an optimisation under way holds them."""
    lat = _lattice(c)
    k = c["scans"]
    shape = (c["R"], lat["nz"], lat["ny"], lat["nx"], 3)
    if _is_body(c):
        phi = 0.1 * _randn(g, k, *shape)
        phi[:, 0, ..., 2] += 0.3
        t = torch.arange(rows, device="cuda") * (60.0 / rows)
        w = torch.stack([3.0 * torch.sin(2 * math.pi * t / 4.25) ** 2, 0.9 * torch.sin(4 * math.pi * t / 4.25),
                         2.0 * torch.sin(2 * math.pi * t / 90.0), 0.5 * torch.sin(2 * math.pi * t / 0.9)], 1)
        w = w[:, :c["R"]].repeat(k, 1) + 0.1 * _randn(g, rows * k, c["R"])
    else:
        phi = _randn(g, k, *shape)
        w = 0.7 * _randn(g, rows * k, c["R"])
    return (phi if k > 1 else phi[0]).contiguous(), w.contiguous()


def _rays(v):
    """Origins and directions [nv][nu][3] (float64) of a view's rays, and the pixel centres."""
    f = lambda x: torch.tensor(x, dtype=torch.float64, device="cuda")  # noqa: E731
    src, det, eu, ev = f(v["src"]), f(v["det_c"]), f(v["e_u"]), f(v["e_v"])
    i = (torch.arange(v["nu"], device="cuda", dtype=torch.float64) - (v["nu"] - 1) / 2 + v["off_u"]) * v["du"]
    j = (torch.arange(v["nv"], device="cuda", dtype=torch.float64) - (v["nv"] - 1) / 2 + v["off_v"]) * v["dv"]
    X = det + i[None, :, None] * eu + j[:, None, None] * ev
    d = (det - src).expand_as(X) if v["parallel"] else X - src
    return X, d / d.norm(dim=-1, keepdim=True)


def _chord(o, d, ell, dz):
    c, s = (torch.tensor(x, dtype=torch.float64, device="cuda") for x in ell)
    p, q = (o - c - dz * torch.tensor([0.0, 0.0, 1.0], dtype=torch.float64, device="cuda")) / s, d / s
    a, b, e = (q * q).sum(-1), (p * q).sum(-1), (p * p).sum(-1) - 1.0
    return 2.0 * torch.sqrt((b * b - a * e).clamp_min(0.0)) / a


def _measured(c, views, g):
    """Line integrals of the phantom, its lungs displaced by the breathing, with a little noise."""
    out = []
    for k, v in enumerate(views):
        X, d = _rays(v)
        dz = 6.0 * math.sin(1.3 * k) ** 2
        if _is_body(c):
            m = 0.02 * _chord(X, d, ((0.0, 0.0, 0.0), BODY), 0.0) + 0.016 * _chord(X, d, TUMOUR, dz)
            for ell in LUNGS:
                m = m - 0.016 * _chord(X, d, ell, dz)
        else:
            m = 0.04 * _chord(X, d, ((0.0, 0.0, 0.0), (32.0, 32.0, 32.0)), 0.1 * dz)
        out.append(m.float())
    m = torch.stack(out)
    return (m + 0.01 * _randn(g, *m.shape)).contiguous()


def _scene(c, seed):
    g = _gen(seed)
    clouds = [_cloud(c, n, g) for n in _scan_sizes(c)]
    gauss = [torch.cat([s[a] for s in clouds]).contiguous() for a in range(4)]
    views, ids, rows = _views(c, seed)
    phi, w = _motion(c, rows, g)
    return gauss, phi, w, views, ids, g


def _grid(c):
    half = (128.0, 100.0, 128.0) if _is_body(c) else (35.0, 35.0, 35.0)
    dims = (c["gx"], c["gy"], c["gz"])
    h = [2.0 * half[a] / dims[a] for a in range(3)]
    return {"nx": dims[0], "ny": dims[1], "nz": dims[2], "origin": [0.5 * h[a] - half[a] for a in range(3)], "spacing": h}


def _moments(case, total, g):
    """Adam's moments of a run under way: steady second moments, first moments within their spread."""
    return 0.1 * MOMENT * _randn(g, total), MOMENT ** 2 * (0.5 + _rand(g, total))


def _pictures(case, seed):
    """Projections of bodies of several widths, their angles and the weights that a training pair has."""
    g = _gen(seed)
    B, e = case["batch"], case.get("edge", 128)
    y, x = torch.meshgrid(torch.linspace(-1, 1, e, device="cuda"), torch.linspace(-1, 1, e, device="cuda"), indexing="ij")
    a = (0.55 + 0.2 * _rand(g, B, 1, 1)), (0.6 + 0.2 * _rand(g, B, 1, 1))
    img = 4.0 * (1.0 - (x / a[0]) ** 2 - (y / a[1]) ** 2).clamp_min(0.0).sqrt()
    for _ in range(2):
        cx, cy, s = 0.6 * _rand(g, B, 1, 1) - 0.3, 0.4 * _rand(g, B, 1, 1) - 0.2, 0.15 + 0.15 * _rand(g, B, 1, 1)
        img = img - 0.8 * (1.0 - ((x - cx) / s) ** 2 - ((y - cy) / (1.6 * s)) ** 2).clamp_min(0.0).sqrt()
    img = (img + 0.02 * _randn(g, B, e, e)).contiguous()
    t = 2 * math.pi * _rand(g, B)
    return img, torch.stack([torch.cos(t), torch.sin(t)], 1).contiguous(), _randn(g, B, case["R"]), g


def _net(case, seed):
    """A predictor whose parameters are drawn from the seed: He-normal weights, small biases."""
    net = pkg.WeightPredictor(case["R"], seed=0, input_scale=0.25)
    net.params.copy_(_net_params(case, seed, net.params.numel()))
    return net


def _net_layout(R):
    out = []
    for l in range(4):
        out += [((CNN_CHANNELS[l + 1], 3, 3, CNN_CHANNELS[l]), 9 * CNN_CHANNELS[l]), ((CNN_CHANNELS[l + 1],), 0)]
    return out + [((128, 8194), 8194), ((128,), 0), ((R, 128), 128), ((R,), 0)]


def _net_params(case, seed, total):
    g = _gen(seed + 77)
    p = torch.cat([(_randn(g, math.prod(s)) * (math.sqrt(2.0 / f) if f else 0.05)) for s, f in _net_layout(case["R"])])
    assert p.numel() == total
    return p


# ---- prepare and run --------------------------------------------------------------------------------
def prepare(case, seed):
    k = case["kind"]
    if k.startswith("cnn"):
        img, cs, target, g = _pictures(case, seed)
        s = {"kind": k, "net": _net(case, seed), "img": img, "cs": cs, "target": target}
        if k == "cnn_train":
            s["img"] = (img * s["net"].input_scale).contiguous()
            s["net"].m[:], s["net"].v[:] = _moments(case, s["net"].m.numel(), g)
            s["net"].v *= 1e6
            s["net"].m *= 1e3
            s["net"].step_count = 400
        if k == "cnn_fp32":
            s["img"] = (img * s["net"].input_scale).contiguous()
            s["grad_w"] = (2.0 / (case["batch"] * case["R"]) * target).contiguous()
        s["net"]._ws(min(case["batch"], 512))
        return s
    if k == "volume":
        c = dict(case, scans=1, views=1)
        g = _gen(seed)
        gauss = _cloud(c, c["n"], g)
        phi, w = _motion(c, 16, g)
        return {"kind": k, "gauss": gauss, "phi": phi, "w": w[5].contiguous(), "lat": _lattice(c), "grid": _grid(c)}
    gauss, phi, w, views, ids, g = _scene(case, seed)
    lat = _lattice(case)
    if k in ("step", "replay"):
        rec = pkg.Reconstruction(*gauss, phi, w, lat, D.adam_config(LR0, [LR1 * x for x in LR0], TOTAL_ITERS),
                                 tile=case["tile"], bwd_lanes=case["lanes"],
                                 scan_sizes=_scan_sizes(case) if case["scans"] > 1 else None)
        rec.m[:], rec.v[:] = _moments(case, rec.m.numel(), g)
        rec.state.iter = AT_ITER
        s = {"kind": k, "rec": rec, "meas": _measured(case, views, g), "ids": ids, "views": views}
        if k == "replay":
            rec.clone().step(s["meas"], ids, views)  # an eager step on a copy loads the kernels
            s["graph"] = rec.capture([(s["meas"], ids, views)])[0]
        else:
            rec._reserve(views, len(ids), ids)
        return s
    w = w[torch.as_tensor(ids, device="cuda")].contiguous()
    pj = pkg.Projector(lat, views, tile=case["tile"], bwd_lanes=case["lanes"], ewa=case["model"] == "ewa")
    args = [*gauss, phi, w]
    pj.reserve(*args)
    s = {"kind": k, "pj": pj, "args": args}
    if k == "loss":
        s["meas"] = _measured(case, views, g)
    if k == "render":
        s["args"] = [t.requires_grad_() for t in args]
        s["up"] = _randn(g, case["views"], case["nv"], case["nu"])
    return s


def run(s):
    k = s["kind"]
    if k == "forward":
        return s["pj"].forward(*s["args"])
    if k == "loss":
        img = torch.empty_like(s["meas"])
        return {"loss": s["pj"].loss(*s["args"], s["meas"], proj=img), "proj": img}
    if k == "render":
        img = pkg.DigsRender.apply(s["pj"], *s["args"])
        return [img.detach(), *torch.autograd.grad(img, s["args"], s["up"])]
    if k in ("step", "replay"):
        rec = s["rec"]
        if k == "replay":
            s["graph"].replay()
        else:
            rec.step(s["meas"], s["ids"], s["views"])
        return {"loss": rec.loss, "grad": rec.grad, "mu0": rec.mu0, "scale": rec.scale, "quat": rec.quat,
                "rho": rec.rho, "phi": rec.phi, "w": rec.w}
    if k == "cnn_train":
        net = s["net"]
        loss = net.train_step(s["img"], s["cs"], s["target"], 3e-4)
        return {"loss": loss, "grad": net.grad, "params": net.params}
    if k == "cnn_predict":
        net = s["net"]
        return net.predict(net.prepare(s["img"]), s["cs"])
    if k == "cnn_fp32":
        net = s["net"]
        out = net.forward(s["img"], s["cs"])
        return {"out": out, "grad": net.backward(s["grad_w"])}
    vol = D.voxelize(*s["gauss"], s["phi"], s["w"], s["lat"], s["grid"])
    return {"volume": vol, "dvf": D.dvf(s["phi"], s["w"], s["lat"], s["grid"])}


# ---- the same in 64 bits ----------------------------------------------------------------------------
def _bspline(u):
    return torch.stack([(1 - u) ** 3 / 6, (3 * u ** 3 - 6 * u ** 2 + 4) / 6, (-3 * u ** 3 + 3 * u ** 2 + 3 * u + 1) / 6,
                        u ** 3 / 6], -1)


def _bspline_d(u):
    return torch.stack([-(1 - u) ** 2 / 2, (3 * u ** 2 - 4 * u) / 2, (-3 * u ** 2 + 2 * u + 1) / 2, u ** 2 / 2], -1)


def _ffd64(phi, lat, x, jacobian=True):
    """u_r(x) [n][R][3] and its gradient [n][R][3][3]; phi [R][nz][ny][nx][3]."""
    h = lat["spacing"]
    p = (x - torch.tensor(lat["origin"], dtype=x.dtype, device=x.device)) / torch.tensor(h, dtype=x.dtype, device=x.device)
    f = torch.floor(p).detach()
    B = [_bspline(p[:, a] - f[:, a]) for a in range(3)]
    dB = [_bspline_d(p[:, a] - f[:, a]) / h[a] for a in range(3)]
    f = f.long() - 1
    n = (lat["nx"], lat["ny"], lat["nz"])
    flat = phi.reshape(phi.shape[0], -1, 3)
    U, dU = 0.0, 0.0
    for c in range(4):
        for b in range(4):
            for a in range(4):
                i, j, k = f[:, 0] + a, f[:, 1] + b, f[:, 2] + c
                ok = (i >= 0) & (i < n[0]) & (j >= 0) & (j < n[1]) & (k >= 0) & (k < n[2])
                at = torch.where(ok, (k * n[1] + j) * n[0] + i, 0)
                d = (flat.index_select(1, at) * ok[None, :, None]).permute(1, 0, 2)
                U = U + (B[0][:, a] * B[1][:, b] * B[2][:, c])[:, None, None] * d
                if jacobian:
                    g = torch.stack([dB[0][:, a] * B[1][:, b] * B[2][:, c], B[0][:, a] * dB[1][:, b] * B[2][:, c],
                                     B[0][:, a] * B[1][:, b] * dB[2][:, c]], -1)
                    dU = dU + d[..., None] * g[:, None, None, :]
    return U, dU


def _inv3(m):
    a, b, c = m[:, 0], m[:, 1], m[:, 2]
    r = torch.stack([torch.linalg.cross(b, c), torch.linalg.cross(c, a), torch.linalg.cross(a, b)], -1)
    det = (a * torch.linalg.cross(b, c)).sum(-1)
    return r / det[:, None, None], det


def _cov64(scale, quat):
    q = quat / quat.norm(dim=-1, keepdim=True)
    w, x, y, z = q.unbind(-1)
    R = torch.stack([1 - 2 * (y * y + z * z), 2 * (x * y - w * z), 2 * (x * z + w * y), 2 * (x * y + w * z),
                     1 - 2 * (x * x + z * z), 2 * (y * z - w * x), 2 * (x * z - w * y), 2 * (y * z + w * x),
                     1 - 2 * (x * x + y * y)], -1).reshape(-1, 3, 3)
    M = R * scale[:, None, :]
    return M @ M.transpose(1, 2)


def _deformed64(mu0, scale, quat, U, dU, w):
    K = torch.eye(3, dtype=mu0.dtype, device=mu0.device) + torch.einsum("r,nrij->nij", w, dU)
    mu = mu0 + torch.einsum("r,nri->ni", w, U)
    S = K @ _cov64(scale, quat) @ K.transpose(1, 2)
    return mu, S, _inv3(K)[1]


def _coefs64(v, ewa, mu, S, rho):
    """Per Gaussian, what its pixel values are made of, and a box that holds its cutoff region.

    Exact cone beam: a (6 coefficients in i, j), b (3), c and rho with E = c - b^2 / a.  Parallel beam and the
    2D-Gaussian model: E as 6 coefficients and the amplitude."""
    t = lambda x: torch.tensor(x, dtype=mu.dtype, device=mu.device)  # noqa: E731
    src, det, eu, ev = t(v["src"]), t(v["det_c"]), t(v["e_u"]), t(v["e_v"])
    nd = torch.linalg.cross(eu, ev)
    nd = nd if torch.dot(nd, det - src) > 0 else -nd
    ci, cj = (v["nu"] - 1) / 2 - v["off_u"], (v["nv"] - 1) / 2 - v["off_v"]
    X0 = det - ci * v["du"] * eu - cj * v["dv"] * ev
    gi, gj = v["du"] * eu, v["dv"] * ev
    P = _inv3(S)[0]
    sdd = torch.dot(det - src, nd)
    quad = lambda Q, p, q: torch.einsum("...i,nij,...j->n", p, Q, q)  # noqa: E731
    if v["parallel"]:
        d = (det - src) / (det - src).norm()
        s = ((det - mu) @ nd) / torch.dot(d, nd)
        xc = ci + ((mu - det + s[:, None] * d) @ eu) / v["du"]
        yc = cj + ((mu - det + s[:, None] * d) @ ev) / v["dv"]
        J = torch.stack([eu - torch.dot(d, eu) / torch.dot(d, nd) * nd, ev - torch.dot(d, ev) / torch.dot(d, nd) * nd])
        J = (J / t([v["du"], v["dv"]])[:, None]).expand(mu.shape[0], 2, 3)
        alive = torch.ones_like(rho, dtype=torch.bool)
    else:
        rel = mu - src
        tx, ty, tz = rel @ eu, rel @ ev, rel @ nd
        fa, fb = sdd / v["du"], sdd / v["dv"]
        xc, yc = ci + (torch.dot(src - det, eu) + sdd * tx / tz) / v["du"], cj + (torch.dot(src - det, ev) + sdd * ty / tz) / v["dv"]
        J = torch.stack([(fa / tz)[:, None] * eu - (fa * tx / tz ** 2)[:, None] * nd,
                         (fb / tz)[:, None] * ev - (fb * ty / tz ** 2)[:, None] * nd], 1)
        alive = tz > 0
    C = J @ S @ J.transpose(1, 2)
    hx, hy = CUTOFF * C[:, 0, 0].sqrt() * 1.08 + 2.0, CUTOFF * C[:, 1, 1].sqrt() * 1.08 + 2.0
    box = torch.stack([(xc - hx).ceil().clamp(0, v["nu"]), (xc + hx).floor().clamp(-1, v["nu"] - 1),
                       (yc - hy).ceil().clamp(0, v["nv"]), (yc + hy).floor().clamp(-1, v["nv"] - 1)], 1).detach().long()
    if not v["parallel"] and not ewa:
        D0, m = X0 - src, src - mu
        Pm = torch.einsum("nij,nj->ni", P, m)
        cc = (m * Pm).sum(-1)
        co = torch.stack([quad(P, D0, D0), 2 * quad(P, D0, gi), 2 * quad(P, D0, gj), quad(P, gi, gi),
                          2 * quad(P, gi, gj), quad(P, gj, gj), Pm @ D0, Pm @ gi, Pm @ gj, cc, rho], 1)
        return co, box, alive & (cc > CUTOFF ** 2)
    if v["parallel"]:
        Pd = P @ d
        a = Pd @ d
        Q = P - Pd[:, :, None] * Pd[:, None, :] / a[:, None, None]
        amp = rho * torch.sqrt(2 * math.pi / a)
        m = X0 - mu
        Qm = torch.einsum("nij,nj->ni", Q, m)
        co = torch.stack([(m * Qm).sum(-1), 2 * Qm @ gi, 2 * Qm @ gj, quad(Q, gi, gi), 2 * quad(Q, gi, gj),
                          quad(Q, gj, gj), amp], 1)
        return co, box, alive
    det2 = C[:, 0, 0] * C[:, 1, 1] - C[:, 0, 1] ** 2
    n00, n01, n11 = C[:, 1, 1] / det2, -C[:, 0, 1] / det2, C[:, 0, 0] / det2
    J3 = torch.cat([J, (rel / rel.norm(dim=1, keepdim=True))[:, None, :]], 1)
    C3 = J3 @ S @ J3.transpose(1, 2)
    amp = rho * torch.sqrt(2 * math.pi * _inv3(C3)[1] / det2)
    co = torch.stack([n00 * xc ** 2 + 2 * n01 * xc * yc + n11 * yc ** 2, -2 * (n00 * xc + n01 * yc),
                      -2 * (n01 * xc + n11 * yc), n00, 2 * n01, n11, amp], 1)
    return co, box, alive


def _pieces(box, alive, limit=12_000_000):
    """The (Gaussian, pixel) pairs of the boxes in pieces: Gaussian numbers, their pair counts, i, j."""
    w, h = (box[:, 1] - box[:, 0] + 1).clamp_min(0), (box[:, 3] - box[:, 2] + 1).clamp_min(0)
    count = torch.where(alive, w * h, 0)
    keep = torch.nonzero(count).flatten()
    ends = torch.cumsum(count[keep], 0).cpu().numpy()
    at = 0
    while at < len(ends):
        base = ends[at - 1] if at else 0
        to = max(at + 1, int(np.searchsorted(ends, base + limit)))
        sel = keep[at:to]
        cnt = count[sel]
        own = torch.repeat_interleave(torch.arange(len(sel), device=box.device), cnt)
        first = torch.cumsum(cnt, 0) - cnt
        r = torch.arange(len(own), device=box.device) - first[own]
        ww = w[sel][own]
        yield sel, cnt, own, box[sel, 0][own] + r % ww, box[sel, 2][own] + r // ww
        at = to


def _values64(v, cone, co, own, i, j):
    """V of every pair (zero beyond the cutoff), and what its derivative needs."""
    g = co.t().contiguous()
    x, y = i.double(), j.double()
    q = [g[k][own] for k in range(6)]
    p = q[0] + x * (q[1] + x * q[3] + y * q[4]) + y * (q[2] + y * q[5])
    if not cone:
        V = torch.where(p <= CUTOFF ** 2, torch.exp(-0.5 * p), 0.0)
        return V * g[6][own], V, None, None, x, y
    b = g[6][own] + x * g[7][own] + y * g[8][own]
    s = b / p
    E = g[9][own] - b * s
    X, Y = (x - (v["nu"] - 1) / 2 + v["off_u"]) * v["du"], (y - (v["nv"] - 1) / 2 + v["off_v"]) * v["dv"]
    d2 = 1500.0 ** 2 + X ** 2 + Y ** 2
    V = torch.where(E <= CUTOFF ** 2, torch.sqrt(2 * math.pi * d2 / p) * torch.exp(-0.5 * E), 0.0)
    return V * g[10][own], V, p, s, x, y


def _render64(v, cone, co, box, alive):
    img = torch.zeros(v["nv"] * v["nu"], dtype=torch.float64, device="cuda")
    for sel, cnt, own, i, j in _pieces(box, alive):
        img.index_add_(0, j * v["nu"] + i, _values64(v, cone, co[sel], own, i, j)[0])
    return img.reshape(v["nv"], v["nu"])


def _coef_grad64(v, cone, co, box, alive, up):
    """dL/d(coefficients) for dL/dI = up."""
    out = torch.zeros_like(co)
    up = up.reshape(-1)
    for sel, cnt, own, i, j in _pieces(box, alive):
        full, V, p, s, x, y = _values64(v, cone, co[sel], own, i, j)
        g = up[j * v["nu"] + i]
        gV = g * full
        if cone:  # E = c - b^2 / p, V ~ p^-1/2 e^(-E/2)
            a = -0.5 * gV * (1.0 / p + s * s)
            b, last = gV * s, [-0.5 * gV, g * V]
        else:
            a, b, last = -0.5 * gV, None, [g * V]
        cols = [a, a * x, a * y, a * x * x, a * x * y, a * y * y] + ([b, b * x, b * y] if cone else []) + last
        end = torch.cumsum(cnt, 0) - 1
        for k, t in enumerate(cols):
            total = torch.cumsum(t, 0)[end]
            out[sel, k] = torch.diff(total, prepend=total.new_zeros(1))
    return out


def _project64(c, gauss, phi, w, views, up_of, need_grad=True):
    """Images of every view and, with dL/dI from up_of(image, number), the gradients of every input.

    phi: [scans][R]...; w: one row per view."""
    leaf = [t.double().requires_grad_() for t in (*gauss, phi, w)]
    mu0, scale, quat, rho, phi, w = leaf
    sizes = _scan_sizes(c)
    offs = np.concatenate([[0], np.cumsum(sizes)])
    lat = _lattice(c)
    imgs = [None] * len(views)
    ewa = c["model"] == "ewa"
    for s in range(len(sizes)):
        if not any(v["scan"] == s for v in views):
            continue
        at = slice(int(offs[s]), int(offs[s + 1]))
        U, dU = _ffd64(phi[s] if c["scans"] > 1 else phi, lat, mu0[at])
        Ul, dUl = U.detach().requires_grad_(), dU.detach().requires_grad_()
        for b, v in enumerate(views):
            if v["scan"] != s:
                continue
            mu, S, detK = _deformed64(mu0[at], scale[at], quat[at], Ul, dUl, w[b])
            co, box, alive = _coefs64(v, ewa, mu, S, rho[at])
            alive = alive & (detK > 1e-6)
            cone = not v["parallel"] and not ewa
            with torch.no_grad():
                cd = co.detach()
                imgs[b] = _render64(v, cone, cd, box, alive)
                if not need_grad:
                    continue
                gc = _coef_grad64(v, cone, cd, box, alive, up_of(imgs[b], b))
            co.backward(torch.where(alive[:, None], gc, 0.0))
        if need_grad:
            torch.autograd.backward([U, dU], [Ul.grad, dUl.grad])
    return torch.stack(imgs), [torch.zeros_like(t) if t.grad is None else t.grad for t in leaf]


def _adam64(kind, p, g, m, v, lr, it, beta1=0.9, beta2=0.999, eps=1e-15):
    if kind == 1:
        g = g * p
    elif kind == 2:
        g = g * -torch.expm1(-p)
    m, v = beta1 * m + (1 - beta1) * g, beta2 * v + (1 - beta2) * g * g
    step = lr * (m / (1 - beta1 ** it)) / ((v / (1 - beta2 ** it)).sqrt() + eps)
    if kind == 1:
        return p * torch.exp(-step)
    if kind == 2:
        return torch.log1p(torch.expm1(p) * torch.exp(-step))
    return p - step


def _exact_projector(case, seed):
    gauss, phi, w, views, ids, g = _scene(case, seed)
    k = case["kind"]
    at = torch.as_tensor(ids, device="cuda")
    if k in ("forward", "loss"):
        img, _ = _project64(case, gauss, phi, w[at], views, None, need_grad=False)
        if k == "forward":
            return img
        meas = _measured(case, views, g).double()
        return {"loss": ((img - meas) ** 2).mean().reshape(1), "proj": img}
    if k == "render":
        up = _randn(g, case["views"], case["nv"], case["nu"]).double()
        img, grads = _project64(case, gauss, phi, w[at], views, lambda i, b: up[b])
        return [img, *grads]
    total = 11 * case["n"] + phi.numel() + w.numel()
    m, v = (t.double() for t in _moments(case, total, g))
    meas = _measured(case, views, g).double()
    scale = 2.0 / meas.numel()
    img, grads = _project64(case, gauss, phi, w[at], views, lambda i, b: scale * (i - meas[b]))
    gw = torch.zeros_like(w, dtype=torch.float64).index_add_(0, at, grads[5])
    grads[5] = gw
    out = {"loss": ((img - meas) ** 2).mean().reshape(1), "grad": torch.cat([t.reshape(-1) for t in grads])}
    lr_at = min(AT_ITER / (TOTAL_ITERS - 1), 1.0)
    off = 0
    for q, (name, p, kind) in enumerate(zip(("mu0", "scale", "quat", "rho", "phi", "w"), (*gauss, phi, w), (0, 1, 0, 2, 0, 0))):
        n = p.numel()
        lr0, lr1 = float(np.float32(LR0[q])), float(np.float32(LR1 * LR0[q]))
        one = _adam64(kind, p.double().reshape(-1), grads[q].reshape(-1), m[off:off + n], v[off:off + n],
                      lr0 + (lr1 - lr0) * lr_at, AT_ITER + 1)
        out[name] = one.reshape(case["scans"], -1) if name == "phi" and case["scans"] > 1 else one.reshape(p.shape)
        off += n
    return out


def _exact_cnn(case, seed):
    img, cs, target, g = _pictures(case, seed)
    k = case["kind"]
    total = sum(math.prod(s) for s, _ in _net_layout(case["R"]))
    flat = _net_params(case, seed, total).double()
    x = img.double()
    if k == "cnn_predict":
        x = 0.25 * (x if case["edge"] == 128 else torch.nn.functional.avg_pool2d(x[:, None], 2)[:, 0])
    else:
        x = (img * 0.25).double()
    p, parts = flat.requires_grad_(k != "cnn_predict"), []
    off = 0
    for s, _ in _net_layout(case["R"]):
        parts.append(p[off:off + math.prod(s)].reshape(s))
        off += math.prod(s)

    def net(x, cs):
        x = x[:, None]
        for l in range(4):
            n, ci, e = x.shape[0], CNN_CHANNELS[l], CNN_EDGES[l + 1]
            col = torch.nn.functional.unfold(x, 3, padding=1, stride=2)  # [n][ci 9][e e]
            wt = parts[2 * l].permute(0, 3, 1, 2).reshape(CNN_CHANNELS[l + 1], ci * 9)
            x = torch.relu((wt @ col).reshape(n, -1, e, e) + parts[2 * l + 1][None, :, None, None])
        f = torch.cat([x.permute(0, 2, 3, 1).reshape(x.shape[0], -1), cs], 1)
        return torch.relu(f @ parts[8].t() + parts[9]) @ parts[10].t() + parts[11]

    if k == "cnn_predict":
        with torch.no_grad():
            return torch.cat([net(x[s:s + 64], cs[s:s + 64].double()) for s in range(0, x.shape[0], 64)])
    outs, grad = [], torch.zeros_like(flat)
    B = case["batch"]
    for s in range(0, B, 64):
        o = net(x[s:s + 64], cs[s:s + 64].double())
        t = target[s:s + 64].double()
        up = 2.0 / (B * case["R"]) * ((o.detach() - t) if k == "cnn_train" else t)
        grad += torch.autograd.grad(o, p, up, retain_graph=True)[0]
        outs.append(o.detach())
    out = torch.cat(outs)
    if k == "cnn_fp32":
        return {"out": out, "grad": grad}
    m, v = (t.double() for t in _moments(case, total, g))
    new = _adam64(0, flat.detach(), grad, 1e3 * m, 1e6 * v, 3e-4, 401, eps=1e-8)
    return {"loss": ((out - target.double()) ** 2).mean().reshape(1), "grad": grad, "params": new}


def _exact_volume(case, seed):
    c = dict(case, scans=1, views=1)
    g = _gen(seed)
    mu0, scale, quat, rho = (t.double() for t in _cloud(c, c["n"], g))
    phi, w = _motion(c, 16, g)
    phi, w = phi.double(), w[5].double()
    lat, grid = _lattice(c), _grid(c)
    U, dU = _ffd64(phi, lat, mu0)
    mu, S, detK = _deformed64(mu0, scale, quat, U, dU, w)
    P = _inv3(S)[0]
    dims = torch.tensor([grid["nx"], grid["ny"], grid["nz"]], device="cuda")
    h, o = (torch.tensor(np.float32(grid[k]).astype(np.float64), device="cuda") for k in ("spacing", "origin"))
    half = CUTOFF * torch.diagonal(S, dim1=1, dim2=2).sqrt() + 1e-6
    lo = torch.maximum(((mu - half - o) / h).ceil().long(), torch.zeros_like(dims))
    hi = torch.minimum(((mu + half - o) / h).floor().long(), dims - 1)
    ext = (hi - lo + 1).clamp_min(0)
    count = torch.where(detK > 1e-6, ext.prod(1), 0)
    vol = torch.zeros(int(dims.prod()), dtype=torch.float64, device="cuda")
    n, at = c["n"], 0
    ends = torch.cumsum(count, 0).cpu().numpy()
    while at < n:
        base = ends[at - 1] if at else 0
        to = max(at + 1, int(np.searchsorted(ends, base + 12_000_000)))
        own = torch.repeat_interleave(torch.arange(at, to, device="cuda"), count[at:to])
        first = torch.cumsum(count[at:to], 0) - count[at:to]
        r = torch.arange(len(own), device="cuda") - first[own - at]
        ex, ey = ext[own, 0], ext[own, 1]
        i, j, k = lo[own, 0] + r % ex, lo[own, 1] + (r // ex) % ey, lo[own, 2] + r // (ex * ey)
        d = torch.stack([i, j, k], 1) * h + o - mu[own]
        E = ((P[own] @ d[:, :, None])[:, :, 0] * d).sum(1)
        vol.index_add_(0, (k * dims[1] + j) * dims[0] + i, torch.where(E <= CUTOFF ** 2, rho[own] * torch.exp(-0.5 * E), 0.0))
        at = to
    vol = vol.reshape(grid["nz"], grid["ny"], grid["nx"])
    k, j, i = torch.meshgrid(*(torch.arange(grid[a], device="cuda", dtype=torch.float64) for a in ("nz", "ny", "nx")), indexing="ij")
    pts = torch.stack([i, j, k], -1).reshape(-1, 3) * h + o
    field = torch.cat([torch.einsum("r,nri->ni", w, _ffd64(phi, lat, q, jacobian=False)[0]) for q in pts.split(1 << 19)])
    return {"volume": vol, "dvf": field.reshape(*vol.shape, 3)}


def exact(case, seed):
    if case["kind"].startswith("cnn"):
        return _exact_cnn(case, seed)
    if case["kind"] == "volume":
        return _exact_volume(case, seed)
    return _exact_projector(case, seed)
