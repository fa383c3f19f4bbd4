"""What is timed of this library: the calls its users make, over the sizes
they make them at.

A case names one public entry point and its sizes.  `prepare` builds what a
program holds before that call (a resident scene, cameras, masks on the
device, a captured solve, a server), `run` makes the call, `work` gives the
bytes and operations the call cannot do without, `exact` evaluates it in FP64
with plain torch where that is affordable.

Scenes and masks follow the distributions of the package's own generators
(clustered Gaussians, log-normal scales, sigmoid-normal opacities, silhouettes
of the clusters with noisy labels), made on the GPU so that a state takes a
second or less.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2409_08270_gb300 import flashsplat as fs
from paper_2409_08270_gb300 import synth

DEV = "cuda"

# n: Gaussians; views of w x h pixels; E: labels, background included;
# orbit: cameras around the scene (else a forward-facing arc)
_SOLVE = {"call": "solve", "orbit": False, "mask": "uint8", "gamma": 0.5, "form": "f32",
          "coverage": 0}


def listed():
    return [
        # the smallest solve: a toy scene, a test, an interactive preview
        dict(_SOLVE, name="solve tiny", n=2000, views=8, w=128, h=128, E=2),
        # one object of a forward-facing capture: the benchmark's workload
        dict(_SOLVE, name="solve binary", n=1_000_000, views=100, w=1008, h=756, E=2),
        # every instance of a 360-degree capture at once (the benchmark's
        # multi-instance workload with half its views)
        dict(_SOLVE, name="solve multi", n=3_000_000, views=100, w=1256, h=828, E=33,
             orbit=True, mask="int32"),
        # a scene stored as BF16/FP16 and solved with reduced-precision records
        dict(_SOLVE, name="solve reduced", n=1_000_000, views=48, w=1008, h=756, E=2,
             form="reduced"),
        # a mid-size scene trained with the standard rasteriser: its 3-sigma
        # tile coverage is asked for
        dict(_SOLVE, name="solve 3sigma", n=333_333, views=37, w=799, h=601, E=12, orbit=True,
             coverage=1),
        # the same scene solved again and again for new masks: one CUDA graph
        dict(_SOLVE, name="replay", call="replay", n=500_000, views=50, w=1008, h=756, E=5,
             orbit=True),
        # a solve resumed view by view: one new full-size view into the table
        dict(_SOLVE, name="accumulate view", call="accumulate", n=300_000, views=1, w=1600,
             h=1200, E=2),
        # the decision alone, for a new background bias, from a resident table
        {"name": "assign", "call": "assign", "n": 3_000_000, "E": 33, "table": "float32",
         "gamma": 0.5},
        # the Gaussians left after objects are removed
        {"name": "removal", "call": "remove", "n": 3_000_000, "E": 33},
        # masks of a segmentation in views that have none
        dict(_SOLVE, name="novel masks", call="render", n=500_000, views=8, w=1008, h=756, E=9,
             orbit=True, planes=False),
        # a small scene inside a program that may not allocate
        dict(_SOLVE, name="solve noalloc", call="noalloc", n=12_000, views=4, w=384, h=384, E=2),
        # four requests in flight on the request server, masks in host memory
        dict(_SOLVE, name="serve", call="serve", n=300_000, views=24, w=512, h=512, E=7,
             orbit=True, requests=4),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case of the same calls and ranges; no drawn case holds more
    (view, Gaussian) slots or more pixels than the largest listed one."""
    call = rng.choice(["solve", "solve", "solve", "solve", "replay", "accumulate", "assign",
                       "remove", "render", "noalloc", "serve"])
    if call in ("assign", "remove"):
        case = {"call": call, "n": _log(rng, 20_000, 3_000_000), "E": _log(rng, 2, 33)}
        if call == "assign":
            case["table"] = rng.choice(["float32", "float64"])
            case["gamma"] = rng.choice([-0.4, 0.0, 0.5])
        return case
    c = dict(_SOLVE, call=call)
    c["orbit"] = rng.random() < 0.5
    c["E"] = _log(rng, 2, 33)
    c["mask"] = rng.choice(["uint8", "int32"])
    c["gamma"] = rng.choice([-0.4, 0.0, 0.5])
    c["w"], c["h"] = _log(rng, 120, 1600), _log(rng, 100, 1200)
    c["n"] = _log(rng, 2000, 1_500_000)
    if call == "solve":
        c["views"] = min(_log(rng, 2, 100), max(2, 75_000_000 // (c["w"] * c["h"])))
        c["form"] = "reduced" if rng.random() < 0.25 else "f32"
        c["coverage"] = 1 if rng.random() < 0.25 else 0
    elif call == "replay":
        c["n"], c["views"] = min(c["n"], 600_000), _log(rng, 2, 50)
    elif call == "accumulate":
        c["views"] = _log(rng, 1, 8)
    elif call == "render":
        c["n"], c["views"], c["E"] = min(c["n"], 600_000), _log(rng, 1, 8), min(c["E"], 9)
        c["planes"] = rng.random() < 0.5
    elif call == "noalloc":
        c["n"], c["views"] = _log(rng, 500, 16_000), _log(rng, 1, 8)
        c["w"], c["h"] = _log(rng, 64, 512), _log(rng, 64, 512)
    else:
        c["n"], c["views"], c["requests"] = min(c["n"], 400_000), _log(rng, 4, 32), 4
        c["w"], c["h"] = min(c["w"], 800), min(c["h"], 600)
    return c


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------

def _generator(seed, salt):
    g = torch.Generator(device=DEV)
    g.manual_seed((int(seed) * 1_000_003 + salt) % (1 << 62))
    return g


def _rotations(q):
    w, x, y, z = (q / q.norm(dim=1, keepdim=True)).unbind(1)
    return torch.stack([
        torch.stack([1 - 2 * (y * y + z * z), 2 * (x * y - w * z), 2 * (x * z + w * y)], 1),
        torch.stack([2 * (x * y + w * z), 1 - 2 * (x * x + z * z), 2 * (y * z - w * x)], 1),
        torch.stack([2 * (x * z - w * y), 2 * (y * z + w * x), 1 - 2 * (x * x + y * y)], 1)], 1)


def _scene(case, seed):
    """Gaussians (mean, quat, scale, opacity: FP32 on the device) in clusters,
    and the clusters' 2-sigma ellipsoids (centre, rotation, radii)."""
    g = _generator(seed, 1)
    n = case["n"]
    small = n <= 20_000  # toy scenes: fewer clusters and larger Gaussians
    k = 6 if small else 32 if case["orbit"] else 20
    half = torch.tensor([1.5, 1.5, 1.5] if case["orbit"] else [1.0, 1.0, 0.5], device=DEV)

    def uniform(*shape):
        return torch.rand(shape, generator=g, device=DEV)

    def normal(*shape):
        return torch.randn(shape, generator=g, device=DEV)

    centre = (2 * uniform(k, 3) - 1) * half
    rot, std = _rotations(normal(k, 4)), 0.05 + 0.25 * uniform(k, 3)
    edges = torch.cumsum(0.5 + uniform(k), 0)
    cl = torch.searchsorted(edges / edges[-1], (torch.arange(n, device=DEV) + 0.5) / n)
    cl = cl.clamp_(max=k - 1)
    mean = centre[cl] + torch.einsum("nij,nj->ni", rot[cl], normal(n, 3) * std[cl])
    quat = normal(n, 4)
    mu, sd = (-3.0, 0.5) if small else (-4.0, 1.0)
    gauss = {"mean": mean.contiguous(),
             "quat": (quat / quat.norm(dim=1, keepdim=True)).contiguous(),
             "scale": torch.exp(mu + sd * normal(n, 3)),
             "opacity": torch.sigmoid(1.5 * normal(n))}
    if case["form"] == "reduced":
        gauss["quat"] = gauss["quat"].to(torch.bfloat16)
        gauss["scale"] = gauss["scale"].to(torch.bfloat16)
        gauss["opacity"] = gauss["opacity"].to(torch.float16)
    return gauss, (centre, rot, 2.0 * std)


def _cameras(case, seed):
    rng = np.random.default_rng([int(seed), 2])
    w, h, v = case["w"], case["h"], case["views"]
    fx = synth.fx_from_hfov(w, 60.0)
    cams = []
    for i in range(v):
        if case["orbit"]:
            el = math.radians(15.0 if 2 * i < v else 40.0)
            az = 2 * math.pi * (i + rng.uniform(-0.2, 0.2)) / max(1, v // 2)
            p = (5 * math.cos(el) * math.sin(az), 5 * math.sin(el),
                 -5 * math.cos(el) * math.cos(az))
        else:
            az = math.radians(rng.uniform(-30.0, 30.0))
            p = (4 * math.sin(az), 0.0, -4 * math.cos(az))
        cams.append(synth.camera(p, w, h, fx))
    return cams


def _masks(case, cams, ellipsoids, seed):
    """Per view the nearest cluster's label at each pixel (0: background).
    E = 2: one cluster is the object and 4.5 % of the pixels are flipped;
    else the clusters are grouped into E - 1 labels and 3 % of the pixels take
    a neighbour's label."""
    g = _generator(seed, 3)
    centre, rot, rad = (t.double() for t in ellipsoids)
    E, k = case["E"], centre.shape[0]
    if E == 2:
        lab_of = torch.zeros(k, dtype=torch.int64, device=DEV)
        lab_of[torch.argmin(centre.norm(dim=1))] = 1
    else:
        lab_of = 1 + torch.arange(k, device=DEV) % (E - 1)
    w, h = case["w"], case["h"]
    dtype = torch.uint8 if case["mask"] == "uint8" else torch.int32
    inv = rot.transpose(1, 2) / rad[:, :, None]
    masks = []
    for c in cams:
        R = torch.as_tensor(np.asarray(c["R"]), device=DEV)
        o = -(R.T @ torch.as_tensor(np.asarray(c["t"]), device=DEV))
        M = (inv @ R.T).float()
        o2 = torch.einsum("kij,kj->ki", inv, o[None] - centre).float()
        u = (torch.arange(w, device=DEV) + 0.5 - c["cx"]) / c["fx"]
        v = (torch.arange(h, device=DEV) + 0.5 - c["cy"]) / c["fy"]
        d = (M[:, :, 0, None, None] * u + M[:, :, 1, None, None] * v[:, None]
             + M[:, :, 2, None, None])
        a = d.square().sum(1)
        b = (d * o2[:, :, None, None]).sum(1)
        disc = b * b - a * (o2.square().sum(1) - 1)[:, None, None]
        s = torch.where(disc >= 0, (-b - disc.clamp(min=0).sqrt()) / a, math.inf)
        best, who = torch.where(s > 0, s, math.inf).min(0)
        lab = torch.where(torch.isfinite(best), lab_of[who], 0)
        noise = torch.rand((h, w), generator=g, device=DEV)
        if E == 2:
            lab = torch.where(noise < 0.045, 1 - lab, lab)
        else:
            lab = torch.where(noise < 0.015, lab.roll(1, 1), lab)
            lab = torch.where(noise > 0.985, lab.roll(1, 0), lab)
        masks.append(lab.to(dtype).contiguous())
    return masks


def _inputs(case, seed):
    gauss, ell = _scene(case, seed)
    cams = _cameras(case, seed)
    return gauss, cams, _masks(case, cams, ell, seed), ell


def _membership(case, seed):
    """Membership bits of a segmentation: mostly one label, some none or two
    (how many of each does not depend on the seed, who they are does)."""
    n, E = case["n"], case["E"]
    at = torch.arange(n, device=DEV)
    one = torch.ones((), dtype=torch.int64, device=DEV)
    bits = torch.where(at * 10 < n, 0, one << (at % E))
    bits = torch.where(at * 20 > 19 * n, bits | (one << ((at + 1) % E)), bits)
    return bits[torch.randperm(n, generator=_generator(seed, 4), device=DEV)].contiguous()


def _table(case, seed):
    """A contribution table: most of a Gaussian's weight in one label, noise in
    the others, some Gaussians never seen."""
    g = _generator(seed, 5)
    n, E = case["n"], case["E"]
    t = torch.rand((n, E), generator=g, device=DEV).pow_(4)
    main = torch.randint(0, E, (n, 1), generator=g, device=DEV)
    t.scatter_add_(1, main, 8 * torch.rand((n, 1), generator=g, device=DEV))
    t *= torch.exp(2 * torch.randn((n, 1), generator=g, device=DEV))
    t[torch.rand(n, generator=g, device=DEV) < 0.05] = 0
    return t.to(torch.float64 if case["table"] == "float64" else torch.float32)


def _solver(case, gauss):
    return fs.Solver(gauss, record_precision=fs.FS_F16 if case["form"] == "reduced" else 0,
                     coverage=case["coverage"])


def prepare(case, seed):
    call = case["call"]
    s = {"case": case, "call": call}
    if call == "assign":
        one = torch.ones(1, device=DEV)
        s["solver"] = fs.Solver({"mean": one.expand(1, 3), "quat": one.expand(1, 4),
                                 "scale": one.expand(1, 3), "opacity": one})
        s["table"] = _table(case, seed)
        return s
    if call == "remove":
        one = torch.ones(1, device=DEV)
        s["solver"] = fs.Solver({"mean": one.expand(1, 3), "quat": one.expand(1, 4),
                                 "scale": one.expand(1, 3), "opacity": one})
        s["bits"] = _membership(case, seed)
        s["labels"] = list(range(1, case["E"], 3))
        return s
    if call == "render":
        gauss, ell = _scene(case, seed)
        s["cams"] = _cameras(case, seed)
        s["solver"] = _solver(case, gauss)
        s["bits"] = _objects(case, gauss, ell, seed)
        return s
    gauss, s["cams"], s["masks"], _ = _inputs(case, seed)
    if call == "serve":
        host = {k: v.float().cpu().numpy() for k, v in gauss.items()}
        s["server"] = fs.Server(slots=4)
        s["scene"] = s["server"].add_scene(host)
        base = [m.cpu().numpy() for m in s.pop("masks")]
        s["requests"] = [[np.roll(m, (3 * r, 5 * r), (0, 1)) for m in base]
                         for r in range(case["requests"])]
    elif call == "noalloc":
        s["gauss"] = gauss
        s["g"] = fs.fs_gaussians(n=case["n"], mean=gauss["mean"].data_ptr(),
                                 quat=gauss["quat"].data_ptr(), scale=gauss["scale"].data_ptr(),
                                 opacity=gauss["opacity"].data_ptr(), quat_dtype=fs.FS_F32,
                                 scale_dtype=fs.FS_F32, opacity_dtype=fs.FS_F32,
                                 memory=fs.FS_MEM_DEVICE)
        s["fs_cams"] = fs.make_cameras(s["cams"])
        n, E = case["n"], case["E"]
        s["out"] = {"table": torch.empty((n, E), device=DEV),
                    "bits": torch.empty(n, dtype=torch.int64, device=DEV),
                    "label": torch.empty(n, dtype=torch.int32, device=DEV),
                    "margin": torch.empty(n, device=DEV)}
    else:
        s["solver"] = _solver(case, gauss)
        if call == "replay":
            s["graph"] = s["solver"].capture(s["cams"], s["masks"], case["E"], case["gamma"])
    return s


def _objects(case, gauss, ell, seed):
    """Membership as a segmentation leaves it: each cluster's Gaussians belong
    to one object, a few to none."""
    g = _generator(seed, 6)
    centre = ell[0]
    near = torch.cat([(m[:, None] - centre).square().sum(2).argmin(1)
                      for m in gauss["mean"].split(100_000)])
    lab = near % case["E"]  # label 0: background
    out = torch.ones((), dtype=torch.int64, device=DEV) << lab
    keep = torch.rand(case["n"], generator=g, device=DEV) > 0.03
    return torch.where(keep, out, 0).contiguous()


def run(state):
    s, case, call = state, state["case"], state["call"]
    if call == "solve":
        r = s["solver"].solve(s["cams"], s["masks"], case["E"], case["gamma"])
        return {k: r[k] for k in ("table", "bits", "label", "margin")}
    if call == "replay":
        s["graph"].launch()
        s["graph"].synchronize()
        return s["graph"].outputs
    if call == "accumulate":
        table = torch.zeros((case["n"], case["E"]), device=DEV)
        s["solver"].accumulate(s["cams"], s["masks"], case["E"], table)
        return table
    if call == "assign":
        return s["solver"].assign(s["table"], case["gamma"])
    if call == "remove":
        return s["solver"].keep_after_removal(s["bits"], s["labels"])
    if call == "render":
        return s["solver"].render_masks(s["cams"], s["bits"], case["E"],
                                        want_planes=case["planes"])
    if call == "noalloc":
        o, m = s["out"], s["masks"]
        fs.fs_solve_noalloc(0, s["g"], s["fs_cams"], [x.data_ptr() for x in m],
                            fs.FS_U8 if case["mask"] == "uint8" else fs.FS_I32, case["E"],
                            case["gamma"], o["table"].data_ptr(), o["bits"].data_ptr(),
                            o["label"].data_ptr(), o["margin"].data_ptr(),
                            torch.cuda.current_stream().cuda_stream)
        return o
    srv = s["server"]
    tickets = [srv.submit(s["scene"], s["cams"], m, case["E"], case["gamma"])
               for m in s["requests"]]
    done = [srv.fetch(t) for t in tickets]
    return [{"bits": d["bits"].view(np.int64), "label": d["label"], "margin": d["margin"]}
            for d in done]


# (pixel, Gaussian) pairs that take part in the compositing of a pixel: about
# 70 per pixel on the benchmark's binary workload (counted there); 19 FP32
# operations each.  The projection of a Gaussian into a view: about 300.
PAIRS_PER_PIXEL, PAIR_FLOPS, PROJECT_FLOPS = 70.0, 19.0, 300.0


def work(case):
    n, E, call = case["n"], case["E"], case["call"]
    if call == "assign":
        size = 8 if case["table"] == "float64" else 4
        return {"bytes": n * (E * size + 16), "flops": n * E * 6.0}
    if call == "remove":
        return {"bytes": n * (8 + 4), "flops": float(n)}
    pixels = case["views"] * case["w"] * case["h"]
    scene = n * (24 if case["form"] == "reduced" else 44)
    flops = case["views"] * n * PROJECT_FLOPS + pixels * PAIRS_PER_PIXEL * PAIR_FLOPS
    mask = pixels * (1 if case["mask"] == "uint8" else 4)
    if call == "render":
        planes = pixels * (case["E"] - 1) * 8 if case["planes"] else 0
        return {"bytes": scene + 8 * n + pixels + planes, "flops": flops}
    times = case.get("requests", 1)
    out = n * E * 4 if call == "accumulate" else n * 16 if call == "serve" else n * (E * 4 + 16)
    return {"bytes": times * (scene + mask + out), "flops": times * flops}


# ---------------------------------------------------------------------------
# FP64 evaluation with plain torch
# ---------------------------------------------------------------------------

def exact(case, seed):
    call = case["call"]
    if call == "assign":
        margin = _margin(_table(case, seed).double(), case["gamma"])
        return (None, None, margin)
    if call == "remove":
        return None
    slots, pixels = case["n"] * case["views"], case["views"] * case["w"] * case["h"]
    if case["form"] == "reduced" or case["coverage"] or slots > 400_000 or pixels > 2_500_000:
        return None
    if call == "render":
        gauss, ell = _scene(case, seed)
        cams, bits = _cameras(case, seed), _objects(case, gauss, ell, seed)
        if not case["planes"]:
            return None
        out = {"masks": [None] * len(cams), "rho": [], "depth": []}
        for c in cams:
            planes = [_composite(gauss, c, keep=(bits >> e) & 1 == 1) for e in range(1, case["E"])]
            out["rho"].append(torch.stack([p[0] for p in planes]))
            out["depth"].append(torch.stack([p[1] for p in planes]))
        return out
    gauss, cams, masks, _ = _inputs(case, seed)

    def solved(labels):
        table = torch.zeros((case["n"], case["E"]), dtype=torch.float64, device=DEV)
        for c, m in zip(cams, labels):
            _composite(gauss, c, mask=m, table=table)
        return table

    if call == "serve":
        out = []
        for r in range(case["requests"]):
            t = solved([m.roll((3 * r, 5 * r), (0, 1)) for m in masks])
            out.append({"bits": None, "label": None, "margin": _margin(t, case["gamma"])})
        return out
    table = solved(masks)
    if call == "accumulate":
        return table
    return {"table": table, "bits": None, "label": None, "margin": _margin(table, case["gamma"])}


def _margin(table, gamma):
    """min over labels of |(1 - g) A - (1 + g) (S - A)| / S; +inf unseen."""
    gamma = float(np.float32(gamma))
    S = table.sum(1, keepdim=True)
    m = ((1 - gamma) * table - (1 + gamma) * (S - table)).abs() / S
    return torch.where(S[:, 0] > 0, m.min(1).values, math.inf)


def _composite(gauss, cam, mask=None, table=None, keep=None):
    """One view composited front to back in FP64 over 16x16 tiles.  With a
    mask: alpha T is added to table[Gaussian, label].  Without: the sum of
    alpha T and the alpha T-weighted mean depth per pixel."""
    W, H = cam["width"], cam["height"]
    R = torch.as_tensor(np.asarray(cam["R"]), device=DEV)
    t = torch.as_tensor(np.asarray(cam["t"]), device=DEV)
    o = gauss["opacity"].double()
    p = gauss["mean"].double() @ R.T + t
    use = (p[:, 2] > 0.2) & (gauss["opacity"] >= np.float32(1 / 255))
    if keep is not None:
        use &= keep
    idx = use.nonzero()[:, 0]
    idx = idx[torch.argsort(p[idx, 2], stable=True)]  # depth order, ties by index
    p, o = p[idx], o[idx]
    A = _rotations(gauss["quat"][idx].double()) * gauss["scale"][idx].double()[:, None, :]
    x, y, z = p.unbind(1)
    fx, fy = cam["fx"], cam["fy"]
    ux, uy = x / z, y / z
    mx, my = fx * ux + cam["cx"], fy * uy + cam["cy"]
    lx, ly = 1.3 * 0.5 * W / fx, 1.3 * 0.5 * H / fy
    J0 = (fx / z)[:, None] * (R[0] - ux.clamp(-lx, lx)[:, None] * R[2])
    J1 = (fy / z)[:, None] * (R[1] - uy.clamp(-ly, ly)[:, None] * R[2])
    v0 = torch.einsum("ni,nij->nj", J0, A)
    v1 = torch.einsum("ni,nij->nj", J1, A)
    sxx, sxy, syy = v0.square().sum(1) + 0.3, (v0 * v1).sum(1), v1.square().sum(1) + 0.3
    det = sxx * syy - sxy * sxy
    r2 = 2 * torch.log(255 * o).clamp(min=0)
    hx, hy = torch.sqrt(sxx * r2) + 1, torch.sqrt(syy * r2) + 1
    nx, ny = (W + 15) // 16, (H + 15) // 16

    def span(m, half, size, tiles):
        a = torch.floor((m - half) / 16).clamp(0, tiles).long()
        b = torch.floor((m + half) / 16).clamp(-1, tiles - 1).long()
        return a, torch.where((m + half >= 0) & (m - half <= size), b, -1)

    x0, x1 = span(mx, hx, W, nx)
    y0, y1 = span(my, hy, H, ny)
    cols, rows = (x1 - x0 + 1).clamp(min=0), (y1 - y0 + 1).clamp(min=0)
    count = cols * rows
    owner = torch.repeat_interleave(torch.arange(len(idx), device=DEV), count)
    local = torch.arange(len(owner), device=DEV) - (torch.cumsum(count, 0) - count)[owner]
    tile = (y0[owner] + local // cols[owner]) * nx + x0[owner] + local % cols[owner]
    order = torch.argsort(tile, stable=True)
    owner, tile = owner[order], tile[order]
    length = torch.bincount(tile, minlength=nx * ny)
    start = torch.cumsum(length, 0) - length
    rho = torch.zeros((ny * 16, nx * 16), dtype=torch.float64, device=DEV)
    zsum = torch.zeros_like(rho)
    pix = torch.arange(256, device=DEV)
    todo, lens = torch.argsort(length), length.sort().values.tolist()
    k = 0
    while k < len(lens):
        if lens[k] == 0:
            k += 1
            continue
        e = k + 1  # tiles of similar length together, some 24 million pairs at a time
        while e < len(lens) and (e + 1 - k) * lens[e] * 256 <= 24_000_000:
            e += 1
        tl = todo[k:e]
        L = lens[e - 1]
        j = torch.arange(L, device=DEV)
        on = j < length[tl][:, None]
        g = owner[torch.where(on, start[tl][:, None] + j, 0)]
        px = ((tl % nx) * 16)[:, None] + pix % 16
        py = ((tl // nx) * 16)[:, None] + pix // 16
        dx = px[:, None, :] + 0.5 - mx[g][:, :, None]
        dy = py[:, None, :] + 0.5 - my[g][:, :, None]
        q = (syy[g][:, :, None] * dx * dx - 2 * sxy[g][:, :, None] * dx * dy
             + sxx[g][:, :, None] * dy * dy) / det[g][:, :, None]
        a = (o[g][:, :, None] * torch.exp(-0.5 * q)).clamp(max=0.99)
        a = torch.where((a >= 1 / 255) & on[:, :, None], a, 0.0)
        after = torch.cumprod(1 - a, 1)
        before = torch.cat([torch.ones_like(after[:, :1]), after[:, :-1]], 1)
        c = torch.where(after >= 1e-4, a * before, 0.0)
        if mask is not None:
            inside = (px < W) & (py < H)
            lab = mask.long()[py.clamp(max=H - 1), px.clamp(max=W - 1)]
            hot = torch.nn.functional.one_hot(lab, table.shape[1]).double() * inside[:, :, None]
            rows_ = torch.bmm(c, hot)
            table.index_add_(0, idx[g].reshape(-1), rows_.reshape(-1, table.shape[1]))
        else:
            rho[py, px] = c.sum(1)
            zsum[py, px] = (c * z[g][:, :, None]).sum(1)
        k = e
    if mask is None:
        rho, zsum = rho[:H, :W], zsum[:H, :W]
        return rho, torch.where(rho > 0, zsum / rho, 0.0)
    return table
