"""The workloads that the library's speed is measured on.

Each case is one call (or one training step) through the public entry points
of ``paper_2606_00817_gb300.ddf``, on inputs made on the GPU from a seed:

  rays      ``DDF.query``: t and visibility of a batch of rays
  noalloc   ``ddf_query_rays_noalloc``: the allocation-free query
  shadow    ``DDF.shadow``: t, visibility and the shadow decision
  ao        ``ddf_query_ao``: a ragged ambient-occlusion batch, graph mode
  hashgrid  ``DDF.shadow`` on the hash-grid field
  hg_train  ``ddf_train_step`` on the hash-grid field (forward, backward, Adam)
  train     ``ddf_train_step`` on a sinusoidal field
  trace     ``ddf_sphere_trace`` through an SDF field
  gs        ``ddf_render_gs_depth``: depth images of 3D Gaussians

The networks are random: Xavier weights for the ray fields (as
``inputs.xavier_blob``), tables uniform in +-1 for the hash grid, and for the
SDF field weights that approximate the distance to a bumpy sphere, so that a
trace takes the steps a trained field takes. Rays start on the surfaces of a
random sphere scene or, for plain queries, anywhere in the box.
"""
import math

import numpy as np
import torch

from paper_2606_00817_gb300 import ddf
from paper_2606_00817_gb300 import inputs as I

DEV = "cuda:0"
LIGHT = (3.0, 3.0, 3.0)
WIDE = {"octaves": 10, "width": 1280, "hidden": 8}    # the paper-sized field (11.6 M weights)
SMALL = {"octaves": 6, "width": 128, "hidden": 4}     # the small field of the tests
SDF = {"octaves": 8, "width": 512, "hidden": 6}       # the supervision study's neural surface
EPS, T_MAX, MAX_STEPS = 1e-3, 4.0, 128
GAUSSIANS, VIEW = 60000, 128


def listed():
    return [
        # the smallest call: the rays under a cursor or a probe's few directions
        {"name": "pick", "kind": "rays", **WIDE, "precision": "bf16", "tuned": False, "n": 193},
        # a renderer's per-frame callback, which may not allocate: a 64 x 64 tile and a few more
        {"name": "callback", "kind": "noalloc", **WIDE, "precision": "bf16", "tuned": False,
         "n": 4099},
        # the small field, one batch as a training loop validates it
        {"name": "small field", "kind": "rays", **SMALL, "precision": "bf16", "tuned": False,
         "n": 16384},
        # the headline: shadow rays of a 2048 x 2048 image, with the tiles the autotuner picks
        {"name": "shadow frame", "kind": "shadow", **WIDE, "precision": "bf16", "tuned": True,
         "n": 4194304},
        # ambient occlusion of a 64 x 64 tile of shading points, 4 to 64 rays each, e4m3 weights,
        # no tuning: what a program gets that only loads its field
        {"name": "ambient occlusion", "kind": "ao", **WIDE, "precision": "fp8", "tuned": False,
         "points": 4096},
        # full precision: a reference image's rays
        {"name": "fp32 rays", "kind": "rays", **WIDE, "precision": "fp32", "tuned": False,
         "n": 16387},
        # the paper's final field: the shadow rays of a 1024 x 1024 image
        {"name": "hash grid shadow", "kind": "hashgrid", "hidden": 2, "precision": "bf16",
         "n": 1048576},
        # the same field in full precision, a ragged batch
        {"name": "hash grid fp32", "kind": "hashgrid", "hidden": 2, "precision": "fp32",
         "n": 100003},
        # a step of the paper's distillation schedule: batch 16,384, 30,000 of them a scene
        {"name": "hash grid step", "kind": "hg_train", "hidden": 2, "batch": 16384},
        # a distillation step of the paper-sized field
        {"name": "wide field step", "kind": "train", **WIDE, "batch": 65536},
        # the sphere-traced baseline on the camera rays of a 256 x 256 view
        {"name": "sphere trace", "kind": "trace", **SDF, "n": 65536},
        # supervision depth: views of a splatting scene
        {"name": "gaussian depth", "kind": "gs", "views": 32, "size": VIEW},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["rays", "rays", "noalloc", "shadow", "ao", "fp32", "hashgrid", "hashgrid",
                       "hg_train", "train", "trace", "gs"])
    if kind == "rays":
        net = rng.choice([WIDE, SMALL, SMALL, {"octaves": 8, "width": 256, "hidden": 3}])
        return {"kind": "rays", **net, "precision": "bf16", "tuned": False,
                "n": _log(rng, 1, 300000)}
    if kind == "noalloc":
        net = rng.choice([WIDE, SMALL])
        return {"kind": "noalloc", **net, "precision": "bf16", "tuned": False,
                "n": _log(rng, 16, 6000)}
    if kind == "shadow":
        return {"kind": "shadow", **WIDE, "precision": rng.choice(["bf16", "fp8"]), "tuned": True,
                "n": _log(rng, 30000, 2000000)}
    if kind == "ao":
        return {"kind": "ao", **WIDE, "precision": rng.choice(["bf16", "fp8"]),
                "tuned": rng.random() < 0.3, "points": _log(rng, 64, 16384)}
    if kind == "fp32":
        net = rng.choice([WIDE, SMALL, {"octaves": 8, "width": 200, "hidden": 3}])
        return {"kind": "rays", **net, "precision": "fp32", "tuned": False,
                "n": _log(rng, 64, 60000)}
    if kind == "hashgrid":
        return {"kind": "hashgrid", "hidden": rng.choice([1, 2, 2, 3]),
                "precision": rng.choice(["bf16", "bf16", "fp32"]), "n": _log(rng, 256, 3000000)}
    if kind == "hg_train":
        return {"kind": "hg_train", "hidden": rng.choice([2, 2, 3]),
                "batch": 8 * _log(rng, 64, 8192)}
    if kind == "train":
        return {"kind": "train", **rng.choice([WIDE, WIDE, SMALL]),
                "batch": 8 * _log(rng, 128, 8192)}
    if kind == "trace":
        return {"kind": "trace", **SDF, "n": _log(rng, 300, 150000)}
    return {"kind": "gs", "views": _log(rng, 1, 64), "size": rng.choice([96, 100, VIEW, 200])}


# ------------------------------------------------------------------- inputs

def _gen(seed, stream):
    g = torch.Generator(device=DEV)
    g.manual_seed((seed * 1000003 + stream) & 0x7FFFFFFFFFFFFFFF)
    return g


def _u(g, *shape, lo=0.0, hi=1.0, dtype=torch.float64):
    return lo + (hi - lo) * torch.rand(*shape, generator=g, device=DEV, dtype=dtype)


def _unit(g, n):
    d = torch.randn(n, 3, generator=g, device=DEV, dtype=torch.float64)
    return d / d.norm(dim=1, keepdim=True).clamp_min(1e-12)


def _xavier(dims, g):
    """Float32 blob (on the GPU) of (fan_out, fan_in) layers, W then b."""
    parts = []
    for fo, fi in dims:
        a, b = math.sqrt(6.0 / (fi + fo)), 1.0 / math.sqrt(fi)
        parts.append(_u(g, fo * fi, lo=-a, hi=a, dtype=torch.float32))
        parts.append(_u(g, fo, lo=-b, hi=b, dtype=torch.float32))
    return torch.cat(parts)


def _dims(case):
    if case["kind"] in ("hashgrid", "hg_train"):
        return [(64, ddf.HASHGRID_CODE)] + [(64, 64)] * (case["hidden"] - 1) + [(2, 64)]
    W, k = case["width"], 3 if case["kind"] == "trace" else 6
    return [(W, k + 2 * k * case["octaves"])] + [(W, W)] * (case["hidden"] - 1) + \
        [(1 if case["kind"] == "trace" else 2, W)]


def _blob(case, seed):
    g = _gen(seed, 1)
    dims = _dims(case)
    if case["kind"] in ("hashgrid", "hg_train"):
        table = _u(g, 2 * sum(_hg_sizes()), lo=-1, hi=1, dtype=torch.float32)
        return torch.cat([table, _xavier(dims, g)])
    if case["kind"] == "trace":
        # |p| is 4 times the mean of relu(n . p) over directions n: layer 1 holds the
        # directions and some detail, the layers between pass it on, the head sums it up
        W, H = case["width"], case["hidden"]
        w1 = _u(g, W, dims[0][1], lo=-0.01, hi=0.01, dtype=torch.float32)
        w1[:, :3] = _unit(g, W).float()
        parts = [w1.reshape(-1), torch.zeros(W, device=DEV)]
        for _ in range(H - 1):
            w = torch.eye(W, device=DEV) + _u(g, W, W, lo=-1e-3, hi=1e-3, dtype=torch.float32)
            parts += [w.reshape(-1), torch.zeros(W, device=DEV)]
        return torch.cat(parts + [torch.full((W,), 4.0 / W, device=DEV),
                                  torch.tensor([-0.6], device=DEV)])
    return _xavier(dims, g)


def _scene(seed):
    """64 spheres, centres in the box, radii 0.05 to 0.3."""
    g = _gen(seed, 2)
    return _u(g, 64, 3, lo=-1, hi=1), _u(g, 64, lo=0.05, hi=0.3)


def _surface(seed, n):
    """n points uniform by area on the outside of the scene, and their normals."""
    c, r = _scene(seed)
    g = _gen(seed, 3)
    ps, ns, have = [], [], 0
    while have < n:
        m = int((n - have) * 1.6) + 1024
        i = torch.multinomial((r * r).float(), m, replacement=True, generator=g) if m < (1 << 24) \
            else torch.randint(0, 64, (m,), generator=g, device=DEV)
        nrm = _unit(g, m)
        p = c[i] + r[i, None] * nrm
        inside = torch.zeros(m, dtype=torch.bool, device=DEV)
        for j in range(64):
            inside |= ((p - c[j]).square().sum(1) < r[j] * r[j]) & (i != j)
        ps.append(p[~inside])
        ns.append(nrm[~inside])
        have += ps[-1].shape[0]
    return torch.cat(ps)[:n], torch.cat(ns)[:n]


def _soa(o, d):
    return [x.float().contiguous() for x in (*o.unbind(1), *d.unbind(1))]


def _uniform_rays(seed, n):
    g = _gen(seed, 4)
    return _soa(_u(g, n, 3, lo=-1, hi=1), _unit(g, n))


def _shadow_rays(seed, n):
    p, nrm = _surface(seed, n)
    o = p + 1e-3 * nrm
    d = torch.tensor(LIGHT, device=DEV, dtype=torch.float64) - o
    return _soa(o, d / d.norm(dim=1, keepdim=True))


def _ao_batch(seed, points):
    """CSR batch: 4 to 64 cosine-weighted directions for each surface point."""
    p, nrm = _surface(seed, points)
    g = _gen(seed, 5)
    counts = torch.randint(4, 65, (points,), generator=g, device=DEV)
    off = torch.zeros(points + 1, dtype=torch.int64, device=DEV)
    off[1:] = counts.cumsum(0)
    own = torch.repeat_interleave(torch.arange(points, device=DEV), counts)
    d = nrm[own] + 0.999 * _unit(g, own.numel())
    return _soa(p[own] + 1e-3 * nrm[own], d / d.norm(dim=1, keepdim=True)), off.int()


def _camera_rays(seed, n):
    """Rays from the box's faces towards points inside it."""
    g = _gen(seed, 6)
    o = _u(g, n, 3, lo=-1, hi=1)
    face = torch.randint(0, 6, (n,), generator=g, device=DEV)
    o[torch.arange(n, device=DEV), face // 2] = (face % 2).double() * 2 - 1
    d = _u(g, n, 3, lo=-0.9, hi=0.9) - o
    return o, d / d.norm(dim=1, keepdim=True)


def _train_batch(seed, n):
    """Half camera rays, half surface rays, with exact distances to the scene."""
    o, d = _camera_rays(seed, n)
    p, nrm = _surface(seed, n - n // 2)
    o[n // 2:] = p + 1e-3 * nrm
    d[n // 2:] = _unit(_gen(seed, 7), n - n // 2)
    o, d = o.float().double(), d.float().double()
    c, r = _scene(seed)
    t = torch.full((n,), float("inf"), device=DEV, dtype=torch.float64)
    for j in range(64):
        v = o - c[j]
        b = (v * d).sum(1)
        q = b * b - (v * v).sum(1) + r[j] * r[j]
        s = q.clamp_min(0).sqrt()
        for root in (-b - s, -b + s):
            t = torch.where((q >= 0) & (root > 0) & (root < t), root, t)
    return _soa(o, d), t.float(), torch.isfinite(t).to(torch.uint8)


def prepare(case, seed):
    k = case["kind"]
    if k == "gs":
        scene, _ = I.table_scene()
        means, covs, op = I.surface_gaussians(scene, GAUSSIANS, seed=seed % (1 << 31))
        n = case["views"] * case["size"] ** 2
        return {"case": case, "gauss": [torch.from_numpy(a).to(DEV) for a in (means, covs, op)],
                "cams": I.orbit_cameras(case["views"], seed=seed % (1 << 31)),
                "t": torch.empty(n, device=DEV),
                "hit": torch.empty(n, dtype=torch.uint8, device=DEV)}
    hg = k in ("hashgrid", "hg_train")
    m = ddf.DDF(4 if hg else case["octaves"], 64 if hg else case["width"], case["hidden"],
                precision=case.get("precision", "bf16"), device=0,
                kind="hashgrid" if hg else "sdf" if k == "trace" else "ray")
    s = {"case": case, "m": m}
    m.load(_blob(case, seed).cpu().numpy())
    if case.get("tuned"):  # what ddf_autotune picks for large batches of the paper-sized field
        ddf.ddf_set_tile(m.h, (256, 4, 1, 1, 0), 0)
        ddf.ddf_set_tile(m.h, (256, 8, 0, 1, 1), 1)
    if k in ("rays", "noalloc"):
        s["rays"] = _uniform_rays(seed, case["n"])
        s["t"], s["vis"] = torch.empty(case["n"], device=DEV), torch.empty(case["n"], device=DEV)
    elif k in ("shadow", "hashgrid"):
        s["rays"] = _shadow_rays(seed, case["n"])
    elif k == "ao":
        s["rays"], s["off"] = _ao_batch(seed, case["points"])
        s["hard"] = torch.empty(case["points"], device=DEV)
        s["soft"] = torch.empty(case["points"], device=DEV)
        ddf.ddf_set_graph_mode(m.h, True)
    elif k in ("train", "hg_train"):
        s["rays"], s["target"], s["hit"] = _train_batch(seed, case["batch"])
        s["loss"] = torch.empty(1, device=DEV)
        s["grad"] = torch.empty(m.n_params, device=DEV)
    elif k == "trace":
        s["rays"] = _soa(*_camera_rays(seed, case["n"]))
        s["t"] = torch.empty(case["n"], device=DEV)
        s["hit"] = torch.empty(case["n"], dtype=torch.uint8, device=DEV)
        s["steps"] = torch.empty(case["n"], dtype=torch.int32, device=DEV)
    if case.get("precision") == "fp8":
        cal = _uniform_rays(seed + 1, 65536)
        ddf.ddf_calibrate_fp8(m.h, cal, 65536, torch.cuda.current_stream())
    return s


def run(s):
    case, k = s["case"], s["case"]["kind"]
    st = torch.cuda.current_stream()
    if k == "gs":
        ddf.ddf_render_gs_depth(*s["gauss"], GAUSSIANS, s["cams"], case["size"], case["size"],
                                s["t"], s["hit"], st)
        return {"t": s["t"], "hit": s["hit"]}
    m = s["m"]
    if k == "rays":
        return dict(zip(("t", "vis"), m.query(s["rays"])))
    if k == "noalloc":
        ddf.ddf_query_rays_noalloc(m.h, s["rays"], case["n"], s["t"], s["vis"], st)
        return {"t": s["t"], "vis": s["vis"]}
    if k in ("shadow", "hashgrid"):
        return dict(zip(("t", "vis", "occluded"), m.shadow(s["rays"], LIGHT)))
    if k == "ao":
        ddf.ddf_query_ao(m.h, s["rays"], s["rays"][0].numel(), s["off"], case["points"], s["hard"],
                         s["soft"], st)
        return {"hard": s["hard"], "soft": s["soft"]}
    if k == "trace":
        ddf.ddf_sphere_trace(m.h, s["rays"], case["n"], MAX_STEPS, EPS, T_MAX, s["t"], s["hit"],
                             s["steps"], st)
        return {"t": s["t"], "hit": s["hit"], "steps": s["steps"]}
    lr = 3e-3 if k == "hg_train" else 1e-4
    ddf.ddf_train_step(m.h, s["rays"], s["target"], s["hit"], case["batch"], lr, s["loss"], st)
    ddf.ddf_copy_grad(m.h, s["grad"], st)
    return {"loss": s["loss"], "grad": s["grad"]}


# --------------------------------------------------------------------- work

def work(case):
    k = case["kind"]
    if k == "gs":  # each Gaussian read once a view, each pixel written once; an alpha is about
        # 20 operations and a pixel meets some 30 Gaussians before it is opaque
        px = case["views"] * case["size"] ** 2
        return {"bytes": 40 * GAUSSIANS + 5 * px, "flops": 600 * px + 200 * GAUSSIANS * case["views"]}
    macs = sum(a * b for a, b in _dims(case))
    if k in ("hashgrid", "hg_train"):
        n = case.get("n") or case["batch"]
        entries = 13058044 // 2
        if k == "hg_train":  # weights and both Adam moments in and out, the gradient out
            touched = min(entries, 128 * n)
            return {"bytes": 13058044 * 28 + 8 * touched + 29 * n,
                    "flops": 6 * macs * n + 16 * 8 * 12 * n}
        e = 4 if case["precision"] == "bf16" else 8
        return {"bytes": e * min(entries, 128 * n) + 33 * n, "flops": 2 * macs * n + 16 * 8 * 6 * n}
    e = {"fp32": 4, "bf16": 2, "fp8": 1}[case.get("precision", "bf16")]
    if k == "train":
        n = case["batch"]
        return {"bytes": 32 * macs + 29 * n, "flops": 6 * macs * n}
    if k == "trace":  # about 9 evaluations a ray
        return {"bytes": e * macs + 33 * case["n"], "flops": 9 * 2 * macs * case["n"]}
    n = case["n"] if "n" in case else 34 * case["points"]
    return {"bytes": e * macs + 24 * n + (8 * case["points"] if k == "ao" else 9 * n),
            "flops": 2 * macs * n}


# -------------------------------------------------------------------- exact

def _encode(x, bands):
    """[x, then per coordinate and band sin(pi 2^k x_c), cos(pi 2^k x_c)]."""
    a = x[:, :, None] * (math.pi * 2.0 ** torch.arange(bands, device=x.device, dtype=x.dtype))
    return torch.cat([x, torch.stack([a.sin(), a.cos()], 3).reshape(x.shape[0], -1)], 1)


def _layers(blob, dims):
    out, at = [], 0
    for fo, fi in dims:
        out.append((blob[at:at + fo * fi].reshape(fo, fi), blob[at + fo * fi:at + fo * fi + fo]))
        at += fo * fi + fo
    return out


def _mlp(x, layers):
    for w, b in layers[:-1]:
        x = torch.relu(x @ w.T + b)
    return x @ layers[-1][0].T + layers[-1][1]


def _hg_sizes():
    return [min(2 ** 19, (int(16 * 1.5 ** l) + 1) ** 3) for l in range(16)]


def _hg_code(o, d, table):
    feats, at = [], 0
    x = ((o + 1) * 0.5).clamp(0, 1)
    for l, size in enumerate(_hg_sizes()):
        res = int(16 * 1.5 ** l)
        u = x * res
        i0 = u.floor().long().clamp_max(res - 1)
        w = u - i0
        f = 0
        for c in range(8):
            b = torch.tensor([(c >> a) & 1 for a in range(3)], device=DEV)
            i = i0 + b
            if (res + 1) ** 3 <= size:
                e = i[:, 0] + (res + 1) * (i[:, 1] + (res + 1) * i[:, 2])
            else:
                e = (i[:, 0] ^ (i[:, 1] * 2654435761) ^ (i[:, 2] * 805459861)) & (2 ** 19 - 1)
            f = f + torch.where(b == 1, w, 1 - w).prod(1, keepdim=True) * table[at + e]
        feats.append(f)
        at += size
    return torch.cat(feats + [_encode(d, 4)], 1)


def _loss(z, t_target, hit):
    t = torch.nn.functional.softplus(z[:, 0])
    y = hit.double()
    l1 = ((t.clamp_max(4) - t_target.double().clamp_max(4)).abs())[hit.bool()].sum()
    ce = (torch.nn.functional.softplus(z[:, 1]) - y * z[:, 1]).sum()
    return l1 / max(1.0, float(y.sum())) + 0.3 * ce / z.shape[0]


def _exact_gs(s):
    """The splatting composite of every Gaussian against every pixel, in pixel blocks."""
    case = s["case"]
    means, covs, op = (a.double() for a in s["gauss"])
    C = covs[:, [0, 1, 2, 1, 3, 4, 2, 4, 5]].reshape(-1, 3, 3)
    W = case["size"]
    th = lambda a: torch.tensor(a, device=DEV, dtype=torch.float64)  # noqa: E731
    out_t, out_a = [], []
    for cam in np.asarray(s["cams"], np.float64):
        eye, f, up = cam[:3], cam[3:6] - cam[:3], cam[6:9]
        f = f / np.linalg.norm(f)
        r = np.cross(f, up)
        r /= np.linalg.norm(r)
        u = np.cross(r, f)
        V = th(np.stack([r, u, f]))
        tan = math.tan(0.5 * cam[9])
        fx = W / (2 * tan)
        x, y, z = ((means - th(eye)) @ V.T).unbind(1)
        keep = z > 0.05
        order = torch.sort(torch.where(keep, z, th(float("inf"))), stable=True)[1][:int(keep.sum())]
        x, y, z, o = x[order], y[order], z[order], op[order]
        J = torch.zeros(order.numel(), 2, 3, device=DEV, dtype=torch.float64)
        J[:, 0, 0], J[:, 0, 2] = fx / z, -fx * x / z ** 2
        J[:, 1, 1], J[:, 1, 2] = -fx / z, fx * y / z ** 2
        JV = J @ V
        S = JV @ C[order] @ JV.transpose(1, 2)
        a, b, c = S[:, 0, 0] + 0.3, S[:, 0, 1], S[:, 1, 1] + 0.3
        det = a * c - b * b
        mx, my = x / z * fx + (W - 1) / 2, -y / z * fx + (W - 1) / 2
        pix = torch.arange(W * W, device=DEV)
        px, py = (pix % W).double(), (pix // W).double()
        sx, sy = (2 * (px + 0.5) / W - 1) * tan, (1 - 2 * (py + 0.5) / W) * tan
        cosf = 1 / (1 + sx * sx + sy * sy).sqrt()
        for at in range(0, W * W, 2048):
            ex = px[at:at + 2048, None] - mx
            ey = py[at:at + 2048, None] - my
            q = (c * ex * ex - 2 * b * ex * ey + a * ey * ey) / det
            al = (o * torch.exp(-0.5 * q)).clamp_max(0.99)
            al = torch.where(al >= 1 / 255, al, 0.0)
            T = torch.cumprod(1 - al, 1)
            T = torch.cat([torch.ones_like(T[:, :1]), T[:, :-1]], 1)
            w = torch.where(T >= 1e-4, T * al, 0.0)
            D, A = w @ z, w.sum(1)
            out_t.append(D / A / cosf[at:at + 2048])
            out_a.append(A)
    t, A = torch.cat(out_t), torch.cat(out_a)
    return {"t": torch.where(A > 0, t, th(float("inf"))), "hit": None}


def exact(case, seed):
    k = case["kind"]
    macs = sum(a * b for a, b in _dims(case)) if k != "gs" else 0
    if k in ("rays", "noalloc", "shadow") and case["n"] * macs > 6e12:
        return None  # over 20 seconds in 64 bits
    if k == "gs":
        if case["views"] * case["size"] ** 2 > 1200000:
            return None
        return _exact_gs(prepare(case, seed))
    if k == "trace":
        return None  # a grazing ray stops or goes on by the last bit of s, and t jumps with it
    blob = _blob(case, seed).double()
    dims = _dims(case)
    if k in ("train", "hg_train"):
        rays, t_target, hit = _train_batch(seed, case["batch"])
        o, d = (torch.stack(rays[3 * i:3 * i + 3], 1).double() for i in (0, 1))
        blob.requires_grad_(True)
        loss, n = 0.0, case["batch"]
        if k == "hg_train":
            size = 2 * sum(_hg_sizes())
            loss = _loss(_mlp(_hg_code(o, d, blob[:size].reshape(-1, 2)),
                              _layers(blob[size:], dims)), t_target, hit)
        else:
            if n * macs > 1e12:
                return None  # over 20 seconds in 64 bits
            loss = _loss(_mlp(_encode(torch.cat([o, d], 1), case["octaves"]),
                              _layers(blob, dims)), t_target, hit)
        loss.backward()
        return {"loss": loss.detach().reshape(1), "grad": blob.grad}
    off = None
    if k == "ao":
        rays, off = _ao_batch(seed, case["points"])
    else:
        rays = (_uniform_rays if k in ("rays", "noalloc") else _shadow_rays)(seed, case["n"])
    o, d = (torch.stack(rays[3 * i:3 * i + 3], 1).double() for i in (0, 1))
    zs = []
    for at in range(0, o.shape[0], 65536):
        a, b = o[at:at + 65536], d[at:at + 65536]
        if k == "hashgrid":
            size = 2 * sum(_hg_sizes())
            zs.append(_mlp(_hg_code(a, b, blob[:size].reshape(-1, 2)), _layers(blob[size:], dims)))
        else:
            zs.append(_mlp(_encode(torch.cat([a, b], 1), case["octaves"]), _layers(blob, dims)))
    z = torch.cat(zs)
    t, vis = torch.nn.functional.softplus(z[:, 0]), torch.sigmoid(z[:, 1])
    if k in ("rays", "noalloc"):
        return {"t": t, "vis": vis}
    if k in ("shadow", "hashgrid"):
        return {"t": t, "vis": vis, "occluded": None}
    n = (off[1:] - off[:-1]).long()
    own = torch.repeat_interleave(torch.arange(n.numel(), device=DEV), n)
    mean = lambda v: 1 - torch.zeros(n.numel(), device=DEV, dtype=torch.float64).index_add_(  # noqa
        0, own, v) / n
    return {"hard": None, "soft": mean(vis)}  # hard: a count of decisions
