"""Performance cases of the library: the calls a program makes with it, at the
sizes it makes them.

Families (``kind``): an uplift of mask, RGB-like or descriptor maps
(``uplift``), the FP8-stored uplift with its quantiser (``fp8``), a batch of
uneven uplifts (``batch``), the render-back of uplifted features (``render``),
the diffusion graph of a scene with a 100-step diffusion (``graph``), the
segmentation / multi-query diffusion of a filtered scene (``paper``), and the
scores of text queries (``relevancy``).  Scenes, cameras and feature fields come
from the package's generator; the sizes are those of its workloads, or odd
ones within the same ranges.
"""
import math

import numpy as np
import torch

from paper_2410_14462_gb300 import inputs, ludvig

# Contributors per pixel of a paper-scale view (5.35 G weights over 150 views of
# 980x546): the multiply-adds an uplift or a render cannot do without.
CONTRIB = 65

DTYPES = {"f32": torch.float32, "bf16": torch.bfloat16}


def listed():
    return [
        # An interactive mask uplift on a small scene: the smallest call, where
        # launches and latency count.
        {"name": "mask_small", "kind": "uplift", "scene": "uniform", "n": 20_000, "views": 8, "width": 128,
         "height": 128, "d": 1, "dtype": "f32"},
        # Three-channel maps (mask stacks, colours) in 16 bits over many views.
        {"name": "rgb_bf16", "kind": "uplift", "scene": "clusters", "n": 100_000, "views": 60, "width": 640,
         "height": 480, "d": 3, "dtype": "bf16"},
        # PCA-reduced patch descriptors of a captured scene (40 channels, portrait
        # photographs with ragged tile edges).
        {"name": "pca40_f32", "kind": "uplift", "scene": "clusters", "n": 600_000, "views": 40, "width": 724,
         "height": 986, "d": 40, "dtype": "f32"},
        # The paper-scale descriptor uplift (20 of its 150 views).
        {"name": "field384_f32", "kind": "uplift", "scene": "clusters", "n": 1_000_000, "views": 20, "width": 980,
         "height": 546, "d": 384, "dtype": "f32"},
        # Text-image embeddings in 16 bits, the serving form's images.
        {"name": "embed512_bf16", "kind": "uplift", "scene": "clusters", "n": 500_000, "views": 48, "width": 640,
         "height": 480, "d": 512, "dtype": "bf16"},
        # A descriptor whose width the tensor cores do not take, on odd images.
        {"name": "odd100_f32", "kind": "uplift", "scene": "clusters", "n": 100_000, "views": 10, "width": 331,
         "height": 227, "d": 100, "dtype": "f32"},
        # Features stored in 8 bits: quantise once, uplift the codes.
        {"name": "fp8_512", "kind": "fp8", "scene": "clusters", "n": 250_000, "views": 12, "width": 640,
         "height": 480, "d": 512, "dtype": "f32"},
        # A queue of uneven 16-bit uplifts on several scenes, run as one batch.
        {"name": "batch_mixed", "kind": "batch", "jobs": 10, "job_seed": 3, "pool_views": 40, "n_min": 50_000,
         "n_max": 1_000_000, "v_min": 8, "v_max": 40, "width": 640, "height": 480},
        # Uplifted descriptors reprojected into some of the views.
        {"name": "render384", "kind": "render", "scene": "clusters", "n": 1_000_000, "views": 6, "width": 980,
         "height": 546, "d": 384},
        # The neighbour graph of a scene and one mask diffused on it.
        {"name": "graph_diffuse", "kind": "graph", "scene": "clusters", "n": 1_000_000, "k": 16, "d": 384,
         "steps": 100},
        # Filtering, the feature-distance graph, a segmentation prompt and 21
        # text queries diffused together.
        {"name": "segment_queries", "kind": "paper", "scene": "clusters", "n": 500_000, "k": 16, "d": 384,
         "steps": 100, "queries": 21},
        # Scores of text queries against canonical phrases.
        {"name": "relevancy", "kind": "relevancy", "n": 500_000, "d": 512, "queries": 21, "phrases": 4},
    ]


def _logint(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["uplift", "uplift", "uplift", "fp8", "batch", "render", "graph", "paper", "relevancy"])
    if kind == "batch":
        n_min = _logint(rng, 20_000, 80_000)
        v_min = rng.randint(4, 10)
        pool = rng.randint(14, 40)
        return {"kind": kind, "jobs": rng.randint(3, 10), "job_seed": rng.randint(1, 10_000), "pool_views": pool,
                "n_min": n_min, "n_max": _logint(rng, 2 * n_min, 900_000), "v_min": v_min, "v_max": pool,
                "width": rng.choice([320, 417, 640]), "height": rng.choice([240, 301, 480])}
    if kind == "graph":
        return {"kind": kind, "scene": "clusters", "n": _logint(rng, 20_000, 1_000_000), "k": rng.choice([8, 16, 16]),
                "d": rng.choice([40, 64, 100, 384]), "steps": rng.randint(20, 100)}
    if kind == "paper":
        return {"kind": kind, "scene": "clusters", "n": _logint(rng, 20_000, 500_000), "k": rng.choice([8, 16, 16]),
                "d": rng.choice([40, 64, 384]), "steps": rng.randint(20, 100), "queries": rng.randint(2, 21)}
    if kind == "relevancy":
        return {"kind": kind, "n": _logint(rng, 10_000, 500_000), "d": rng.choice([48, 100, 384, 512]),
                "queries": rng.randint(1, 21), "phrases": rng.randint(1, 4)}
    width, height = _logint(rng, 61, 900), _logint(rng, 45, 700)
    case = {"kind": kind, "scene": rng.choice(["clusters", "clusters", "uniform"]), "n": _logint(rng, 5_000, 900_000),
            "width": width, "height": height}
    if kind == "uplift":
        d = rng.choice([1, 3, 8, 27, 40, 64, 100, 192, 384, 512])
        # at most the values of the largest listed case, and of the odd widths'
        most = 4_000_000_000 if d != 100 else 75_000_000
        case.update(d=d, dtype=rng.choice(["f32", "bf16"]), views=_views(rng, width, height, d, most, 60))
        return case
    if kind == "fp8":
        d = rng.choice([3, 48, 64, 384, 512])
        case.update(d=d, dtype=rng.choice(["f32", "bf16"]), views=_views(rng, width, height, d, 1_800_000_000, 20))
        return case
    d = rng.choice([3, 40, 64, 384])
    case.update(d=d, views=_views(rng, width, height, d, 1_200_000_000, 12))
    return case


def _views(rng, width, height, d, most, cap):
    hi = max(1, min(cap, int(most // (width * height * d))))
    return rng.randint(1, hi)


# ------------------------------------------------------------------ inputs

def _host_scene(case, seed):
    if case.get("scene") == "uniform":
        return inputs.scene_uniform(case["n"], seed=seed)
    return inputs.scene_clusters(case["n"], seed=seed)


def _cameras(case):
    w, h = case["width"], case["height"]
    if case.get("scene") == "uniform":
        return inputs.cameras_orbit(case["views"], 3.0, w, h, 120.0 * w / 128.0, hemisphere=False)
    return inputs.cameras_orbit(case["views"], 4.0, w, h, 900.0 * max(w, h) / 980.0, hemisphere=True)


def _maps(case, cams, seed, d, dtype):
    """Feature maps [V,H,W,d] on the GPU: masks for one channel, else the smooth
    unit-norm field."""
    out = torch.empty((cams.v, cams.height, cams.width, d), dtype=dtype, device="cuda")
    for v in range(cams.v):
        if d == 1:
            centre = 0.1 * np.random.default_rng([seed, 3]).standard_normal(3)
            m = inputs.sphere_masks(cams.subset([v]), center=centre)[0]
            out[v] = torch.from_numpy(m).to(device="cuda", dtype=dtype)
        else:
            out[v] = inputs.feature_field(seed, v, d, cams.height, cams.width, device="cuda", dtype=dtype)
    return out


def _gaussian_features(means, d, seed):
    """Per-Gaussian descriptors as an uplift leaves them: smooth over the scene,
    with some noise."""
    g = torch.Generator(device="cuda").manual_seed(1000 + seed)
    m = torch.from_numpy(means).cuda()
    a = torch.randn((3, d), device="cuda", generator=g) * 1.5
    ph = torch.rand((d,), device="cuda", generator=g) * 6.2831853
    f = torch.cos(m @ a + ph)
    f += 0.3 * torch.randn(f.shape, device="cuda", generator=g)
    return f / f.norm(dim=1, keepdim=True)


def prepare(case, seed):
    kind = case["kind"]
    if kind in ("uplift", "fp8"):
        cams = _cameras(case)
        return {"case": case, "scene": ludvig.Scene.from_inputs(_host_scene(case, seed)), "cams": cams,
                "feats": _maps(case, cams, seed, case["d"], DTYPES[case["dtype"]])}
    if kind == "render":
        host = _host_scene(case, seed)
        return {"case": case, "scene": ludvig.Scene.from_inputs(host), "cams": _cameras(case),
                "f": _gaussian_features(host.means, case["d"], seed).contiguous()}
    if kind == "batch":
        cams, specs = _batch(case)
        pools = {d: _maps(case, cams, seed, d, torch.bfloat16) for d in sorted({s.d for s in specs})}
        jobs = [(ludvig.Scene.from_inputs(inputs.scene_clusters(s.n, seed=seed * 100 + j)),
                 cams.params[s.v0:s.v0 + s.views], cams.width, cams.height, pools[s.d][s.v0:s.v0 + s.views], None, None)
                for j, s in enumerate(specs)]
        return {"case": case, "jobs": jobs}
    if kind == "relevancy":
        g = torch.Generator(device="cuda").manual_seed(seed)
        f = torch.randn((case["n"], case["d"]), device="cuda", generator=g)
        return {"case": case, "f": f / f.norm(dim=1, keepdim=True),
                "q": torch.randn((case["queries"], case["d"]), device="cuda", generator=g),
                "c": torch.randn((case["phrases"], case["d"]), device="cuda", generator=g)}
    host = _host_scene(case, seed)
    f = _gaussian_features(host.means, case["d"], seed)
    g = torch.Generator(device="cuda").manual_seed(seed)
    means = torch.from_numpy(host.means).cuda()
    dist = (means - means[seed % host.n]).norm(dim=1)
    seen = torch.rand((host.n,), device="cuda", generator=g) > 0.2
    state = {"case": case, "scene": ludvig.Scene.from_inputs(host)}
    if kind == "graph":
        # Gaussians that no view sees have zero features; a mask around one centre
        state["f"] = (f * seen[:, None]).contiguous()
        state["x0"] = (dist < 0.15).float()
        return state
    state["f"] = f.contiguous()
    state["beta"] = torch.exp(torch.randn((host.n,), device="cuda", generator=g)) * seen
    state["u"] = torch.clamp(1.0 - dist / 0.5, min=0.0) * seen
    x0 = torch.zeros((host.n - host.n // 2, case["queries"]), device="cuda")
    q = torch.arange(case["queries"], device="cuda")
    x0[(q * 997 + seed) % x0.shape[0], q] = 1.0
    state["x0"] = x0
    return state


def _batch(case):
    cams = inputs.cameras_orbit(case["pool_views"], 4.0, case["width"], case["height"],
                                inputs.FORM_FOCAL * case["width"] / inputs.FORM_WIDTH, hemisphere=True)
    return cams, inputs.batch_jobs(case["jobs"], seed=case["job_seed"], pool_views=case["pool_views"],
                                   n_range=(case["n_min"], case["n_max"]), views_range=(case["v_min"], case["v_max"]))


# ------------------------------------------------------------------ passes

def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "uplift":
        return ludvig.uplift(state["scene"], state["cams"].params, case["width"], case["height"], state["feats"])
    if kind == "fp8":
        q, s = ludvig.fp8_quantize(state["feats"])
        out, beta = ludvig.uplift_fp8(state["scene"], state["cams"].params, case["width"], case["height"], q, s)
        return q, s, out, beta
    if kind == "batch":
        return [t for pair in ludvig.uplift_batch(state["jobs"])[0] for t in pair]
    if kind == "render":
        return ludvig.render(state["scene"], state["cams"].params, case["width"], case["height"], state["f"])
    if kind == "relevancy":
        return ludvig.relevancy(state["f"], state["q"], state["c"], 10.0)
    if kind == "graph":
        graph = ludvig.Graph(state["scene"], case["k"], state["f"], spatial_h=0.01)
        y = graph.diffuse(state["x0"], case["steps"])
        graph.close()
        return y
    scene, n = state["scene"], case["n"]
    kept = ludvig.beta_select(scene, state["beta"], n - n // 2)
    sub = scene.subset(kept)
    idx = kept.long()
    f, u = state["f"][idx].contiguous(), state["u"][idx].contiguous()
    graph = ludvig.Graph.rbf(sub, case["k"], f)
    scale = graph.feature_scale
    g0 = ludvig.topfrac_positive(sub, u, 10)
    unary = graph.unary_anchor(f, g0, 5.0)
    graph.reweight(0.5, unary, binarize=1e-5, row_normalize=False)
    h = graph.reach_weight(g0, case["steps"], unary)
    graph.reweight(0.5, None, binarize=0.0, row_normalize=True)
    y = graph.diffuse(state["x0"], case["steps"])
    graph.close()
    sub.close()
    return kept, scale, g0, unary, h, y


def work(case):
    kind = case["kind"]
    if kind == "relevancy":
        n, d, q, c = case["n"], case["d"], case["queries"], case["phrases"]
        return {"bytes": 4 * (n * d + (q + c) * d + n * q), "flops": 2 * n * d * (q + c)}
    if kind in ("graph", "paper"):
        # the features once, an edge list of about 1.4 k n entries written once
        # and read once per step (8 B), the columns read and written per step
        n = case["n"] if kind == "graph" else case["n"] - case["n"] // 2
        nnz = int(1.4 * case["k"] * n)
        cols = 1 if kind == "graph" else case["queries"]
        passes = case["steps"] + 1 if kind == "graph" else 2 * case["steps"] + 1
        return {"bytes": 4 * case["n"] * (case["d"] + 13) + passes * 8 * nnz + case["steps"] * 8 * n * cols,
                "flops": 2 * nnz * case["d"] + 2 * nnz * cols * case["steps"]}
    if kind == "batch":
        _, specs = _batch(case)
        px = case["width"] * case["height"]
        return {"bytes": sum(2 * s.views * px * s.d + 44 * s.n + 4 * s.n * (s.d + 1) for s in specs),
                "flops": sum(2 * CONTRIB * s.views * px * (s.d + 1) for s in specs)}
    n, d, px = case["n"], case["d"], case["views"] * case["width"] * case["height"]
    flops = 2 * CONTRIB * px * (d + 1)
    if kind == "render":
        return {"bytes": 4 * px * d + 44 * n + 4 * n * d, "flops": flops}
    size = 4 if case["dtype"] == "f32" else 2
    bytes_ = size * px * d + 44 * n + 4 * n * (d + 1)
    if kind == "fp8":
        bytes_ += 2 * px * d   # codes written and read
    return {"bytes": bytes_, "flops": flops}


# ------------------------------------------------------------------ 64-bit values

# (view, tile) products the 64-bit rasteriser forms in under 20 seconds.
EXACT_TILES = 16_000


def exact(case, seed):
    kind = case["kind"]
    if kind == "relevancy":
        return _exact_relevancy(prepare(case, seed))
    if kind == "batch":
        return None
    if kind in ("graph", "paper"):
        if case["n"] > 250_000:
            return None
        return _exact_graph(case, seed) if kind == "graph" else _exact_paper(case, seed)
    tiles = case["views"] * -(-case["width"] // 16) * -(-case["height"] // 16)
    if tiles > EXACT_TILES:
        return None
    host, cams = _host_scene(case, seed), _cameras(case)
    if kind == "render":
        f = _gaussian_features(host.means, case["d"], seed).double()
        out = torch.zeros((cams.v, cams.height, cams.width, case["d"]), dtype=torch.float64, device="cuda")
        for v in range(cams.v):
            for ys, xs, ids, w in _tiles(host, cams, v):
                out[v, ys, xs] += (w.T @ f[ids]).reshape(ys.stop - ys.start, xs.stop - xs.start, -1)
        return out
    feats = _maps(case, cams, seed, case["d"], DTYPES[case["dtype"]])
    codes = None
    if kind == "fp8":
        amax = feats.float().abs().amax(dim=(1, 2, 3))
        scales = torch.where(amax > 0, amax.double() / 448.0, torch.ones_like(amax, dtype=torch.float64))
        s = scales.float()
        codes = [(feats[v].float() / s[v]).to(torch.float8_e4m3fn) for v in range(cams.v)]
    num = torch.zeros((host.n, case["d"]), dtype=torch.float64, device="cuda")
    den = torch.zeros((host.n,), dtype=torch.float64, device="cuda")
    for v in range(cams.v):
        fv = feats[v].double() if codes is None else codes[v].double() * scales[v]
        for ys, xs, ids, w in _tiles(host, cams, v):
            num.index_add_(0, ids, w @ fv[ys, xs].reshape(-1, case["d"]))
            den.index_add_(0, ids, w.sum(dim=1))
    out = torch.where(den[:, None] > 0, num / den[:, None], torch.zeros_like(num))
    return (out, den) if codes is None else (None, scales, out, den)


def _project(host, cams, v):
    """Visible Gaussians of a view in depth order, in float64: index, mean,
    conic, opacity and tile rectangle (the 3DGS rasteriser's rules)."""
    p = torch.from_numpy(cams.params[v]).double().cuda()
    rot, t, (fx, fy, cx, cy) = p[:9].reshape(3, 3), p[9:12], [float(x) for x in p[12:16]]
    mean, sc, q, op = [torch.from_numpy(a).double().cuda() for a in (host.means, host.scales, host.quats, host.opacity)]
    q = q / q.norm(dim=1, keepdim=True)
    w, x, y, z = q.unbind(1)
    r = torch.stack([1 - 2 * (y * y + z * z), 2 * (x * y - w * z), 2 * (x * z + w * y),
                     2 * (x * y + w * z), 1 - 2 * (x * x + z * z), 2 * (y * z - w * x),
                     2 * (x * z - w * y), 2 * (y * z + w * x), 1 - 2 * (x * x + y * y)], dim=1).reshape(-1, 3, 3)
    m = r * sc[:, None, :]
    cam = rot @ (m @ m.transpose(1, 2)) @ rot.T
    tc = mean @ rot.T + t
    tx, ty, tz = tc.unbind(1)
    ids = torch.nonzero(tz > 0.2)[:, 0]
    tx, ty, tz, cam, op = tx[ids], ty[ids], tz[ids], cam[ids], op[ids]
    limx, limy = 1.3 * 0.5 * cams.width / fx, 1.3 * 0.5 * cams.height / fy
    jx, jy = (tx / tz).clamp(-limx, limx) * tz, (ty / tz).clamp(-limy, limy) * tz
    zero = torch.zeros_like(tz)
    j = torch.stack([fx / tz, zero, -fx * jx / tz ** 2, zero, fy / tz, -fy * jy / tz ** 2], dim=1).reshape(-1, 2, 3)
    s2 = j @ cam @ j.transpose(1, 2)
    a, b, c = s2[:, 0, 0] + 0.3, s2[:, 0, 1], s2[:, 1, 1] + 0.3
    det = a * c - b * b
    mid = 0.5 * (a + c)
    rad = torch.ceil(3.0 * torch.sqrt(mid + torch.sqrt((mid * mid - det).clamp(min=0.1))))
    mx, my = fx * tx / tz + cx, fy * ty / tz + cy
    nx, ny = -(-cams.width // 16), -(-cams.height // 16)
    x0, x1 = torch.floor((mx - rad) / 16).clamp(0, nx), (torch.floor((mx + rad) / 16) + 1).clamp(0, nx)
    y0, y1 = torch.floor((my - rad) / 16).clamp(0, ny), (torch.floor((my + rad) / 16) + 1).clamp(0, ny)
    keep = torch.nonzero((det > 0) & (x0 < x1) & (y0 < y1) & (op >= 1.0 / 255.0))[:, 0]
    keep = keep[torch.sort(tz[keep], stable=True)[1]]
    cols = [mx, my, c / det, -b / det, a / det, op, x0, x1, y0, y1]
    return ids[keep], [u[keep] for u in cols]


def _tiles(host, cams, v):
    """The alpha-blending weights of a view tile by tile, in float64: yields the
    tile's rows and columns, Gaussian indices [r] and weights [r, pixels]."""
    ids, cols = _project(host, cams, v)
    for ty in range(-(-cams.height // 16)):
        row = torch.nonzero((cols[8] <= ty) & (cols[9] > ty))[:, 0]
        rcols, rids = [c[row] for c in cols[:8]], ids[row]
        ys = slice(16 * ty, min(16 * ty + 16, cams.height))
        for tx in range(-(-cams.width // 16)):
            sel = torch.nonzero((rcols[6] <= tx) & (rcols[7] > tx))[:, 0]
            xs = slice(16 * tx, min(16 * tx + 16, cams.width))
            px = torch.arange(xs.start, xs.stop, device="cuda").double() + 0.5
            py = torch.arange(ys.start, ys.stop, device="cuda").double() + 0.5
            py, px = [g.reshape(-1) for g in torch.meshgrid(py, px, indexing="ij")]
            trans = torch.ones_like(px)
            for k in range(0, int(sel.numel()), 512):
                s = sel[k:k + 512]
                mx, my, ca, cb, cc, op = [c[s][:, None] for c in rcols[:6]]
                dx, dy = mx - px, my - py
                power = -0.5 * (ca * dx * dx + cc * dy * dy) - cb * dx * dy
                alpha = (op * torch.exp(power.clamp(max=0.0))).clamp(max=0.99)
                alpha = torch.where((power > 0) | (alpha < 1.0 / 255.0), torch.zeros_like(alpha), alpha)
                after = trans * torch.cumprod(1.0 - alpha, dim=0)
                before = torch.cat([trans[None], after[:-1]])
                w = torch.where(after >= 1e-4, alpha * before, torch.zeros_like(alpha))
                hit = torch.nonzero(w.amax(dim=1) > 0)[:, 0]
                if hit.numel():
                    yield ys, xs, rids[s[hit]], w[hit]
                trans = after[-1]
                if float(trans.max()) < 1e-4:
                    break


def _exact_relevancy(state):
    f, q, c = [t.double() for t in (state["f"], state["q"], state["c"])]
    f, q, c = [t / t.norm(dim=1, keepdim=True) for t in (f, q, c)]
    sq, sc = 10.0 * f @ q.T, 10.0 * f @ c.T
    return 1.0 / (1.0 + torch.exp(sc.amax(dim=1, keepdim=True) - sq))


def _edges(means, k):
    """Union of the k-nearest-neighbour lists, without self edges, by (row, col)."""
    m = torch.from_numpy(means).double().cuda()
    n = m.shape[0]
    key = []
    for i in range(0, n, 1024):
        d2 = torch.zeros((min(1024, n - i), n), dtype=torch.float64, device="cuda")
        for a in range(3):
            d2 += (m[i:i + 1024, a, None] - m[None, :, a]) ** 2
        r = torch.arange(i, min(i + 1024, n), device="cuda")
        d2[r - i, r] = math.inf
        c = torch.topk(d2, min(k, n - 1), dim=1, largest=False)[1]
        r = r[:, None].expand_as(c)
        key += [(r * n + c).reshape(-1), (c * n + r).reshape(-1)]
    key = torch.unique(torch.cat(key))
    return m, key // n, key % n


def _matrix(rows, cols, val, n):
    total = torch.zeros((n,), dtype=torch.float64, device="cuda").index_add_(0, rows, val)
    val = torch.where(total[rows] > 0, val / total[rows], torch.zeros_like(val))
    ptr = torch.zeros((n + 1,), dtype=torch.int64, device="cuda")
    ptr[1:] = torch.cumsum(torch.bincount(rows, minlength=n), 0)
    return torch.sparse_csr_tensor(ptr, cols, val, size=(n, n))


def _power_steps(mat, x0, steps):
    g = x0.double().reshape(x0.shape[0], -1)
    for _ in range(steps):
        nrm = g.norm(dim=0)
        g = mat @ torch.where(nrm > 0, g / nrm, torch.zeros_like(g))
    return g.reshape(x0.shape)


def _unit(f):
    f = f.double()
    nrm = f.norm(dim=1, keepdim=True)
    return torch.where(nrm > 0, f / nrm, torch.zeros_like(f))


def _exact_graph(case, seed):
    state = prepare(case, seed)
    m, rows, cols = _edges(_host_scene(case, seed).means, case["k"])
    f = _unit(state["f"])
    val = torch.cat([(f[r] * f[c]).sum(dim=1) for r, c in zip(rows.split(1 << 20), cols.split(1 << 20))])
    val = val.clamp(min=0.0) * torch.exp(-((m[rows] - m[cols]) ** 2).sum(dim=1) / 0.01)
    return _power_steps(_matrix(rows, cols, val, case["n"]), state["x0"], case["steps"])


def _exact_paper(case, seed):
    state = prepare(case, seed)
    n, keep = case["n"], case["n"] - case["n"] // 2
    idx = torch.sort(torch.sort(-state["beta"].double(), stable=True)[1][:keep])[0]
    u = state["u"][idx].double()
    npos = int((u > 0).sum())
    top = torch.sort(-u, stable=True)[1][:(npos * 10 + 99) // 100]
    g0 = torch.zeros_like(u)
    g0[top] = u[top]
    _, rows, cols = _edges(_host_scene(case, seed).means[idx.cpu().numpy()], case["k"])
    f = _unit(state["f"][idx])
    d2 = torch.cat([((f[r] - f[c]) ** 2).sum(dim=1) for r, c in zip(rows.split(1 << 20), cols.split(1 << 20))])
    mid = torch.sort(torch.sqrt(d2))[0][[(d2.numel() - 1) // 2, d2.numel() // 2]]
    scale = float(mid.mean())
    anchor = _unit((f * (g0 > 0)[:, None]).sum(dim=0, keepdim=True))
    unary = torch.exp(-((f - anchor) ** 2).sum(dim=1) / (5.0 * scale * scale))
    sim = torch.exp(-d2 / (0.5 * scale * scale))
    edge = sim * torch.sqrt(unary)[rows] * torch.sqrt(unary)[cols] > 1e-5
    reach = g0 > 0
    for _ in range(case["steps"]):
        step = torch.zeros((keep,), dtype=torch.int32, device="cuda")
        step.index_add_(0, rows, (edge & reach[cols]).int())
        reach = step > 0
    y = _power_steps(_matrix(rows, cols, sim, keep), state["x0"], case["steps"])
    return idx, scale, g0, unary, torch.where(reach, unary, torch.zeros_like(unary)), y
