"""What is measured: the calls that a user of the extractor makes, through the
package's public entry points, over the sizes and options that they are used with.

Every case is a dict of plain values whose "kind" names the call:

  extract   one image, sift_extract into the caller's table
  batch     several images of any sizes, sift_extract_batch into the caller's tables
  serve     a burst of requests, Server.submit / result, copied into the caller's tables
  match     two descriptor sets, Extractor.match
  magsac    correspondences and minimal samples, Extractor.magsac
  pyramid   one image's Gaussian scale space, Extractor.pyramid

Images are synthetic (background, blobs, rectangles, 1/f texture, noise; FP32 in
[0, 1]), made on the GPU from the seed. Handles are kept for the process by
parameter set, as a program that extracts from a stream of images keeps its own.
"""
import math

import numpy as np
import torch
import torch.nn.functional as F

import paper_2605_17869_gb300 as sift

FIELDS = ("x", "y", "sigma", "angle", "response", "octave", "layer", "desc")
ASPECTS = ((4, 3), (3, 4), (16, 9))  # width : height, as in the mixed-resolution batch


def listed():
    return [
        # A tracked patch or a thumbnail: the smallest call, all latency. Odd sides, unaligned rows.
        {"name": "thumbnail", "kind": "extract", "h": 121, "w": 163, "texture": 0.03},
        # One camera frame at VGA, plain SIFT: the usual single call.
        {"name": "vga", "kind": "extract", "h": 480, "w": 640, "texture": 0.0},
        # One 4K frame, the largest image that the server sees.
        {"name": "uhd", "kind": "extract", "h": 2160, "w": 3840, "texture": 0.02},
        # An image sequence under homographies (six 1000 x 750), double image, with the paper's
        # own descriptor options: DSP pooling and RootSIFT.
        {"name": "sequence_dsp", "kind": "batch", "h": 750, "w": 1000, "n": 6, "texture": 0.02,
         "upsample": 1, "dsp": 1, "rootsift": 1, "max_kpts": 8000},
        # Indexing a collection: 64 images of mixed resolution in one call.
        {"name": "mixed64", "kind": "batch", "n": 64, "mixed": 1, "texture": 0.05, "max_kpts": 2048},
        # The same use where device memory is short: binary16 storage above octave 0.
        {"name": "mixed16_fp16", "kind": "batch", "n": 16, "mixed": 2, "texture": 0.05,
         "fp16_pyramid": 1, "max_kpts": 2048},
        # Reconstruction from strongly textured photographs, double image, the cap of 8192 reached:
        # orientation and descriptor carry the load.
        {"name": "textured_up2", "kind": "batch", "h": 1200, "w": 1600, "n": 4, "texture": 0.12,
         "upsample": 1, "max_kpts": 8192},
        # Finer sampling of scale (five layers per octave) on a small batch: other blur radii and
        # more levels per octave than the defaults.
        {"name": "five_scales", "kind": "batch", "h": 768, "w": 1024, "n": 4, "texture": 0.05,
         "n_scales": 5, "max_kpts": 8192},
        # A burst at the server: two camera frames, an HD and a 4K frame at once.
        {"name": "serve_burst", "kind": "serve", "n": 4, "texture": 0.02},
        # The descriptors of two capped images against each other; ragged sizes.
        {"name": "match_8k", "kind": "match", "na": 8192, "nb": 7801},
        # Verifying one image pair: about a thousand matches, 1,500 minimal samples.
        {"name": "magsac", "kind": "magsac", "n": 1003, "n_hyp": 1500},
        # The scale space itself, for callers with detectors of their own: one HD frame.
        {"name": "pyramid_hd", "kind": "pyramid", "h": 1080, "w": 1920, "texture": 0.02},
    ]


def _log_uniform(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def _sides(rng, px):
    a = math.exp(rng.uniform(math.log(0.5), math.log(2.0)))
    return max(33, int(math.sqrt(px / a))), max(33, int(math.sqrt(px * a)))


def draw(rng):
    kind = rng.choice(("extract", "extract", "batch", "batch", "batch", "serve", "match", "magsac", "pyramid"))
    c = {"kind": kind}
    if kind == "match":
        c.update(na=int(_log_uniform(rng, 64, 8192)), nb=int(_log_uniform(rng, 64, 8192)))
        return c
    if kind == "magsac":
        c.update(n=int(_log_uniform(rng, 64, 8192)), n_hyp=int(_log_uniform(rng, 500, 4000)))
        return c
    c["texture"] = rng.choice((0.0, 0.02, 0.05, 0.05, 0.12))
    if kind == "serve":
        c.update(n=rng.randint(1, 8), frames=rng.randint(1, 1 << 20))
        return c
    if rng.random() < 0.4:
        c["upsample"] = 1
    if rng.random() < 0.2:
        c["n_scales"] = rng.choice((4, 5))
    elif rng.random() < 0.2:
        c["fp16_pyramid"] = 1
    if kind == "pyramid":
        c["h"], c["w"] = _sides(rng, _log_uniform(rng, 2e4, 2.5e6))
        return c
    if rng.random() < 0.25:
        c.update(dsp=1, rootsift=1)
    if rng.random() < 0.1:
        c["upright"] = 1
    c["max_kpts"] = rng.choice((1024, 2048, 8192))
    most = 4 if c.get("upsample") else 1  # octave-0 pixels per input pixel
    if kind == "extract":
        c["h"], c["w"] = _sides(rng, _log_uniform(rng, 2e4, 8e6 / most))
    elif rng.random() < 0.5 and not c.get("upsample"):
        c["n"] = int(_log_uniform(rng, 2, 48))
        c["mixed"] = rng.randint(3, 1 << 20)
    else:
        c["n"] = int(_log_uniform(rng, 2, 24))
        c["h"], c["w"] = _sides(rng, _log_uniform(rng, 1e5, 2e6) / max(1, c["n"] * most / 16))
    return c


# ------------------------------------------------------------------ inputs

def _params(case):
    keys = ("upsample", "dsp", "rootsift", "fp16_pyramid", "n_scales", "upright", "max_kpts")
    return {k: case[k] for k in keys if k in case}


def _shapes(case):
    if case["kind"] == "serve":  # half VGA, a third HD, the rest 4K
        sizes = ((480, 640), (1080, 1920), (480, 640), (2160, 3840))
        if "frames" not in case:
            return [sizes[i % len(sizes)] for i in range(case["n"])]
        rng = np.random.default_rng(case["frames"])
        return [sizes[int(k)] for k in rng.choice((0, 1, 3), size=case["n"], p=(0.5, 0.35, 0.15))]
    if "mixed" not in case:
        return [(case["h"], case["w"])] * case.get("n", 1)
    rng = np.random.default_rng(case["mixed"])  # a collection's shapes do not depend on its pixels
    out = []
    for _ in range(case["n"]):
        side = int(rng.integers(480, 1601))
        a, b = ASPECTS[int(rng.integers(0, 3))]
        out.append((int(round(side * b / a)), side) if a >= b else (side, int(round(side * a / b))))
    return out


def _image(gen, h, w, texture):
    """Background 0.5, blobs (sigma 2 .. 30 px), rectangles, 1/f texture and noise, clipped to [0, 1]."""
    dev = "cuda"
    n_blob, n_rect = (200 if texture > 0.03 else 40), 10

    def u(n, lo=0.0, hi=1.0):
        return torch.rand(n, generator=gen, device=dev) * (hi - lo) + lo

    yy = torch.arange(h, device=dev, dtype=torch.float32)
    xx = torch.arange(w, device=dev, dtype=torch.float32)
    s = torch.exp(u(n_blob, math.log(2.0), math.log(30.0)))[:, None]
    gy = torch.exp(-((yy - u(n_blob, 0, h)[:, None]) / s) ** 2 / 2) * u(n_blob, -0.3, 0.3)[:, None]
    gx = torch.exp(-((xx - u(n_blob, 0, w)[:, None]) / s) ** 2 / 2)
    ya, yb = u(n_rect, 0, h)[:, None], u(n_rect, 0, h)[:, None]
    xa, xb = u(n_rect, 0, w)[:, None], u(n_rect, 0, w)[:, None]
    ry = ((yy >= torch.minimum(ya, yb)) & (yy <= torch.maximum(ya, yb))).float() * u(n_rect, -0.2, 0.2)[:, None]
    rx = ((xx >= torch.minimum(xa, xb)) & (xx <= torch.maximum(xa, xb))).float()
    img = 0.5 + torch.cat([gy, ry]).T @ torch.cat([gx, rx])
    if texture > 0:
        spec = torch.fft.rfft2(torch.randn(h, w, generator=gen, device=dev))
        f = torch.hypot(torch.fft.fftfreq(h, device=dev)[:, None], torch.fft.rfftfreq(w, device=dev)[None])
        f = torch.clamp(f, min=1.0 / max(h, w))
        f[0, 0] = math.inf
        tex = torch.fft.irfft2(spec / f, s=(h, w))
        img = img + tex * (texture / tex.std())
    img = img + 0.01 * torch.randn(h, w, generator=gen, device=dev)
    return img.clamp_(0.0, 1.0).contiguous()


def _images(case, seed):
    gen = torch.Generator(device="cuda").manual_seed(seed)
    return [_image(gen, h, w, case["texture"]) for h, w in _shapes(case)]


def _descriptors(case, seed):
    """Two sets of SIFT-like descriptors (unit norm, entries clipped at 0.2 before the last
    normalisation); half of the smaller set has a noisy partner in the other."""
    gen = torch.Generator(device="cuda").manual_seed(seed)

    def unit(d):
        d = d / d.norm(dim=1, keepdim=True)
        d = d.clamp(max=0.2)
        return (d / d.norm(dim=1, keepdim=True)).contiguous()

    a = unit(torch.rand(case["na"], 128, generator=gen, device="cuda") ** 3)
    b = torch.rand(case["nb"], 128, generator=gen, device="cuda") ** 3
    m = min(case["na"], case["nb"]) // 2
    pa = torch.randperm(case["na"], generator=gen, device="cuda")[:m]
    pb = torch.randperm(case["nb"], generator=gen, device="cuda")[:m]
    b = unit(b)
    b[pb] = unit((a[pa] + 0.02 * torch.randn(m, 128, generator=gen, device="cuda")).clamp(min=0.0))
    return a, b


def _correspondences(case, seed):
    """Points under a homography with 0.5 px noise; a quarter of them have nothing to do with it."""
    rng = np.random.default_rng(seed)
    n = case["n"]
    th, s = rng.uniform(-0.5, 0.5), rng.uniform(0.7, 1.3)
    H = np.array([[s * math.cos(th), -s * math.sin(th), rng.uniform(-50, 50)],
                  [s * math.sin(th), s * math.cos(th), rng.uniform(-50, 50)],
                  [rng.uniform(-5e-5, 5e-5), rng.uniform(-5e-5, 5e-5), 1.0]])
    xa = rng.uniform((0, 0), (1600, 1200), size=(n, 2))
    q = np.concatenate([xa, np.ones((n, 1))], 1) @ H.T
    xb = q[:, :2] / q[:, 2:] + rng.normal(0, 0.5, size=(n, 2))
    out = rng.random(n) < 0.25
    xb[out] = rng.uniform((0, 0), (1600, 1200), size=(int(out.sum()), 2))
    samples = sift.draw_samples(n, case["n_hyp"], seed=seed)
    return xa.astype(np.float32), xb.astype(np.float32), samples


# ------------------------------------------------------------------ cases

_extractors, _servers = {}, {}


def _extractor(case):
    p = _params(case)
    key = tuple(sorted(p.items()))
    if key not in _extractors:
        _extractors[key] = sift.Extractor(**p)
    return _extractors[key]


def prepare(case, seed):
    kind = case["kind"]
    if kind == "match":
        a, b = _descriptors(case, seed)
        return {"kind": kind, "ex": _extractor(case), "a": a, "b": b}
    if kind == "magsac":
        xa, xb, samples = (torch.from_numpy(v).cuda() for v in _correspondences(case, seed))
        return {"kind": kind, "ex": _extractor(case), "xa": xa, "xb": xb, "samples": samples}
    imgs = _images(case, seed)
    if kind == "pyramid":
        return {"kind": kind, "ex": _extractor(case), "img": imgs[0]}
    # The caller's own result tables, one row of max_kpts entries per image.
    n, k = len(imgs), case.get("max_kpts", 8192)
    out = {f: torch.zeros((n, k), dtype=torch.int32 if f in ("octave", "layer") else torch.float32,
                          device="cuda") for f in FIELDS[:-1]}
    out["desc"] = torch.zeros((n, k, 128), dtype=torch.float32, device="cuda")
    if kind == "serve":
        if "server" not in _servers:
            _servers["server"] = sift.Server(sift.Extractor(max_kpts=k), budget_bytes=8 << 30)
        return {"kind": kind, "srv": _servers["server"], "imgs": imgs, "out": out}
    out["count"] = torch.zeros(n, dtype=torch.int32, device="cuda")
    kpts = [sift.SiftKptsDev(*(out[f][i].data_ptr() for f in FIELDS[:-1])) for i in range(n)]
    return {"kind": kind, "ex": _extractor(case), "imgs": imgs, "out": out,
            "ptrs": [im.data_ptr() for im in imgs], "hs": [im.shape[0] for im in imgs],
            "ws": [im.shape[1] for im in imgs], "pitches": [im.stride(0) for im in imgs],
            "kpts": (sift.SiftKptsDev * n)(*kpts), "descs": [out["desc"][i].data_ptr() for i in range(n)]}


def run(state):
    kind = state["kind"]
    if kind == "extract":
        img, out = state["imgs"][0], state["out"]
        sift.sift_extract(state["ex"].handle, img.data_ptr(), img.shape[0], img.shape[1], img.stride(0),
                          torch.cuda.current_stream().cuda_stream, state["kpts"][0], state["descs"][0],
                          out["count"].data_ptr())
        return out
    if kind == "batch":
        sift.sift_extract_batch(state["ex"].handle, state["ptrs"], state["hs"], state["ws"],
                                state["pitches"], torch.cuda.current_stream().cuda_stream,
                                state["kpts"], state["descs"], state["out"]["count"].data_ptr())
        return state["out"]
    if kind == "serve":
        srv, out = state["srv"], state["out"]
        tickets = [srv.submit(im) for im in state["imgs"]]
        for i, t in enumerate(tickets):  # a result is the server's until it is released
            f = srv.result(t)[0]
            for key in FIELDS:
                out[key][i, :f.count].copy_(getattr(f, key))
        torch.cuda.current_stream().synchronize()
        for t in tickets:
            srv.release(t)
        return out
    if kind == "match":
        return state["ex"].match(state["a"], state["b"])
    if kind == "magsac":
        return state["ex"].magsac(state["xa"], state["xb"], state["samples"])
    return state["ex"].pyramid(state["img"])


def _octaves(case, h, w):
    up = 2 if case.get("upsample") and h * w <= 4000000 else 1
    h, w = h * up, w * up
    while min(h, w) >= 16:
        yield h, w
        h, w = h // 2, w // 2


def work(case):
    kind = case["kind"]
    if kind == "match":
        na, nb = case["na"], case["nb"]
        return {"bytes": 512 * (na + nb) + 4 * na, "flops": 2 * na * nb * 128}
    if kind == "magsac":  # about 1,500 operations for a model, 60 for a residual and its loss
        n, m = case["n"], case["n_hyp"]
        return {"bytes": 17 * n + 20 * m + 84, "flops": m * (1500 + 60 * n)}
    S = case.get("n_scales", 3)
    taps = sum(2 * math.ceil(4 * 1.6 * math.sqrt(4.0 ** (i / S) - 4.0 ** ((i - 1) / S))) + 1
               for i in range(1, S + 3))
    px_in = px = 0
    for h, w in _shapes(case):
        px_in += h * w
        px += sum(a * b for a, b in _octaves(case, h, w))
    flops = px * (4 * taps + S * 30)  # separable blurs; differences and comparisons
    if kind == "pyramid":
        return {"bytes": 4 * px_in + 4 * px * (S + 3), "flops": px * 4 * taps}
    # Features: about one in 1,500 pixels of an ordinary image, up to the cap on texture; each one
    # some 1,500 descriptor samples of 60 operations and 540 bytes out.
    rate = 1 / 400 if case["texture"] > 0.1 else 1 / 1500
    n = sum(min(case.get("max_kpts", 8192), a * b * (4 if case.get("upsample") else 1) * rate)
            for a, b in _shapes(case))
    return {"bytes": 4 * px_in + 540 * n, "flops": flops + n * 1500 * 60 * (4 if case.get("dsp") else 1)}


# ------------------------------------------------------------------ the same in 64 bits

def exact(case, seed):
    """Scale space, homography scores and, for images of moderate size, the whole list of
    features, in 64 bits. The lists of large images and batches have no such value: among
    thousands of features some comparison falls within FP32 rounding, and the list then has
    another length. Nor have the binary16 octaves, whose values depend on every rounding before.
    Matches are whole numbers."""
    kind = case["kind"]
    if kind == "magsac":
        return _exact_magsac(*_correspondences(case, seed))
    if kind not in ("pyramid", "extract") or case.get("fp16_pyramid"):
        return None
    if kind == "extract" and (case.get("dsp") or sum(a * b for a, b in _octaves(case, case["h"], case["w"])) > 4.5e5):
        return None
    pyr = _pyramid64(case, _images(case, seed)[0])
    return pyr if kind == "pyramid" else _features64(case, pyr)


def _exact_magsac(xa, xb, samples):
    a, b, s = (torch.from_numpy(np.ascontiguousarray(v)).cuda().double() for v in (xa, xb, samples))
    pa, pb = a[s.long()], b[s.long()]  # (hypotheses, 4, 2)

    def normalise(p):
        c = p.mean(1, keepdim=True)
        sc = math.sqrt(2.0) / (p - c).norm(dim=2).mean(1)
        T = torch.zeros(len(p), 3, 3, dtype=torch.float64, device=p.device)
        T[:, 0, 0] = T[:, 1, 1] = sc
        T[:, :2, 2] = -sc[:, None] * c[:, 0]
        T[:, 2, 2] = 1.0
        return (p - c) * sc[:, None, None], T

    def collinear(p):
        tri = ((0, 1, 2), (0, 1, 3), (0, 2, 3), (1, 2, 3))
        area = [((p[:, j, 0] - p[:, i, 0]) * (p[:, k, 1] - p[:, i, 1])
                 - (p[:, j, 1] - p[:, i, 1]) * (p[:, k, 0] - p[:, i, 0])).abs() / 2 for i, j, k in tri]
        return torch.stack(area).amin(0) < 1e-6

    (pa, Ta), (pb, Tb) = normalise(pa), normalise(pb)
    bad = collinear(pa) | collinear(pb)
    x, y, u, v = pa[..., 0], pa[..., 1], pb[..., 0], pb[..., 1]
    one, zero = torch.ones_like(x), torch.zeros_like(x)
    M = torch.cat([torch.stack([x, y, one, zero, zero, zero, -u * x, -u * y], -1),
                   torch.stack([zero, zero, zero, x, y, one, -v * x, -v * y], -1)], 1)
    M[bad] = torch.eye(8, dtype=torch.float64, device=M.device)
    h = torch.linalg.solve(M, torch.cat([u, v], 1)[..., None])[..., 0]
    H = torch.linalg.inv(Tb) @ torch.cat([h, torch.ones_like(h[:, :1])], 1).view(-1, 3, 3) @ Ta
    bad |= ~((h * h).sum(1) <= 1e18) | ~(H[:, 2, 2].abs() >= 1e-12 * H.abs().amax((1, 2)))
    H = H / H[:, 2:, 2:]
    # The loss: chi with 4 degrees of freedom, sigma uniform on (0, 1], truncated at the 0.99 quantile.
    yq = 6.0
    for _ in range(60):
        yq -= (math.exp(-yq) * (1 + yq) - 0.01) / (-math.exp(-yq) * yq)
    k2 = 2.0 * yq

    def g15(t):
        return 0.5 * math.sqrt(math.pi) * torch.erfc(t.sqrt()) + t.sqrt() * torch.exp(-t)

    def rho(r2):
        t = r2.clamp(max=k2) / 2
        g25 = 1.5 * g15(t) + t * t.sqrt() * torch.exp(-t)
        gk = g15(torch.tensor(k2 / 2, dtype=torch.float64, device=t.device))
        return 0.25 * 2.0 ** 1.5 * (0.75 * math.sqrt(math.pi) - g25 + t * (g15(t) - gk))

    q = torch.cat([a, torch.ones_like(a[:, :1])], 1)
    scores = []
    for part in H.split(256):
        w = q @ part.transpose(1, 2)
        r2 = (w[..., :2] / w[..., 2:] - b).square().sum(-1)
        scores.append(rho(torch.nan_to_num(r2, nan=math.inf)).sum(1))
    scores = torch.cat(scores)
    scores[bad] = math.inf
    best = int(scores.argmin())
    return {"H": H[best], "best": None, "score": scores[best:best + 1], "inliers": None, "scores": scores}


def _f32(v):
    return float(np.float32(v))


def _blur64(img, sigma):
    r = math.ceil(4 * sigma)
    w = torch.exp(-torch.arange(-r, r + 1, dtype=torch.float64, device=img.device) ** 2 / (2 * sigma * sigma))
    w = (w / w.sum()).tolist()
    h, wd = img.shape
    p = F.pad(img[None, None], (0, 0, r, r), mode="reflect")[0, 0]
    img = sum(w[j] * p[j:j + h] for j in range(2 * r + 1))
    p = F.pad(img[None, None], (r, r, 0, 0), mode="reflect")[0, 0]
    return sum(w[j] * p[:, j:j + wd] for j in range(2 * r + 1))


def _pyramid64(case, img):
    S, s0 = case.get("n_scales", 3), _f32(1.6)
    octs = list(_octaves(case, *img.shape))
    up = octs[0][0] != img.shape[0]
    g = img.double()
    for axis in (1, 0) if up else ():
        nxt = torch.cat([g.narrow(axis, 1, g.shape[axis] - 1), g.narrow(axis, g.shape[axis] - 1, 1)], axis)
        g = torch.stack([g, 0.5 * (g + nxt)], axis + 1).flatten(axis, axis + 1)
    sig = [s0 * 2.0 ** (i / S) for i in range(S + 3)]
    out = []
    for h, w in octs:
        if out:
            g = out[-1][S, 0:2 * h:2, 0:2 * w:2]
        else:
            g = _blur64(g, math.sqrt(s0 * s0 - (1.0 if up else 0.25)))
        levels = [g]
        for i in range(1, S + 3):
            levels.append(_blur64(levels[-1], math.sqrt(sig[i] ** 2 - sig[i - 1] ** 2)))
        out.append(torch.stack(levels))
    return out


def _refine64(D, s, y, x, S):
    """Up to five Newton steps per candidate; (kept, s, y, x, offsets, response)."""
    _, H, W = D.shape
    live = torch.ones_like(s, dtype=torch.bool)
    conv = torch.zeros_like(live)
    d = torch.zeros(len(s), 3, dtype=torch.float64, device=D.device)
    resp = torch.zeros(len(s), dtype=torch.float64, device=D.device)
    edge_ok = torch.zeros_like(live)
    for _ in range(5):
        def v(ds, dy, dx):
            return D[s + ds, y + dy, x + dx]
        c = v(0, 0, 0)
        g = torch.stack([v(0, 0, 1) - v(0, 0, -1), v(0, 1, 0) - v(0, -1, 0), v(1, 0, 0) - v(-1, 0, 0)], 1) / 2
        xx, yy, ss = (v(0, 0, 1) + v(0, 0, -1) - 2 * c, v(0, 1, 0) + v(0, -1, 0) - 2 * c,
                      v(1, 0, 0) + v(-1, 0, 0) - 2 * c)
        xy = (v(0, 1, 1) - v(0, 1, -1) - v(0, -1, 1) + v(0, -1, -1)) / 4
        xs = (v(1, 0, 1) - v(1, 0, -1) - v(-1, 0, 1) + v(-1, 0, -1)) / 4
        ys = (v(1, 1, 0) - v(1, -1, 0) - v(-1, 1, 0) + v(-1, -1, 0)) / 4
        Hs = torch.stack([xx, xy, xs, xy, yy, ys, xs, ys, ss], 1).view(-1, 3, 3)
        sing = torch.linalg.det(Hs) == 0
        Hs[sing] = torch.eye(3, dtype=torch.float64, device=D.device)
        step = torch.linalg.solve(Hs, -g)
        live &= ~sing
        done = live & (step.abs().amax(1) < 0.5)
        d[done] = step[done]
        resp[done] = (c + 0.5 * (g * step).sum(1))[done].abs()
        tr, dt = xx + yy, xx * yy - xy * xy
        edge_ok[done] = ((dt > 0) & (tr * tr * 10.0 < 121.0 * dt))[done]
        conv |= done
        live &= ~done
        move = (step.abs().clamp(max=1e7) + 0.5).floor() * step.sign()
        live &= step.abs().amax(1) <= 1e7
        nx, ny, ns = x + move[:, 0].long(), y + move[:, 1].long(), s + move[:, 2].long()
        live &= (ns >= 1) & (ns <= S) & (nx >= 5) & (nx < W - 5) & (ny >= 5) & (ny < H - 5)
        x, y, s = torch.where(live, nx, x), torch.where(live, ny, y), torch.where(live, ns, s)
    keep = conv & edge_ok & (resp >= _f32(_f32(0.04) / 3.0))
    return keep, s, y, x, d, resp


def _window(G, s, y, x, R, most):
    """Offsets (i, j) of the square of half side `most` and the gradients there; ok: inside each
    feature's own radius R and the image."""
    _, H, W = G.shape
    o = torch.arange(-most, most + 1, device=G.device)
    j, i = (t.reshape(1, -1) for t in torch.meshgrid(o, o, indexing="ij"))
    py, px = y[:, None] + j, x[:, None] + i
    ok = (i.abs() <= R[:, None]) & (j.abs() <= R[:, None]) & (px >= 1) & (px <= W - 2) & (py >= 1) & (py <= H - 2)
    py, px, sl = py.clamp(1, H - 2), px.clamp(1, W - 2), s[:, None]
    return i, j, ok, G[sl, py, px + 1] - G[sl, py, px - 1], G[sl, py + 1, px] - G[sl, py - 1, px]


def _orient64(G, s, y, x, sig):
    """(feature, angle in degrees) of every peak of the smoothed 36-bin histograms."""
    sw = 1.5 * sig
    R = (3.0 * sw + 0.5).floor().long()
    i, j, ok, gx, gy = _window(G, s, y, x, R, int(R.max()))
    th = torch.atan2(gy, gx) % (2 * math.pi)
    b = (36 * th / (2 * math.pi) + 0.5).floor().long() % 36
    q = torch.where(gy > 0, torch.where(gx > 0, 0, 1), torch.where(gx < 0, 2, 3))
    b = torch.where((gx.abs() == gy.abs()) & (gx != 0), (36 * (2 * q + 1) + 4) // 8 % 36, b)
    wt = torch.exp(-(i * i + j * j) / (2 * sw * sw)[:, None]) * torch.hypot(gx, gy) * ok
    h = torch.zeros(len(s), 36, dtype=torch.float64, device=G.device).scatter_add_(1, b, wt)
    h = 0.25 * h.roll(1, 1) + 0.5 * h + 0.25 * h.roll(-1, 1)
    hm, hp = h.roll(1, 1), h.roll(-1, 1)
    peak = (h > hm) & (h > hp) & (h >= _f32(0.8) * h.amax(1, keepdim=True))
    k, bin_ = peak.nonzero(as_tuple=True)
    a, c, e = hm[peak], h[peak], hp[peak]
    return k, ((bin_ + 0.5 * (a - e) / (a - 2 * c + e)) % 36) * 10.0


def _describe64(G, s, y, x, d, sig, ang):
    w = 3.0 * sig
    R = (w * math.sqrt(2.0) * 2.5 + 0.5).floor().long()
    i, j, ok, gx, gy = _window(G, s, y, x, R, int(R.max()))
    th = (ang * (math.pi / 180))[:, None]
    ox, oy = i - d[:, :1], j - d[:, 1:2]
    rx = (th.cos() * ox + th.sin() * oy) / w[:, None]
    ry = (-th.sin() * ox + th.cos() * oy) / w[:, None]
    u, v = rx + 1.5, ry + 1.5
    ok = ok & (u > -1) & (u < 4) & (v > -1) & (v < 4)
    o = ((torch.atan2(gy, gx) - th) % (2 * math.pi)) * (8 / (2 * math.pi))
    wt = torch.hypot(gx, gy) * torch.exp(-(rx * rx + ry * ry) / 8) * ok
    hist = torch.zeros(len(s), 128, dtype=torch.float64, device=G.device)
    for dv in (0, 1):
        for du in (0, 1):
            for do in (0, 1):
                uu, vv, oo = u.floor() + du, v.floor() + dv, o.floor() + do
                f = (1 - (u - uu).abs()) * (1 - (v - vv).abs()) * (1 - (o - oo).abs()) * wt
                f = f * ((uu >= 0) & (uu < 4) & (vv >= 0) & (vv < 4))
                at = (vv.clamp(0, 3) * 4 + uu.clamp(0, 3)) * 8 + oo % 8
                hist.scatter_add_(1, at.long(), f)
    return hist


def _features64(case, pyr):
    S, up = case.get("n_scales", 3), bool(case.get("upsample"))
    gate = 0.5 * _f32(_f32(0.04) / 3.0)
    rows = {k: [] for k in FIELDS}
    for o, G in enumerate(pyr):
        D = G[1:] - G[:-1]
        _, H, W = D.shape
        c = D[1:S + 1, 5:H - 5, 5:W - 5]
        near = torch.stack([D[1 + a:S + 1 + a, 5 + b:H - 5 + b, 5 + e:W - 5 + e] for a in (-1, 0, 1)
                            for b in (-1, 0, 1) for e in (-1, 0, 1) if (a, b, e) != (0, 0, 0)])
        hit = (c.abs() > gate) & ((c > near.amax(0)) | (c < near.amin(0)))
        s, y, x = hit.nonzero(as_tuple=True)
        if not len(s):
            continue
        keep, s, y, x, d, resp = _refine64(D, s + 1, y + 5, x + 5, S)
        s, y, x, d, resp = s[keep], y[keep], x[keep], d[keep], resp[keep]
        for at in torch.arange(len(s), device=G.device).split(128):
            sig = _f32(1.6) * 2.0 ** ((s[at] + d[at, 2]) / S)
            if case.get("upright"):
                k, ang = torch.arange(len(at), device=G.device), torch.zeros(len(at), dtype=torch.float64, device=G.device)
            else:
                k, ang = _orient64(G, s[at], y[at], x[at], sig)
            if not len(k):
                continue
            m, sig, scale = at[k], sig[k], 2.0 ** o * (0.5 if up else 1.0)
            hist = _describe64(G, s[m], y[m], x[m], d[m], sig, ang)
            for key, val in (("x", (x[m] + d[m, 0]) * scale), ("y", (y[m] + d[m, 1]) * scale),
                             ("sigma", sig * scale), ("angle", ang), ("response", resp[m]),
                             ("octave", torch.full_like(m, o)), ("layer", s[m]), ("desc", hist)):
                rows[key].append(val)
    if not rows["x"]:
        return None
    f = {k: torch.cat(v) for k, v in rows.items()}
    cap = case.get("max_kpts", 8192)
    if len(f["x"]) > cap:
        at = torch.sort(f["response"], descending=True, stable=True)[1][:cap].sort()[0]
        f = {k: v[at] for k, v in f.items()}
    d = F.normalize(F.normalize(f["desc"], dim=1).clamp(max=_f32(0.2)), dim=1)
    f["desc"] = (d / d.sum(1, keepdim=True).clamp(min=1e-300)).sqrt() if case.get("rootsift") else d
    out = {k: torch.zeros((1, cap) + v.shape[1:], dtype=v.dtype, device=v.device) for k, v in f.items()}
    for k, v in f.items():
        out[k][0, :len(v)] = v
    return {**out, "count": None}
