"""What the performance of this library is measured on.

Each case is one call (or one short sequence of calls) that a program using the package
makes, through its public entry points, at sizes taken from the repository's own configurations
(320x240, 481x321 with K = 1000, the uneven batch, 3840x2160, the learned start at
spacing 15) or, where drawn, spread over the ranges around them:

  single    Superpixels.segment on one image (CIELAB conversion, EM, labels)
  steps     the step-by-step calls on one image: reinit, em_iters, labels, get_params
  batch     SuperpixelsBatch.segment on a list of images (uneven, or one size)
  learned   SuperpixelsBatch.segment_stacked from the trained network's start
  forward   the network's forward pass on CIELAB images
  grad      one training step's loss and gradient
  connect   connectivity post-processing of a batch's label maps
  connect1  connectivity post-processing of one label map (the context-free call)
  metrics   BR, UE and ASA of label maps against ground-truth maps

Images are seeded Voronoi mosaics as the repository's generator draws them (a constant
colour and a linear gradient per region, Gaussian noise, rounded to 8 bits); label maps
for the post-processing and the metrics assign every pixel to one of its 3x3 seeds by
distance and colour, which gives the speckled boundaries that EM labels have.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_1612_08792_gb300 as gm
from paper_1612_08792_gb300 import learned_init

SIGMA = 8.0
BATCH_SIZES = [(320, 240), (481, 321), (640, 480), (1280, 720), (1920, 1080)]
METRIC_KEYS = ("br", "ue", "asa", "br_recovered", "br_total", "ue_sum", "asa_sum")


# ---------------------------------------------------------------- the cases
def listed():
    return [
        # the smallest configuration: one preview-sized image, launch latency counts; the
        # plain call, which allocates its label map
        dict(name="single_320x240", kind="single", W=320, H=240, K=0, spacing=12, iters=10, regions=40,
             colour="full", input="rgb8", loglik=False, out=False),
        # one photograph at the paper's size, K = 1000, with the log-likelihood trace, into
        # a label map that the program keeps (ragged: 481 and 321 are no multiples of 12)
        dict(name="single_481x321", kind="single", W=481, H=321, K=1000, spacing=0, iters=10, regions=150,
             colour="full", input="rgb8", loglik=True, out=True),
        # one 4K image, K = 20000: the largest single image
        dict(name="single_3840x2160", kind="single", W=3840, H=2160, K=20000, spacing=0, iters=10, regions=2000,
             colour="full", input="rgb8", loglik=False, out=True),
        # stepwise control of one odd-sized CIELAB image: reinit, EM with the log-likelihood
        # trace, labels, fitted parameters on the host
        dict(name="steps_641x479_lab", kind="steps", W=641, H=479, K=0, spacing=15, iters=10, regions=160),
        # a folder of images of five sizes in one batch context, tuned once, plain EM
        dict(name="batch_uneven_256", kind="batch", n=256, sizes="uneven", W=0, H=0, spacing=15, iters=10,
             colour="full", input="rgb8", loglik=False, tune=True),
        # grey-level images of one size, an untuned context, with log-likelihoods
        dict(name="batch_gray_640x480", kind="batch", n=64, sizes="one", W=640, H=480, spacing=15, iters=10,
             colour="gray", input="gray8", loglik=True, tune=False),
        # the learned start and 2 EM iterations on 256 photographs-sized images: the headline
        dict(name="learned_481x321_256", kind="learned", n=256, W=481, H=321, iters=2, tune=True),
        # the network alone: a training batch's forward pass
        dict(name="forward_481x321_32", kind="forward", n=32, W=481, H=321, spacing=15),
        # one training step's loss and gradient on the training batch
        dict(name="grad_481x321_32", kind="grad", n=32, W=481, H=321, spacing=15),
        # Algorithm 1, step 8 on a batch of label maps
        dict(name="connect_481x321_256", kind="connect", n=256, W=481, H=321, spacing=15),
        # the same on one label map, through the call that needs no context
        dict(name="connect1_481x321", kind="connect1", W=481, H=321, spacing=12),
        # the accuracy metrics of a batch of label maps
        dict(name="metrics_481x321_256", kind="metrics", n=256, W=481, H=321, spacing=15, regions=150),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _size(rng, lo, hi):
    """W, H of an image of lo .. hi pixels (logarithmic), any aspect from 3:4 to 16:9."""
    N = math.exp(rng.uniform(math.log(lo), math.log(hi)))
    a = rng.uniform(0.75, 16 / 9)
    return max(40, int(math.sqrt(N * a))), max(40, int(math.sqrt(N / a)))


def draw(rng):
    """One more case of the listed ones' ranges."""
    kind = rng.choice(["single", "steps", "batch", "learned", "forward", "grad", "connect", "connect1", "metrics"])
    if kind in ("single", "steps", "connect1"):
        W, H = _size(rng, 320 * 240, 3840 * 2160 if kind == "single" else 1920 * 1080)
        v = rng.randint(10, 24)
        c = dict(kind=kind, W=W, H=H, spacing=v)
        if kind != "connect1":
            c.update(K=0, iters=rng.randint(2, 10), regions=max(20, W * H // 2000))
        if kind == "single":
            c.update(colour="full", input=rng.choice(["rgb8", "lab32"]), loglik=rng.random() < 0.5,
                     out=rng.random() < 0.5)
        return c
    if kind in ("forward", "grad", "learned"):
        W, H = _size(rng, 96 * 64, 640 * 480)
        n = max(1, min(_log_int(rng, 1, 256), int(39.5e6 / (W * H)), 32 if kind == "grad" else 256))
        if kind == "learned":
            return dict(kind=kind, n=n, W=W, H=H, iters=rng.randint(1, 3), tune=False)
        return dict(kind=kind, n=n, W=W, H=H, spacing=rng.choice([9, 12, 15, 18, 21]))
    W, H = _size(rng, 160 * 120, 1280 * 720)
    n = max(1, min(_log_int(rng, 1, 256), int(39.5e6 / (W * H))))
    v = rng.randint(10, 24)
    if kind == "batch":
        colour = rng.choice(["full", "full", "split", "gray"])
        return dict(kind=kind, n=n, sizes=rng.choice(["one", "uneven"]) if n <= 64 else "one", W=W, H=H, spacing=v,
                    iters=rng.randint(2, 10), colour=colour,
                    input="gray8" if colour == "gray" else rng.choice(["rgb8", "lab32"]),
                    loglik=rng.random() < 0.5, tune=False)
    c = dict(kind=kind, n=n, W=W, H=H, spacing=v)
    if kind == "metrics":
        c.update(regions=_log_int(rng, 10, 400))
    return c


# ---------------------------------------------------------------- inputs
def _gen(seed, i=0):
    g = torch.Generator(device="cuda")
    g.manual_seed((int(seed) * 1_000_003 + 7919 * i + 17) % (1 << 62))
    return g


def _mosaic(W, H, regions, g, sigma=SIGMA, gray=False):
    """(image uint8 (H, W, 3) or (H, W), region map int32 (H, W)) on the device."""
    R = max(1, int(regions))
    u = torch.rand((R, 9), generator=g, device="cuda")
    sites = u[:, :2] * torch.tensor([W, H], device="cuda", dtype=torch.float32)
    base, angle, amp = 255.0 * u[:, 2:5], 2.0 * math.pi * u[:, 5], 30.0 * u[:, 6:9]
    x = torch.arange(W, device="cuda", dtype=torch.float32)
    y = torch.arange(H, device="cuda", dtype=torch.float32)
    reg = torch.empty((H, W), dtype=torch.int64, device="cuda")
    s2 = (sites ** 2).sum(1)
    rows = max(1, (1 << 28) // (W * R))
    for y0 in range(0, H, rows):  # nearest site, in bands of rows
        yy = y[y0:y0 + rows]
        p = torch.stack([x.expand(len(yy), W), yy[:, None].expand(len(yy), W)], -1).reshape(-1, 2)
        reg[y0:y0 + rows] = torch.addmm(s2, p, sites.T, alpha=-2.0).argmin(1).view(-1, W)
    s = sites[reg]
    proj = ((x - s[..., 0]) * torch.cos(angle)[reg] + (y[:, None] - s[..., 1]) * torch.sin(angle)[reg]) / max(W, H)
    if gray:
        img = base[reg, 0] + amp[reg, 0] * proj
    else:
        img = base[reg] + amp[reg] * proj[..., None]
    img = img + sigma * torch.randn(img.shape, generator=g, device="cuda")
    return img.round_().clamp_(0, 255).to(torch.uint8), reg.to(torch.int32)


_PRIM = [[0.64, 0.33], [0.30, 0.60], [0.15, 0.06]]
_WHITE = [0.95047, 1.0, 1.08883]


def _to_lab(rgb, dtype):
    """CIELAB (D65) of sRGB code values (..., 3), or L* (...) of grey levels."""
    c = rgb.to(dtype) / 255.0
    lin = torch.where(c <= 0.04045, c / 12.92, ((c + 0.055) / 1.055) ** 2.4)

    def f(t):
        return torch.where(t > 216.0 / 24389.0, t.clamp_min(1e-12) ** (1.0 / 3.0), (841.0 / 108.0) * t + 4.0 / 29.0)

    if rgb.dim() == 2:
        return 116.0 * f(lin) - 16.0
    P = np.array([[x / y, 1.0, (1.0 - x - y) / y] for x, y in _PRIM]).T
    M = P * np.linalg.solve(P, np.array(_WHITE))
    xyz = lin @ torch.tensor((M / np.array(_WHITE)[:, None]).T, dtype=dtype, device=rgb.device)
    t = f(xyz)
    return torch.stack([116.0 * t[..., 1] - 16.0, 500.0 * (t[..., 0] - t[..., 1]), 200.0 * (t[..., 1] - t[..., 2])], -1)


def _image(case, seed, i=0, W=0, H=0, regions=0):
    """Image i of a case in its input format."""
    fmt = case.get("input", "lab32" if case["kind"] == "steps" else "rgb8")
    W, H = W or case["W"], H or case["H"]
    img, _ = _mosaic(W, H, regions or case.get("regions") or max(4, W * H // 1030), _gen(seed, i), gray=fmt == "gray8")
    return _to_lab(img, torch.float32).contiguous() if fmt == "lab32" else img


def _batch_sizes(case, seed):
    if case["sizes"] == "one":
        return [(case["W"], case["H"])] * case["n"]
    rng = np.random.default_rng(12345 + case["n"])  # the sizes belong to the case, the images to the seed
    if not case["W"]:
        return [BATCH_SIZES[j] for j in rng.integers(0, len(BATCH_SIZES), case["n"])]
    return [(max(40, int(case["W"] * a)), max(40, int(case["H"] * b)))
            for a, b in zip(rng.uniform(0.5, 1.0, case["n"]), rng.uniform(0.5, 1.0, case["n"]))]


def _batch_images(case, seed):
    return [_image(case, seed, i, W, H, max(1, round(40 * W * H / 76800)))
            for i, (W, H) in enumerate(_batch_sizes(case, seed))]


def _lab_planes(case, seed):
    """(n, 3, H, W) float32 CIELAB planes."""
    n, W, H = case["n"], case["W"], case["H"]
    out = torch.empty((n, 3, H, W), dtype=torch.float32, device="cuda")
    for i in range(n):
        out[i] = _to_lab(_mosaic(W, H, max(4, W * H // 1030), _gen(seed, i))[0], torch.float32).permute(2, 0, 1)
    return out


def _targets(case, seed):
    """Training targets of the distribution that fitted parameters have: mean offsets of a
    fraction of a cell and of a few colour units, log covariance diagonals below the start's."""
    n, v = case["n"], case["spacing"]
    K = (case["W"] // v) * (case["H"] // v)
    mean = torch.tensor([0.0, 0.0, 0.0, 0.0, 0.0, -1.6, -1.6, -1.4, -1.4, -1.4], device="cuda")
    std = torch.tensor([0.25, 0.25, 0.3, 0.55, 0.55, 0.35, 0.35, 0.3, 0.3, 0.3], device="cuda")
    return mean + std * torch.randn((n * K, 10), generator=_gen(seed, 1 << 20), device="cuda")


def _seed_labels(planes, v):
    """(n, H, W) int32: every pixel's nearest of its 3x3 seeds (distance over v, colour over 20: as many
    components as the labels of a fitted model have)."""
    n, _, H, W = planes.shape
    nx, ny = W // v, H // v
    ys, xs = torch.arange(H, device="cuda"), torch.arange(W, device="cuda")
    cx, cy = xs // v, ys // v
    best = torch.full((n, H, W), float("inf"), device="cuda")
    lab = torch.zeros((n, H, W), dtype=torch.int32, device="cuda")
    for dy in (-1, 0, 1):
        for dx in (-1, 0, 1):
            kx, ky = cx + dx, cy + dy
            ok = ((ky >= 0) & (ky < ny))[:, None] & ((kx >= 0) & (kx < nx))[None, :]
            kx, ky = kx.clamp(0, nx - 1), ky.clamp(0, ny - 1)
            px, py = kx * v + v // 2, ky * v + v // 2
            d = ((xs - px).float() / v) ** 2 + (((ys - py).float() / v) ** 2)[:, None]
            d = d + ((planes - planes[:, :, py][:, :, :, px]) ** 2).sum(1) / 400.0
            d = torch.where(ok, d, torch.full_like(d, float("inf")))
            near = d < best
            best = torch.where(near, d, best)
            lab = torch.where(near, (ky[:, None] * nx + kx[None, :]).to(torch.int32), lab)
    return lab


# ---------------------------------------------------------------- prepare and run
def prepare(case, seed):
    """The inputs and the context of one case; every case but the training ones (which follow
    learned_init.train) and the grey batch runs on a stream of its own, as the library's graphs want."""
    kind = case["kind"]
    default = kind in ("forward", "grad") or (kind == "batch" and not case["tune"])
    stream = torch.cuda.default_stream() if default else torch.cuda.Stream()
    st = dict(case=dict(case), stream=stream)
    with torch.cuda.stream(stream):
        if kind in ("single", "steps"):
            st["image"] = _image(case, seed)
            st["sp"] = gm.Superpixels(st["image"], K=case["K"], spacing=case["spacing"], stream=stream,
                                      colour=case.get("colour", "full"))
            shape = (case["H"], case["W"])
            st["out"] = torch.empty(shape, dtype=torch.int32, device="cuda") if case.get("out", True) else None
        elif kind == "batch":
            st["images"] = _batch_images(case, seed)
            st["bt"] = gm.SuperpixelsBatch([(H, W) for W, H in _batch_sizes(case, seed)], spacing=case["spacing"],
                                           stream=stream, colour=case["colour"], gray_input=case["input"] == "gray8",
                                           lab_input=case["input"] == "lab32")
            if case["tune"]:
                st["bt"].autotune(st["images"])
        elif kind == "learned":
            n, W, H = case["n"], case["W"], case["H"]
            st["images"] = torch.stack([_image(case, seed, i) for i in range(n)])
            st["net"] = learned_init.load_pretrained(15, stream=stream)
            st["bt"] = gm.SuperpixelsBatch([(H, W)] * n, spacing=15, stream=stream)
            if case["tune"]:
                st["bt"].autotune(list(st["images"]))
            st["bt"].set_init_net(st["net"])
        elif kind in ("forward", "grad"):
            st["lab"] = _lab_planes(case, seed)
            st["net"] = learned_init.InitNet(case["spacing"], weights=_weights(seed), stream=stream)
            if kind == "grad":
                st["target"] = _targets(case, seed)
        elif kind == "connect":
            n, W, H, v = case["n"], case["W"], case["H"], case["spacing"]
            planes = torch.empty((n, 3, H, W), dtype=torch.float32, device="cuda")
            images = torch.empty((n, H, W, 3), dtype=torch.uint8, device="cuda")
            for i in range(n):
                images[i] = _image(case, seed, i)
                planes[i] = _to_lab(images[i], torch.float32).permute(2, 0, 1)
            st["labels"] = _seed_labels(planes, v).view(-1)
            st["bt"] = gm.SuperpixelsBatch([(H, W)] * n, spacing=v, stream=stream)
            st["bt"].segment_stacked(images, iters=0)  # the context's CIELAB image; its labels are replaced
            torch.cuda.synchronize()
        elif kind == "connect1":
            st["lab"] = _lab_planes(dict(case, n=1), seed)
            st["labels"] = _seed_labels(st["lab"], case["spacing"])[0]
        elif kind == "metrics":
            n, W, H, v = case["n"], case["W"], case["H"], case["spacing"]
            planes, gts = _lab_and_regions(case, seed)
            st["labels"], st["gts"] = list(_seed_labels(planes, v)), list(gts)
            st["K"] = (W // v) * (H // v)
    torch.cuda.synchronize()
    return st


def _lab_and_regions(case, seed):
    n, W, H = case["n"], case["W"], case["H"]
    planes = torch.empty((n, 3, H, W), dtype=torch.float32, device="cuda")
    gts = torch.empty((n, H, W), dtype=torch.int32, device="cuda")
    for i in range(n):
        img, gts[i] = _mosaic(W, H, case["regions"], _gen(seed, i))
        planes[i] = _to_lab(img, torch.float32).permute(2, 0, 1)
    return planes, gts


def _weights(seed):
    """Parameters as training starts from them (He-normal, a small last layer, small biases)."""
    rng = np.random.default_rng(seed)
    w = []
    for layer, (taps, cout) in enumerate(((1, 32), (1, 32), (9, 32), (9, 32), (9, 32), (9, 16))):
        W = rng.normal(0.0, math.sqrt(2.0 / (27 if layer == 0 else taps * 32)), (cout, taps * 32))
        if layer == 0:
            W[:, 27:] = 0.0
        w += [(W * (0.1 if layer == 5 else 1.0)).ravel(), rng.normal(0.0, 0.02, cout)]
    return np.concatenate(w).astype(np.float32)


def run(st):
    case = st["case"]
    kind = case["kind"]
    with torch.cuda.stream(st["stream"]):
        if kind == "single":
            r = st["sp"].segment(st["image"], case["iters"], out=st["out"], want_loglik=case["loglik"])
            return dict(labels=r[0], loglik=r[1]) if case["loglik"] else dict(labels=r)
        if kind == "steps":
            sp = st["sp"]
            sp.reinit(st["image"])
            trace = sp.em_iters(case["iters"], want_loglik=True)
            labels, last = sp.labels(out=st["out"], want_loglik=True)
            mu, cov_s, cov_c = sp.get_params()
            return dict(labels=labels, trace=trace, last=last, mu=mu, cov_s=cov_s, cov_c=cov_c)
        if kind == "batch":
            bt = st["bt"]
            r = bt.segment(st["images"], case["iters"], want_loglik=case["loglik"])
            return dict(labels=bt.labels_buffer, loglik=r[1]) if case["loglik"] else dict(labels=bt.labels_buffer)
        if kind == "learned":
            st["bt"].segment_stacked(st["images"], case["iters"])
            return dict(labels=st["bt"].labels_buffer)
        if kind == "forward":
            return dict(out=st["net"].forward(st["lab"], case["n"], case["W"], case["H"]))
        if kind == "grad":
            loss, g = st["net"].grad(st["lab"], case["n"], case["W"], case["H"], st["target"])
            return dict(loss=loss, grad=g)
        if kind == "connect":
            bt = st["bt"]
            bt.labels_buffer.copy_(st["labels"])  # the call works in place
            stats = bt.connectivity()
            return dict(labels=bt.labels_buffer, **stats)
        if kind == "connect1":
            labels = st["labels"].clone()
            v = case["spacing"]
            stats = gm.gmmsp_enforce_connectivity(labels, st["lab"], case["W"], case["H"],
                                                  (case["W"] // v) * (case["H"] // v))
            return dict(labels=labels, **stats)
        res = gm.gmmsp_segmentation_metrics_many(st["labels"], st["gts"], st["K"], case["regions"])
        return dict(table=np.array([tuple(m.values()) for m in res]))


# ---------------------------------------------------------------- work
def _candidates(W, H, v):
    """Sum over the pixels of the number of candidate superpixels."""
    def axis(extent, n):
        full = sum((c > 0) + 1 + (c + 1 < n) for c in range(n)) * v
        return full + (extent - n * v)
    return axis(W, W // v) * axis(H, H // v)


def _spacing(case, W, H):
    return case["spacing"] or int(math.isqrt(W * H // case["K"]))


def _em_work(case, sizes, start_flops=0.0):
    """Each image read once and each label written once; per pixel and candidate 61 operations
    of an EM iteration (density, posterior, moments) and 29 of the label pass."""
    per = {"full": (61, 29), "split": (53, 25), "gray": (33, 15)}[case.get("colour", "full")]
    px = {"rgb8": 3, "gray8": 1, "lab32": 12}[case.get("input", "lab32" if case["kind"] == "steps" else "rgb8")]
    pixels = sum(W * H for W, H in sizes)
    cand = sum(_candidates(W, H, _spacing(case, W, H)) for W, H in sizes)
    return dict(bytes=(px + 4) * pixels, flops=start_flops + cand * (per[0] * case["iters"] + per[1]))


def _net_flops(cells, v):
    return cells * ((v // 3) ** 2 * 2 * (27 + 32) * 32 + 2 * 288 * (3 * 32 + 16))


def work(case):
    kind = case["kind"]
    if kind in ("single", "steps"):
        w = _em_work(case, [(case["W"], case["H"])])
        if kind == "steps":
            v = case["spacing"]
            w["bytes"] += (case["W"] // v) * (case["H"] // v) * 14 * 8
        return w
    if kind == "batch":
        return _em_work(case, _batch_sizes(case, 0))
    n, W, H = case.get("n", 1), case["W"], case["H"]
    v = case.get("spacing", 15)
    cells, N = n * (W // v) * (H // v), n * W * H
    if kind == "learned":
        return _em_work(dict(case, spacing=15), [(W, H)] * n, _net_flops(cells, 15))
    if kind == "forward":
        return dict(bytes=12 * N + 64 * cells + 4 * 34480, flops=_net_flops(cells, v))
    if kind == "grad":
        return dict(bytes=12 * N + 40 * cells + 8 * 34480, flops=3 * _net_flops(cells, v))
    if kind in ("connect", "connect1"):
        return dict(bytes=(4 + 12 + 4) * N, flops=0)
    return dict(bytes=8 * N, flops=0)


# ---------------------------------------------------------------- the same in 64 bits
def _em64(lab, v, iters, gray=False, eps_s=2.0, eps_c=8.0, lam=8.0):
    """Plain EM of one image in float64: lab (H, W, C) -> (loglik trace, mu, cov_s, cov_c)."""
    H, W, C = lab.shape
    nx, ny = W // v, H // v
    K = nx * ny
    dev = lab.device
    y, x = torch.meshgrid(torch.arange(H, device=dev), torch.arange(W, device=dev), indexing="ij")
    z = torch.cat([x.reshape(-1, 1).double(), y.reshape(-1, 1).double(), lab.reshape(-1, C).double()], 1)
    cx, cy = (x // v).reshape(-1), (y // v).reshape(-1)
    slots = []
    for dy in (-1, 0, 1):
        for dx in (-1, 0, 1):
            kx, ky = cx + dx, cy + dy
            i = torch.nonzero((kx >= 0) & (kx < nx) & (ky >= 0) & (ky < ny)).view(-1)
            slots.append((i, (ky * nx + kx)[i]))
    k = torch.arange(K, device=dev)
    px, py = (k % nx) * v + v // 2, (k // nx) * v + v // 2
    mu = torch.cat([px[:, None].double(), py[:, None].double(), lab[py, px].double()], 1)
    cs = torch.diag(torch.tensor([float(v * v)] * 2, dtype=torch.float64, device=dev)).expand(K, 2, 2)
    cc = torch.diag(torch.tensor([lam * lam] * C, dtype=torch.float64, device=dev)).expand(K, C, C)
    blocks = [(0, 2, eps_s), (2, 2 + C, eps_c)]
    trace = []
    for t in range(iters + 1):
        inv = [torch.linalg.inv(c) for c in (cs, cc)]
        norm = -0.5 * ((2 + C) * math.log(2 * math.pi) + torch.logdet(cs) + torch.logdet(cc))
        logp = torch.full((9, H * W), float("-inf"), dtype=torch.float64, device=dev)
        for s, (i, kk) in enumerate(slots):
            d = z[i] - mu[kk]
            q = norm[kk]
            for (a, b, _), P in zip(blocks, inv):
                q = q - 0.5 * torch.einsum("pi,pij,pj->p", d[:, a:b], P[kk], d[:, a:b])
            logp[s, i] = q
        lse = torch.logsumexp(logp, 0)
        trace.append(float(lse.sum()))
        if t == iters:
            break
        Wk = torch.zeros(K, dtype=torch.float64, device=dev)
        S1 = torch.zeros((K, 2 + C), dtype=torch.float64, device=dev)
        for s, (i, kk) in enumerate(slots):
            r = torch.exp(logp[s, i] - lse[i])
            Wk.index_add_(0, kk, r)
            S1.index_add_(0, kk, r[:, None] * (z[i] - mu[kk]))
        new = mu + S1 / Wk[:, None]
        S2 = [torch.zeros((K, b - a, b - a), dtype=torch.float64, device=dev) for a, b, _ in blocks]
        for s, (i, kk) in enumerate(slots):
            r = torch.exp(logp[s, i] - lse[i])
            d = z[i] - new[kk]
            for (a, b, _), S in zip(blocks, S2):
                S.index_add_(0, kk, r[:, None, None] * d[:, a:b, None] * d[:, None, a:b])
        mu = new
        out = []
        for (a, b, eps), S in zip(blocks, S2):
            if b - a == 1:
                out.append((S / Wk[:, None, None]).clamp_min(eps))
                continue
            e, V = torch.linalg.eigh((S / Wk[:, None, None]).cpu())
            out.append((V @ (e.clamp_min(eps)[..., None] * V.transpose(1, 2))).to(dev))
        cs, cc = out
    return np.array(trace), mu, cs, cc


def _lab64(case, image):
    if image.dtype == torch.float32:
        return image.double()
    lab = _to_lab(image, torch.float64)
    return lab[..., None] if lab.dim() == 2 else lab


def _net64(case, seed, want_grad):
    n, W, H, v = case["n"], case["W"], case["H"], case["spacing"]
    f, nx, ny = v // 3, W // v, H // v
    lab = _lab_planes(case, seed).double()
    flat = torch.tensor(_weights(seed), dtype=torch.float64, device="cuda", requires_grad=want_grad)
    scaled = lab[:, :, :ny * v, :nx * v] * 0.02 - torch.tensor([1.0, 0.0, 0.0], dtype=torch.float64,
                                                                device="cuda")[None, :, None, None]
    p = scaled.view(n, 3, ny, f, 3, nx, f, 3).permute(0, 2, 5, 3, 6, 4, 7, 1).reshape(n, ny, nx, f * f, 27)
    layers, o = [], 0
    for taps, cout in ((1, 32), (1, 32), (9, 32), (9, 32), (9, 32), (9, 16)):
        Wl = flat[o:o + cout * taps * 32].view(cout, taps, 32)
        o += cout * taps * 32
        layers.append((Wl, flat[o:o + cout]))
        o += cout
    h = torch.relu(p @ layers[0][0][:, 0, :27].T + layers[0][1])
    h = torch.relu(h @ layers[1][0][:, 0].T + layers[1][1]).mean(3)
    c = v // 2
    start = scaled[:, :, c::v, c::v].permute(0, 2, 3, 1)
    a = torch.cat([h[..., :29], start], -1).permute(0, 3, 1, 2)
    for l in range(2, 6):
        Wl, b = layers[l]
        pad = torch.nn.functional.pad(a, (1, 1, 1, 1))
        y = b[None, :, None, None]
        for t in range(9):
            win = pad[:, :, t // 3:t // 3 + ny, t % 3:t % 3 + nx]
            y = y + torch.einsum("bchw,oc->bohw", win, Wl[:, t])
        a = torch.relu(y) if l < 5 else y
    out = a.permute(0, 2, 3, 1)
    if not want_grad:
        return dict(out=out.detach())
    loss = ((out[..., :10].reshape(-1, 10) - _targets(case, seed).double()) ** 2).mean()
    loss.backward()
    return dict(loss=float(loss), grad=flat.grad.cpu().numpy())


def _metrics64(case, seed, radius=2, eps=0.05):
    planes, gts = _lab_and_regions(case, seed)
    n, W, H, v, G = case["n"], case["W"], case["H"], case["spacing"], case["regions"]
    labels, K = _seed_labels(planes, v), (W // v) * (H // v)
    rows = []
    for i in range(n):
        lab, gt = labels[i].long(), gts[i].long()

        def boundary(m):
            b = torch.zeros((H, W), dtype=torch.bool, device="cuda")
            d = m[:, 1:] != m[:, :-1]
            b[:, 1:] |= d
            b[:, :-1] |= d
            d = m[1:] != m[:-1]
            b[1:] |= d
            b[:-1] |= d
            return b
        near = torch.nn.functional.max_pool2d(boundary(lab)[None, None].float(), 2 * radius + 1, 1, radius)[0, 0] > 0
        gb = boundary(gt)
        rec, tot = int((gb & near).sum()), int(gb.sum())
        tab = torch.bincount((lab * G + gt).view(-1), minlength=K * G).view(K, G)
        size = tab.sum(1)
        ue = int(((tab.double() > eps * size.double()[:, None]).sum(1) * size).sum())
        asa = int(tab.max(1).values.sum())
        rows.append((rec / tot if tot else 1.0, ue / (W * H) - 1.0, asa / (W * H), rec, tot, ue, asa))
    return dict(table=np.array(rows, dtype=np.float64))


def exact(case, seed):
    kind = case["kind"]
    if kind == "single" and case["loglik"] and case["W"] * case["H"] <= 2_500_000:
        lab = _lab64(case, _image(case, seed))
        trace, *_ = _em64(lab, _spacing(case, case["W"], case["H"]), case["iters"])
        return dict(labels=None, loglik=trace)
    if kind == "steps":
        trace, mu, cs, cc = _em64(_lab64(case, _image(case, seed)), case["spacing"], case["iters"])
        iu2, iu3 = torch.triu_indices(2, 2), torch.triu_indices(3, 3)
        return dict(labels=None, trace=trace[:-1], last=float(trace[-1]), mu=mu, cov_s=cs[:, iu2[0], iu2[1]],
                    cov_c=cc[:, iu3[0], iu3[1]])
    if kind == "batch" and case["loglik"] and case["colour"] != "split":
        sizes = _batch_sizes(case, seed)
        if sum(W * H for W, H in sizes) > 25_000_000:
            return None
        lls = [_em64(_lab64(case, im), case["spacing"], case["iters"])[0][-1] for im in _batch_images(case, seed)]
        return dict(labels=None, loglik=np.array(lls))
    if kind in ("forward", "grad"):
        return _net64(case, seed, kind == "grad")
    if kind == "metrics":
        return _metrics64(case, seed)
    return None
