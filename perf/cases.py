"""The work that programs have this library do, as measurable cases.

A case is one pass through the public entry points of ``paper_1504_01883_gb300.binding``, on
inputs that are on the GPU beforehand, with the context, the packed model and the tracking state
that a program keeps between passes:

  features   face rects of RGB-D frames -> LBP histogram rows and normalised rows
  frame      the per-frame path: features, scores and labels, and for a camera stream identities
  score      normalised rows against a packed SVM
  normalise  stored count rows -> normalised rows (a face database read back)
  train      one-vs-rest RBF SVM training on normalised rows
  roi        colour-detected boxes -> depth-space rects -> exported crops

Sizes are those of the repository's workloads and tests (640x480 frames, faces of side 48..256,
128x128 crops of 16x16 cells, 512 to 8192 support vectors, 5 to 128 classes) and odd ones of the
same ranges.  Frames hold smooth grey with blobs and noise, and an ellipsoid face in front of a
far background with 2 % holes.  Count rows have identity structure (Poisson counts around each
identity's own rates) and models have the form that training gives: sparse, box-bounded
coefficients that sum to zero per class, and a negative bias.
"""
import math

import numpy as np
import torch

from paper_1504_01883_gb300 import binding as B

BINS = 59
IDENTITIES = 64
X_SCALE = 448.0
MASK_MM = 150
ELEM = {"f32": 4, "tf32": 4, "bf16": 2, "fp8": 1, "bf16x3": 4}


def listed():
    return [
        # one already cut 64x64 face against a 5-person linear model: the smallest request, all latency
        dict(name="crop64-linear", kind="frame", frames=1, height=64, width=64, faces=1, smin=64, smax=64, crop=64,
             precut=True, dtype="f32", svs=0, classes=5, track=False, flat=False),
        # one camera frame with four faces, exact fp32 scores against a small database
        dict(name="frame-f32", kind="frame", frames=1, height=480, width=640, faces=4, smin=80, smax=200, crop=128,
             precut=False, dtype="f32", svs=512, classes=10, track=False, flat=True),
        # one frame of a live camera stream against the resident serving model, identities tracked
        dict(name="frame-serve-bf16", kind="frame", frames=1, height=480, width=640, faces=7, smin=48, smax=256,
             crop=128, precut=False, dtype="bf16", svs=8192, classes=64, track=True, flat=False),
        # a recording featurised in bulk: counts to store, bf16 rows to score
        dict(name="features-batch-bf16", kind="features", frames=256, height=480, width=640, faces=16, smin=48,
             smax=256, crop=128, dtype="bf16", flags=0, counts=True),
        # odd frame width, small to very large faces, the >= and ignore-mask options, FP8 rows
        dict(name="features-odd-fp8", kind="features", frames=45, height=240, width=322, faces=13, smin=20, smax=300,
             crop=96, dtype="fp8", flags=3, counts=True),
        # the paper's own descriptor: one 256-bin histogram of each 200x200 face
        dict(name="features-face256", kind="features", frames=64, height=480, width=640, faces=9, smin=48, smax=256,
             crop=200, dtype="f32", flags=4, counts=True),
        # a full batch of faces against a full database
        dict(name="score-batch-bf16", kind="score", rows=4096, svs=4096, classes=64, crop=128, dtype="bf16",
             centred=False, flat=True),
        # a burst of queued frames: more rows than one tile of them, few for the chip, centred FP8 model
        dict(name="score-burst-fp8", kind="score", rows=300, svs=8190, classes=64, crop=128, dtype="fp8",
             centred=True, flat=False),
        # exact fp32 scores of a set of faces, odd sizes
        dict(name="score-exact-f32", kind="score", rows=777, svs=3001, classes=50, crop=128, dtype="f32",
             centred=False, flat=False),
        # stored count rows of a database normalised for scoring or packing
        dict(name="normalise-bf16", kind="normalise", rows=8192, crop=128, dtype="bf16"),
        # all classifiers of a 64-person database trained from 64 views each
        dict(name="train-64x64", kind="train", rows=4096, classes=64, crop=128),
        # colour-detected faces of a recording found in the depth frames and cut out for export
        dict(name="roi-crop", kind="roi", frames=256, height=480, width=640, faces=16, smin=48, smax=256, crop=128),
    ]


# ---------------------------------------------------------------------------------------------
# More cases of the same ranges
# ---------------------------------------------------------------------------------------------

def _log(rng, lo, hi):
    """A whole number of lo..hi, spread over its logarithm."""
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def _camera(rng):
    return rng.choice([(480, 640), (480, 640), (240, 320), (240, 322), (424, 512), (200, 318), (481, 639)])


def draw(rng):
    kind = rng.choice(["features", "features", "frame", "frame", "score", "score", "score", "normalise", "train",
                       "roi"])
    dtype = rng.choice(["f32", "bf16", "bf16", "fp8", "tf32", "bf16x3"])
    crop = rng.choice([32, 64, 96, 128, 128])
    dim = (crop // 8) ** 2 * BINS
    if kind == "features":
        h, w = _camera(rng)
        frames, faces = _log(rng, 1, 200), _log(rng, 1, 20)
        smin = _log(rng, 16, 96)
        flags = rng.choice([0, 0, 0, 1, 2, 3, 4])
        if flags == 4:
            crop, frames = rng.choice([200, 200, 57, 128, 255]), min(frames, 60)
        return dict(kind=kind, frames=frames, height=h, width=w, faces=faces, smin=smin, smax=_log(rng, smin, 300),
                    crop=crop, dtype=dtype, flags=flags, counts=rng.random() < 0.5)
    if kind == "frame":
        h, w = _camera(rng)
        smin = _log(rng, 40, 96)
        track = rng.random() < 0.5
        return dict(kind=kind, frames=1 if not track else _log(rng, 1, 6), height=h, width=w, faces=_log(rng, 1, 12),
                    smin=smin, smax=_log(rng, smin, 256), crop=crop, precut=False, dtype=dtype,
                    svs=_log(rng, 100, 8192), classes=_log(rng, 2, 128), track=track, flat=rng.random() < 0.5)
    if kind == "score":
        rows, svs, classes = _log(rng, 1, 6000), _log(rng, 200, 12000), _log(rng, 2, 128)
        most = {"f32": 6.5e10, "tf32": 2.4e11, "bf16x3": 1.6e11}.get(dtype, 5e11)
        rows = max(1, min(rows, int(most / (2.0 * svs * (dim + classes)))))
        return dict(kind=kind, rows=rows, svs=svs, classes=classes, crop=crop, dtype=dtype,
                    centred=rng.random() < 0.4, flat=rng.random() < 0.5)
    if kind == "normalise":
        return dict(kind=kind, rows=_log(rng, 50, 8000), crop=crop, dtype=dtype)
    if kind == "train":
        classes = _log(rng, 3, 64)
        return dict(kind=kind, rows=_log(rng, max(128, 4 * classes), 4000), classes=classes, crop=crop)
    h, w = _camera(rng)
    smin = _log(rng, 24, 96)
    return dict(kind=kind, frames=_log(rng, 1, 256), height=h, width=w, faces=_log(rng, 1, 16), smin=smin,
                smax=_log(rng, smin, 256), crop=rng.choice([64, 96, 128, 100]))


# ---------------------------------------------------------------------------------------------
# Inputs
# ---------------------------------------------------------------------------------------------

def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed) * 7919 + 17)
    return g


def _rand(g, lo, hi, *shape):
    return torch.rand(shape, generator=g, device="cuda") * (hi - lo) + lo


def _frames(case, g):
    """Grey uint8 and depth int16 (uint16 bits) [F][H][W], and int32 rects [F * faces][5]: square
    rects whose centres lie in the frame, a face under each."""
    F, H, W, n = case["frames"], case["height"], case["width"], case["faces"]
    side = torch.randint(case["smin"], case["smax"] + 1, (F, n), generator=g, device="cuda")
    cx = torch.randint(0, W, (F, n), generator=g, device="cuda")
    cy = torch.randint(0, H, (F, n), generator=g, device="cuda")
    if case.get("precut"):
        cx, cy = torch.full_like(cx, W // 2), torch.full_like(cy, H // 2)
    frame = torch.arange(F, device="cuda")[:, None].expand(F, n)
    rects = torch.stack([frame, cx - side // 2, cy - side // 2, side, side], 2).reshape(-1, 5).int().contiguous()
    yy = torch.arange(H, device="cuda", dtype=torch.float32)[None, :, None]
    xx = torch.arange(W, device="cuda", dtype=torch.float32)[None, None, :]
    x0, y0, s = (cx - side // 2).float(), (cy - side // 2).float(), side.float()
    p = _rand(g, 0, 1, 4, F, 1, 1)
    r = torch.sqrt((xx - W * (0.375 + p[0] / 4)) ** 2 + (yy - H * (0.375 + p[1] / 4)) ** 2) / (0.5 * max(H, W))
    grey = 60 + 100 * p[2] + (30 + 50 * p[3]) * (1 - r)
    depth = _rand(g, 2500, 4000, F, H, W)
    for k in range(n):
        def at(v):
            return v[:, k].reshape(F, 1, 1)
        for _ in range(6):  # blobs
            b = _rand(g, 0, 1, 4, F, 1, 1)
            bx, by = at(x0) + (0.1 + 0.8 * b[0]) * at(s), at(y0) + (0.1 + 0.8 * b[1]) * at(s)
            sig = (3 + 5 * b[2]) * at(s) / 64
            gx = torch.exp(-((xx - bx) ** 2) / (2 * sig * sig))
            gy = torch.exp(-((yy - by) ** 2) / (2 * sig * sig)) * (140 * b[3] - 70)
            grey = grey.addcmul_(gx.expand(F, H, W), gy.expand(F, H, W))
        e = _rand(g, 0, 1, 4, F, 1, 1)
        rho = ((xx + 0.5 - at(x0) - at(s) / 2) / ((0.42 + 0.08 * e[0]) * at(s))) ** 2
        rho = rho + ((yy + 0.5 - at(y0) - at(s) / 2) / ((0.42 + 0.08 * e[1]) * at(s))) ** 2
        surf = 1000 + 100 * e[2] - (60 + 40 * e[3]) * torch.sqrt((1 - rho).clamp_(min=0))
        depth = torch.where(rho < 1, torch.minimum(depth, surf), depth)
    grey = (grey + 8 * torch.randn((F, H, W), generator=g, device="cuda")).round_().clamp_(0, 255).to(torch.uint8)
    depth = depth.round_().masked_fill_(torch.rand((F, H, W), generator=g, device="cuda") < 0.02, 0)
    return grey, depth.to(torch.int16).contiguous(), rects


def _counts(g, n, dim, owner, protos):
    """Count rows (int16 storage) of faces of the identities `owner`."""
    out = torch.empty((n, dim), dtype=torch.int16, device="cuda")
    for r in range(0, n, 2048):
        out[r:r + 2048] = torch.poisson(protos[owner[r:r + 2048]], generator=g).to(torch.int16)
    return out


def _database(case, g, n, dim, identities):
    protos = 3 * _rand(g, 0.5, 1.5, identities, dim)
    owner = torch.randint(0, identities, (n,), generator=g, device="cuda")
    return _counts(g, n, dim, owner, protos), owner, protos


def _model_numbers(case, g, dim):
    """A trained model's support vectors (counts), coefficients, biases and gamma."""
    n_sv, C = case["svs"], case["classes"]
    sv, owner, protos = _database(case, g, n_sv, dim, max(C, IDENTITIES))
    own = owner[None, :] == torch.arange(C, device="cuda")[:, None]
    alpha = _rand(g, 0.2, 1.0, C, n_sv) * own
    rest = _rand(g, 0.0, 1.0, C, n_sv) * ~own * (_rand(g, 0, 1, C, n_sv) < 0.2)
    alpha = alpha - rest * (alpha.sum(1, keepdim=True) / rest.sum(1, keepdim=True).clamp(min=1e-3))
    bias = -0.3 - 0.1 * _rand(g, 0, 1, C)
    return sv, alpha.contiguous(), bias.contiguous(), (1.0 / dim if case["flat"] else 0.5), protos


def _calibration(g):
    u = (2 * torch.rand(6, generator=g, device="cuda") - 1).cpu().tolist()
    rec = np.zeros((), np.dtype([("a", np.int32, 6), ("parallax", np.int32), ("d_min", np.int32),
                                 ("d_max", np.int32), ("colour_w", np.int32), ("colour_h", np.int32)]))
    rec["a"] = [int(65536 * (1 + 0.03 * u[0])), int(655 * u[1]), int(65536 * 8 * u[2]),
                int(655 * u[3]), int(65536 * (1 + 0.03 * u[4])), int(65536 * 8 * u[5])]
    rec["parallax"] = int((25 + 5 * u[0]) * 1000 * 256)
    rec["d_min"], rec["d_max"] = 400, 8000
    return rec


_context = []


def _ctx():
    """The one context that a program keeps."""
    if not _context:
        _context.append(B.Context(0))
    return _context[0]


def _dim(case):
    return 256 if case.get("flags", 0) & 4 else (case["crop"] // 8) ** 2 * BINS


def _inputs(case, seed):
    """The numbers of a case that exist before any call of the library."""
    g, kind, dim = _gen(seed), case["kind"], _dim(case)
    d = {}
    if kind in ("features", "frame", "roi"):
        d["grey"], d["depth"], d["rects"] = _frames(case, g)
    if kind == "frame":
        if case["svs"]:
            d["sv"], d["coef"], d["bias"], d["gamma"], _ = _model_numbers(case, g, dim)
        else:
            d["coef"] = torch.randn((case["classes"], dim), generator=g, device="cuda")
            d["bias"] = torch.randn((case["classes"],), generator=g, device="cuda")
    elif kind == "score":
        d["sv"], d["coef"], d["bias"], d["gamma"], protos = _model_numbers(case, g, dim)
        owner = torch.randint(0, protos.shape[0], (case["rows"],), generator=g, device="cuda")
        d["counts"] = _counts(g, case["rows"], dim, owner, protos)
    elif kind == "normalise":
        d["counts"], _, _ = _database(case, g, case["rows"], dim, IDENTITIES)
    elif kind == "train":
        d["counts"], owner, _ = _database(case, g, case["rows"], dim, case["classes"])
        d["labels"] = owner.int()
    elif kind == "roi":
        n = d["rects"].shape[0]
        box = d["rects"].clone()
        box[:, 1] += torch.randint(15, 36, (n,), generator=g, device="cuda", dtype=torch.int32)
        box[:, 2] += torch.randint(-5, 6, (n,), generator=g, device="cuda", dtype=torch.int32)
        box[:, 3:] = (box[:, 3:4] * _rand(g, 0.95, 1.05, n, 1)).round().int().clamp(min=8)
        d["boxes"], d["calib"] = box.contiguous(), _calibration(g)
        d["calib"]["colour_w"], d["calib"]["colour_h"] = case["width"], case["height"]
    return d


def prepare(case, seed):
    d, ctx, kind = _inputs(case, seed), _ctx(), case["kind"]
    s = dict(d, case=case, ctx=ctx, kind=kind)
    if "coef" in d:
        if "sv" in d:
            s["model"] = B.svm_train_data_pack(ctx, d["sv"], d["coef"], d["bias"], gamma=d["gamma"],
                                               dtype=case["dtype"], centred=case.get("centred", False))
        else:
            s["model"] = B.svm_train_data_pack(ctx, None, d["coef"], d["bias"], kernel=B.KERNEL_LINEAR,
                                               dim=_dim(case))
        s.pop("sv", None)
    if kind == "score":
        s["x"], s["xsq"] = B.lbp_normalize_features(ctx, d["counts"], case["dtype"], x_scale=X_SCALE,
                                                    x_centre=s["model"] if case["centred"] else None)
        s.pop("counts")
    if kind == "train":
        s["x"], s["xsq"] = B.lbp_normalize_features(ctx, d["counts"], "f32")
        s.pop("counts")
    if kind == "roi":
        s["cal"] = B.Calib.from_record(d["calib"])
    if kind == "frame" and case["track"]:
        F = case["frames"]
        s["tracks"] = B.TrackState(8, 16)
        s["stream"] = (torch.arange(F, device="cuda", dtype=torch.int32) % 8).contiguous()
        s["start"] = torch.arange(F + 1, device="cuda", dtype=torch.int32) * case["faces"]
    return s


# ---------------------------------------------------------------------------------------------
# One pass
# ---------------------------------------------------------------------------------------------

def run(s):
    case, ctx, kind = s["case"], s["ctx"], s["kind"]
    if kind == "features":
        feats, x, xsq = B.lbp_fused_features(ctx, s["grey"], s["depth"], s["rects"], crop=case["crop"],
                                             mask_mm=MASK_MM, flags=case["flags"], feats=case["counts"],
                                             x_dtype=case["dtype"], x_scale=X_SCALE)
        return {"counts": feats, "x": x, "xsq": xsq}
    if kind == "frame":
        _, x, xsq = B.lbp_fused_features(ctx, s["grey"], s["depth"], None if case["precut"] else s["rects"],
                                         crop=case["crop"], mask_mm=MASK_MM, feats=False, x_dtype=case["dtype"],
                                         x_scale=X_SCALE)
        scores, labels = B.svm_score(ctx, s["model"], x, xsq, x_scale=X_SCALE)
        out = {"x": x, "xsq": xsq, "scores": scores, "labels": labels}
        if case["track"]:
            out["ids"] = B.rgbd_track_streams(ctx, s["tracks"], s["stream"], s["start"], s["rects"], labels)
        return out
    if kind == "score":
        scores, labels = B.svm_score(ctx, s["model"], s["x"], s["xsq"], x_scale=X_SCALE)
        return {"scores": scores, "labels": labels}
    if kind == "normalise":
        x, xsq = B.lbp_normalize_features(ctx, s["counts"], case["dtype"], x_scale=X_SCALE)
        return {"x": x, "xsq": xsq}
    if kind == "train":
        coef, bias, iters = B.svm_train_rbf(ctx, s["x"], s["xsq"], s["labels"], case["classes"], 0.5, 1.0, 1e-3)
        return {"coef": coef, "bias": bias, "iters": iters}
    rects = B.rgbd_face_roi(ctx, s["depth"], s["cal"], s["boxes"])
    grey, depth = B.rgbd_crop_affine(ctx, s["grey"], s["depth"], rects, case["crop"], case["crop"])
    return {"rects": rects, "grey": grey, "depth": depth}


# ---------------------------------------------------------------------------------------------
# What a pass cannot do without
# ---------------------------------------------------------------------------------------------

def _face_bytes(case):
    """Source bytes of the faces: grey and depth of a mean rect, and no frame more than once."""
    if case.get("precut"):
        return 3.0 * case["crop"] ** 2
    mean = (case["smin"] ** 2 + case["smin"] * case["smax"] + case["smax"] ** 2) / 3.0
    n = case["frames"] * case["faces"]
    frames = 3.0 * case["frames"] * case["height"] * case["width"]
    return min(frames, n * (mean + 2.0 * min(mean, case["crop"] ** 2)))


def work(case):
    kind, dim = case["kind"], _dim(case)
    k_pad = (dim + 127) // 128 * 128
    n = case["frames"] * case["faces"] if kind in ("features", "frame", "roi") else case["rows"]
    esz = ELEM[case.get("dtype", "f32")]
    if kind == "features":
        # about 60 integer operations a crop pixel (resample, mask, 8 compares, count)
        return {"bytes": _face_bytes(case) + n * (esz * k_pad + 4 + 2 * dim * case["counts"]),
                "flops": 60.0 * n * case["crop"] ** 2}
    if kind in ("frame", "score"):
        svs, C = case["svs"], case["classes"]
        rows = esz * n * k_pad + 4 * n
        model = esz * svs * k_pad + 4 * svs + 4 * C * svs if svs else 4 * C * k_pad
        flops = 2.0 * n * svs * (dim + C) if svs else 2.0 * n * dim * C
        more = _face_bytes(case) if kind == "frame" else 0
        return {"bytes": rows + model + 4 * n * (C + 1) + more, "flops": flops}
    if kind == "normalise":
        return {"bytes": n * (2.0 * dim + esz * k_pad + 4), "flops": 4.0 * n * dim}
    if kind == "train":
        # the kernel matrix (half of it is distinct), then its rows during the steps
        return {"bytes": 4.0 * n * k_pad + 4.0 * n * n + 4.0 * n * case["classes"], "flops": 1.0 * n * n * dim}
    return {"bytes": 2.0 * case["frames"] * case["height"] * case["width"] + _face_bytes(case) + 40.0 * n +
            3.0 * n * case["crop"] ** 2, "flops": 30.0 * n * case["crop"] ** 2}


# ---------------------------------------------------------------------------------------------
# The same in plain torch, 64 bits
# ---------------------------------------------------------------------------------------------

def _taps(origin, length, size, limit):
    u = torch.arange(size, device="cuda")[None, :]
    q = origin[:, None] * 65536 + ((2 * u + 1) * length[:, None] * 65536) // (2 * size) - 32768
    a = q >> 16
    return a.clamp(0, limit - 1), (a + 1).clamp(0, limit - 1), (q >> 8) & 255, ((q + 32768) >> 16).clamp(0, limit - 1)


def _cut(grey, depth, rects, size):
    """Crops [n][size][size] (int64) of grey (bilinear, Q8 weights) and depth (nearest)."""
    H, W = grey.shape[1:]
    f, x, y, w, h = (rects[:, i].long() for i in range(5))
    xa, xb, fx, xn = (t[:, None, :] for t in _taps(x, w, size, W))
    ya, yb, fy, yn = (t[:, :, None] for t in _taps(y, h, size, H))
    base = (f * (H * W))[:, None, None]
    g, d = grey.reshape(-1), depth.reshape(-1)
    top = (256 - fx) * g[base + ya * W + xa].long() + fx * g[base + ya * W + xb].long()
    low = (256 - fx) * g[base + yb * W + xa].long() + fx * g[base + yb * W + xb].long()
    return ((256 - fy) * top + fy * low + 32768) >> 16, d[base + yn * W + xn].long() & 0xFFFF


def _ranks():
    c = np.arange(256)
    rot = ((c << 1) | (c >> 7)) & 255
    uniform = np.array([bin(v).count("1") for v in c ^ rot]) <= 2
    return torch.from_numpy(np.where(uniform, np.cumsum(uniform) - 1, BINS - 1)).cuda()


def _histograms(g, d, flags):
    """Count rows (int64) of crops: per 8x8 cell over uniform patterns, or 256 bins a face."""
    n, S = g.shape[:2]
    flat = torch.where(d == 0, 1 << 20, d).reshape(n, -1).sort(1).values
    some = (d != 0).reshape(n, -1).sum(1)
    med = flat.gather(1, ((some - 1).clamp(min=0) // 2)[:, None])[:, :, None]
    valid = (d != 0) & ((d - med).abs() < MASK_MM) & (some > 0)[:, None, None]
    i = torch.arange(S, device="cuda")
    code = torch.zeros_like(g)
    ring = [(-1, -1), (0, -1), (1, -1), (1, 0), (1, 1), (0, 1), (-1, 1), (-1, 0)]
    for p, (dx, dy) in enumerate(ring):
        r, c = (i + dy).clamp(0, S - 1), (i + dx).clamp(0, S - 1)
        gp, vp = g[:, r][:, :, c], valid[:, r][:, :, c]
        code |= (((gp >= g) if flags & 1 else (gp > g)) & (vp | bool(flags & 2))).long() << p
    if flags & 4:
        at, bins = torch.arange(n, device="cuda")[:, None, None] * 256 + code, 256 * n
        return torch.bincount(at[valid], minlength=bins).reshape(n, 256), 256
    G = S // 8
    cell = (i[:, None] // 8) * G + i[None, :] // 8
    at = (torch.arange(n, device="cuda")[:, None, None] * G * G + cell) * BINS + _ranks()[code]
    return torch.bincount(at[valid], minlength=n * G * G * BINS).reshape(n, G * G * BINS), BINS


def _quotients(counts, bins):
    """Per-cell normalised rows, 64 bits (of counts below 2^15)."""
    c = counts.double().reshape(counts.shape[0], -1, bins)
    return (c / c.sum(2, keepdim=True).clamp(min=1)).reshape(counts.shape[0], -1)


def _stored(x32, dtype, scale):
    """The values that rows of a type hold, as 64-bit floats."""
    if dtype == "bf16":
        return x32.bfloat16().double()
    if dtype == "fp8":
        # clamped first: the stored codes saturate
        return (x32 * scale).clamp(-448, 448).to(torch.float8_e4m3fn).double() / scale
    if dtype == "bf16x3":
        hi = x32.bfloat16()
        return hi.double() + (x32 - hi.float()).bfloat16().double()
    return x32.double()


def _rows_exact(q, dtype, k_pad):
    """The row output of a type, and the squared norms of what it holds."""
    x32 = q.float()
    sq = _stored(x32, dtype, X_SCALE).square().sum(1)
    pad = (0, k_pad - q.shape[1])
    if dtype == "fp8":
        return None, sq  # the codes are whole numbers
    if dtype == "bf16x3":
        hi = x32.bfloat16()
        return torch.nn.functional.pad(torch.stack([hi.double(), (x32 - hi.float()).bfloat16().double()]), pad), sq
    return torch.nn.functional.pad(q, pad), sq


def _scores_exact(x, sv, coef, bias, gamma):
    out = torch.empty((x.shape[0], coef.shape[0]), dtype=torch.float64, device="cuda")
    sq = sv.square().sum(1)
    for r in range(0, x.shape[0], 1024):
        xr = x[r:r + 1024]
        d2 = xr.square().sum(1)[:, None] + sq[None, :] - 2 * (xr @ sv.T)
        out[r:r + 1024] = torch.exp(-gamma * d2.clamp(min=0)) @ coef.double().T + bias.double()
    return out


def _model_exact(case, d):
    """The support vectors as the model holds them, and the centre of the rows."""
    sv32 = _quotients(d["sv"], BINS).float()
    mu = None
    if case.get("centred"):
        mu = sv32.double().mean(0).float()
        sv32 = sv32 - mu
    scale = np.float32(448.0) / np.float32(sv32.abs().max().item())
    return _stored(sv32, case["dtype"], float(scale)), mu


def exact(case, seed):
    d, kind, dim = _inputs(case, seed), case["kind"], _dim(case)
    k_pad = (dim + 127) // 128 * 128
    if kind in ("features", "frame"):
        flags, rows = case.get("flags", 0), []
        for r in range(0, d["rects"].shape[0], 128):
            g, z = _cut(d["grey"], d["depth"], d["rects"][r:r + 128], case["crop"])
            h, bins = _histograms(g, z, flags)
            rows.append(_quotients(h, bins).cpu())
        q = torch.cat(rows).cuda()
        x, sq = _rows_exact(q, case["dtype"], k_pad)
        if kind == "features":
            return {"counts": None, "x": x, "xsq": sq}
        held = _stored(q.float(), case["dtype"], X_SCALE)
        if case["svs"]:
            scores = _scores_exact(held, _model_exact(case, d)[0], d["coef"], d["bias"], d["gamma"])
        else:
            scores = held @ d["coef"].double().T + d["bias"].double()
        return {"x": x, "xsq": sq, "scores": scores, "labels": None, "ids": None}
    if kind == "score":
        sv, mu = _model_exact(case, d)
        x32 = _quotients(d["counts"], BINS).float()
        held = _stored(x32 - mu if mu is not None else x32, case["dtype"], X_SCALE)
        return {"scores": _scores_exact(held, sv, d["coef"], d["bias"], d["gamma"]), "labels": None}
    if kind == "normalise":
        x, sq = _rows_exact(_quotients(d["counts"], BINS), case["dtype"], k_pad)
        return {"x": x, "xsq": sq}
    return None  # training stops at a gap, a path and not a number; crops are whole numbers
