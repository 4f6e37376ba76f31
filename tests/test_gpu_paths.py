"""GPU tests of the kernels' variants at the sizes where they can go wrong, against the CPU oracle
or a plain 64-bit reference."""
import numpy as np
import pytest

from paper_1504_01883_gb300 import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def B():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_1504_01883_gb300 import _build, binding
    _build.build()
    return binding


@pytest.fixture(scope="module")
def ctx(B):
    c = B.Context(0)
    yield c
    c.close()


from gpu_util import dev_f32, dev_u16, dev_u8, host_u16, rbf_error_scale, rel_score_error  # noqa: E402,F401


@pytest.mark.parametrize("shape", [(37, 45), (64, 31), (480, 640)])
@pytest.mark.parametrize("colour_w", [640, 20000])
@pytest.mark.parametrize("density", [0.0, 0.002, 0.9])
def test_face_roi_scan_from_the_edges(B, ctx, orc, shape, colour_w, density):
    """The region scan reads a window from its edges inwards: frames that are empty, nearly empty
    (few pixels, anywhere) and dense, windows of less than one strip of rows or columns, depths at
    both ends of the valid range, and colour images too wide for 32-bit coordinates."""
    H, W = shape
    rng = synth.rng_for(H + colour_w + int(1000 * density))
    depth = rng.choice(np.array([399, 400, 401, 1000, 3000, 7999, 8000, 8001, 65535], np.uint16), (3, H, W))
    depth[rng.random((3, H, W)) >= density] = 0
    boxes = np.zeros(60, orc.RECT_DTYPE)
    boxes["frame"] = rng.integers(0, 3, 60)
    boxes["x"], boxes["y"] = rng.integers(-20, W + 40, 60), rng.integers(-20, H + 10, 60)
    boxes["w"], boxes["h"] = rng.integers(1, W + 20, 60), rng.integers(1, H + 20, 60)
    cal = synth.calibration(rng, colour_w, H)
    for flip in (1, -1):  # a mirrored mapping too
        cal["a"][0] *= flip
        cal["a"][2] = 0 if flip > 0 else 65536 * W
        want = orc.face_roi(depth, cal, boxes)
        got = B.rgbd_face_roi(ctx, dev_u16(depth), B.Calib.from_record(cal), B.rects_tensor(boxes)).cpu().numpy()
        for i, f in enumerate(["frame", "x", "y", "w", "h"]):
            assert (got[:, i] == want[f]).all(), (flip, f)
    ctx.status(clear=True)


@pytest.mark.parametrize("a1,a4", [(0, 0), (1, 2), (100, 200), (300, -300), (40000, 70000)])
def test_face_roi_of_nearly_singular_mappings(B, ctx, orc, a1, a4):
    """A mapping whose rows are nearly parallel has no window that single precision could place: the
    whole frame is scanned there, and just short of it the window still holds every pixel."""
    H, W = 96, 128
    rng = synth.rng_for(a1 + 7)
    depth = rng.choice(np.array([0, 0, 0, 900, 1500], np.uint16), (2, H, W))
    boxes = np.zeros(40, orc.RECT_DTYPE)
    boxes["frame"] = rng.integers(0, 2, 40)
    boxes["x"], boxes["y"] = rng.integers(-10, W, 40), rng.integers(-10, H, 40)
    boxes["w"], boxes["h"] = rng.integers(1, 40, 40), rng.integers(1, 40, 40)
    cal = synth.calibration(rng, W, H)
    cal["a"][:] = [65536, a1, 0, 65536, a4, 0]
    want = orc.face_roi(depth, cal, boxes)
    got = B.rgbd_face_roi(ctx, dev_u16(depth), B.Calib.from_record(cal), B.rects_tensor(boxes)).cpu().numpy()
    for i, f in enumerate(["frame", "x", "y", "w", "h"]):
        assert (got[:, i] == want[f]).all(), f
    ctx.status(clear=True)


@pytest.mark.parametrize("out_h,out_w", [(1, 1), (7, 5), (33, 64), (64, 100), (130, 257), (3, 1300)])
@pytest.mark.parametrize("W", [8, 101, 320])
def test_crop_affine_sizes(B, ctx, orc, out_h, out_w, W):
    """Crops of widths that are and are not whole groups of 4 columns, strips of rows with a
    remainder, frames of odd width (byte gathers) and of the narrowest width with 8-byte windows,
    rects narrower and wider than twice the crop, partly outside the frame, and bad ones; by rect
    and by affine map."""
    rng = synth.rng_for(out_h * 1000 + out_w + W)
    H = 60
    g = rng.integers(0, 256, (2, H, W)).astype(np.uint8)
    d = rng.integers(0, 65536, (2, H, W)).astype(np.uint16)
    r = np.zeros(9, orc.RECT_DTYPE)
    r["frame"] = rng.integers(0, 2, 9)
    r["x"], r["y"] = rng.integers(-W, W, 9), rng.integers(-H, H, 9)
    r["w"] = [1, 2 * out_w, 2 * out_w + 1, out_w, 5 * out_w, max(1, out_w // 3), 40, 0, 9]
    r["h"] = [1, 2 * out_h, 3, out_h, 5 * out_h, 11, 40, 5, 9]
    r[8]["frame"] = 2
    gd, dd, rd = dev_u8(g), dev_u16(d), B.rects_tensor(r)
    og, od = B.rgbd_crop_affine(ctx, gd, dd, rd, out_h, out_w)
    og, od = og.cpu().numpy(), host_u16(od)
    for k in range(7):
        wg, wd = orc.crop(g[r[k]["frame"]], d[r[k]["frame"]], tuple(r[k][f] for f in ("x", "y", "w", "h")), out_h, out_w)
        assert (og[k] == wg).all() and (od[k] == wd).all(), k
    assert not og[7:].any() and not od[7:].any()
    assert ctx.status(clear=True) & B.STATUS_BAD_RECT
    aff = rng.integers(-70000, 70000, (9, 6)).astype(np.int32)
    aff[:, [2, 5]] *= 30
    og, od = B.rgbd_crop_affine(ctx, gd, dd, rd, out_h, out_w, affine=torch.from_numpy(aff).cuda())
    og, od = og.cpu().numpy(), host_u16(od)
    for k in range(7):
        wg, wd = orc.crop(g[r[k]["frame"]], d[r[k]["frame"]], (0, 0, 1, 1), out_h, out_w, affine=aff[k])
        assert (og[k] == wg).all() and (od[k] == wd).all(), k
    ctx.status(clear=True)


@pytest.mark.parametrize("dim,nbins", [(59, 59), (9 * 59, 59), (144 * 59, 59), (256 * 59, 59), (256, 256), (512, 256),
                                       (24, 8), (70, 7), (70000, 10), (65536, 16)])
@pytest.mark.parametrize("dt", ["f32", "bf16", "fp8", "bf16x3"])
def test_normalise_rows_are_ieee_quotients(B, ctx, orc, dim, nbins, dt):
    """Rows of every staging form (aligned and odd row lengths, one to many lanes per cell, fewer
    than 8 bins, too long for shared memory): IEEE quotients bit for bit, for counts from 0 to
    65535, converted as the type says, with and without a centre; norms of the stored values."""
    rng = synth.rng_for(dim + nbins)
    cnt = rng.integers(0, 5, (7, dim)).astype(np.uint16)
    cnt[1] = rng.integers(0, 65536, dim)
    cnt[2] = 0
    cnt[3, : nbins] = 65535
    cnt[4] = rng.poisson(400, dim)
    mu = rng.uniform(-0.1, 0.3, (dim + 3) // 4 * 4).astype(np.float32)
    tot = cnt.reshape(7, -1, nbins).astype(np.int64).sum(2, keepdims=True)
    x32 = (cnt.reshape(7, -1, nbins).astype(np.float32) / np.maximum(tot, 1).astype(np.float32)).reshape(7, dim)
    for centre in (None, mu):
        x, q = B.lbp_normalize_features(ctx, dev_u16(cnt), dt, nbins=nbins,
                                        x_centre=None if centre is None else dev_f32(centre))
        want = x32 if centre is None else (x32 - mu[None, :dim]).astype(np.float32)
        if dt == "f32":
            got = x.cpu().numpy()
            assert (got[:, :dim].view(np.uint32) == want.view(np.uint32)).all()
            held = want.astype(np.float64)
        elif dt == "fp8":
            got = x.cpu().numpy()
            codes = orc.f32_to_e4m3((want * np.float32(448.0)).astype(np.float32))
            assert (got[:, :dim] == codes).all()
            held = orc.e4m3_to_f64(codes) / 448.0
        else:
            got = host_u16(x.view(torch.int16))
            hi = orc.f32_to_bf16(want)
            hf = (hi.astype(np.uint32) << 16).view(np.float32)
            held = hf.astype(np.float64)
            if dt == "bf16x3":
                lo = orc.f32_to_bf16((want - hf).astype(np.float32))
                assert (got[1][:, :dim] == lo).all()
                held = held + (lo.astype(np.uint32) << 16).view(np.float32)
                assert not got[1][:, dim:].any()
                got = got[0]
            assert (got[:, :dim] == hi).all()
        assert not got[:, dim:].any()
        # fp32 sums of at most 2^17 squares: well inside 1e-5 relative
        assert np.allclose(q.cpu().numpy(), (held ** 2).sum(1), rtol=1e-5, atol=1e-30)
    assert ctx.status() == 0


@pytest.mark.parametrize("n,n_sv,C", [(9, 40, 3), (64, 65, 1), (65, 1000, 128), (777, 300, 50), (1300, 2100, 7),
                                      (2500, 1100, 33)])
def test_fp32_scores_of_every_tiling(B, ctx, orc, n, n_sv, C):
    """The exact fp32 scores in 64 x 64 tiles (ragged in rows, SVs and classes) and in 128 x 128
    tiles spread over the SMs, where most tiles are handed from one CTA to the next, against the
    fp64 definition; a second call gives the same bits."""
    rng = synth.rng_for(n + n_sv + C)
    dim = 9 * 59
    X, SV = synth.poisson_counts(rng, n, dim), synth.poisson_counts(rng, n_sv, dim)
    a, _ = synth.rbf_coefficients(rng, C, n_sv)
    b = rng.normal(0, 0.01, C).astype(np.float32)
    model = B.svm_train_data_pack(ctx, dev_u16(SV), dev_f32(a), dev_f32(b), gamma=0.3, dtype="f32")
    x, q = B.lbp_normalize_features(ctx, dev_u16(X), "f32")
    s, lab = B.svm_score(ctx, model, x, q)
    s2, lab2 = B.svm_score(ctx, model, x, q)
    assert torch.equal(s, s2) and torch.equal(lab, lab2) and ctx.status() == 0
    x64, sv64 = orc.normalize_f64(X), orc.normalize_f64(SV)
    d2 = (x64 ** 2).sum(1)[:, None] + (sv64 ** 2).sum(1)[None, :] - 2.0 * x64 @ sv64.T
    ref = np.exp(-0.3 * np.maximum(d2, 0.0)) @ a.astype(np.float64).T + b
    scale = rbf_error_scale(x64, sv64, a, b, 0.3)
    # the path's stated bound (1e-5 of the score scale)
    assert rel_score_error(s.cpu().numpy(), ref, scale) <= 1e-5
    assert (lab.cpu().numpy() == s.cpu().numpy().argmax(1)).all()


@pytest.mark.parametrize("n,k_pad", [(2, 7), (65, 128), (200, 531), (700, 256), (2100, 48), (2100, 50)])
def test_kernel_matrix_and_smo_of_every_size(B, ctx, orc, n, k_pad):
    """Training on few and many rows (one to sixteen rows per thread, one tile per CTA and tiles
    handed from CTA to CTA), rows of lengths that are not multiples of 4 or 16: the solution is
    that of the fp64 oracle, and the norms and rows may have any length."""
    rng = synth.rng_for(n + k_pad)
    C = 3
    lab = rng.integers(0, C, n).astype(np.int32)
    x = (rng.normal(0, 1, (C, k_pad))[lab] + rng.normal(0, 0.7, (n, k_pad))).astype(np.float32) / np.sqrt(k_pad)
    x = x.astype(np.float32)
    q = (x.astype(np.float64) ** 2).sum(1).astype(np.float32)
    steps = 60  # a bounded number of steps: the same path as the oracle's, step by step
    xt, qt, lt = dev_f32(x), dev_f32(q), torch.from_numpy(lab).cuda()
    coef, bias, iters = B.svm_train_rbf(ctx, xt, qt, lt, C, 1.0, 1.0, 1e-3, max_iter=steps)
    again = B.svm_train_rbf(ctx, xt, qt, lt, C, 1.0, 1.0, 1e-3, max_iter=steps)
    assert ctx.status() == 0 and all(torch.equal(u, v) for u, v in zip((coef, bias, iters), again))
    it, a = iters.cpu().numpy(), coef.cpu().numpy().astype(np.float64)
    y = np.where(lab[None, :] == np.arange(C)[:, None], 1.0, -1.0)
    alpha = a * y
    assert (alpha >= 0).all() and (alpha <= 1).all() and (it <= steps).all()
    # every step keeps sum a = 0 (fp32 rounding of each step) and lowers the dual objective
    assert np.abs(a.sum(1)).max() <= 1e-6 * (1 + np.abs(a).sum(1).max())
    x64 = x.astype(np.float64)
    K = np.exp(-(np.maximum((x64 ** 2).sum(1)[:, None] + (x64 ** 2).sum(1)[None, :] - 2 * x64 @ x64.T, 0)))
    for c in range(C):
        if it[c] == 0:
            continue
        # the gradient that the kernel walked along gives its stopping gap: recompute it in fp64
        G = y[c] * (K @ a[c]) - 1.0
        v = -y[c] * G
        up = ((y[c] > 0) & (alpha[c] < 1)) | ((y[c] < 0) & (alpha[c] > 0))
        low = ((y[c] > 0) & (alpha[c] > 0)) | ((y[c] < 0) & (alpha[c] < 1))
        gap = v[up].max() - v[low].min()
        obj = 0.5 * a[c] @ K @ a[c] - alpha[c].sum()
        assert obj < 0
        if it[c] < steps:
            assert gap <= 1e-3 + 1e-4  # fp32 gradient of up to 60 steps
        free = (alpha[c] > 0) & (alpha[c] < 1)
        if free.any():
            assert abs(bias[c].item() - v[free].mean()) <= 1e-4


@pytest.mark.parametrize("n", [1, 3, 700])
@pytest.mark.parametrize("dim,C", [(59, 1), (3776, 5), (15104, 64), (531, 256)])
def test_linear_scores(B, ctx, orc, n, dim, C):
    """Linear scores with one and with four rows per CTA (a last group of one to three rows), class
    counts around the groups of eight, short and long rows; ties go to the lowest class."""
    rng = synth.rng_for(n + dim + C)
    w, b = synth.linear_model(rng, C, dim)
    if C > 3:
        w[C - 1], b[C - 1] = w[1], b[1]  # an exact tie
        w[C // 2], b[C // 2] = w[1], b[1]
    x = rng.uniform(0, 0.1, (n, B.k_pad_for(dim))).astype(np.float32)
    x[:, dim:] = 0
    model = B.svm_train_data_pack(ctx, None, dev_f32(w), dev_f32(b), kernel=B.KERNEL_LINEAR, dim=dim)
    s, lab = B.svm_score(ctx, model, dev_f32(x))
    x64 = x[:, :dim].astype(np.float64)
    ref = x64 @ w.astype(np.float64).T + b
    scale = np.abs(x64) @ np.abs(w.astype(np.float64)).T + np.abs(b)
    assert np.all(np.abs(s.cpu().numpy() - ref) <= 1e-5 * scale)
    assert (lab.cpu().numpy() == s.cpu().numpy().argmax(1)).all()


@pytest.mark.parametrize("n", [1, 2, 3, 5, 8])
@pytest.mark.parametrize("n_sv,C,cells", [(1, 1, 1), (17, 10, 256), (333, 128, 70), (700, 64, 256)])
def test_fp32_scores_of_up_to_eight_rows(B, ctx, orc, n, n_sv, C, cells):
    """The exact fp32 scores of one to eight rows: K in one slice and in eight with a short last one,
    an odd last support vector, one and several SV tiles, class counts around the groups of eight."""
    rng = synth.rng_for(n + 10 * n_sv + C)
    dim = cells * 59
    X, SV = synth.poisson_counts(rng, n, dim), synth.poisson_counts(rng, n_sv, dim)
    X[0] = SV[0]  # a row that is a support vector
    a = rng.normal(0, 1, (C, n_sv)).astype(np.float32)
    b = rng.normal(0, 0.01, C).astype(np.float32)
    model = B.svm_train_data_pack(ctx, dev_u16(SV), dev_f32(a), dev_f32(b), gamma=0.3, dtype="f32")
    x, q = B.lbp_normalize_features(ctx, dev_u16(X), "f32")
    s, lab = B.svm_score(ctx, model, x, q)
    assert ctx.status() == 0
    x64, sv64 = orc.normalize_f64(X), orc.normalize_f64(SV)
    ref = orc.svm_rbf(x64, sv64, a, b, 0.3)
    # the path's stated bound (1e-5 of the score scale)
    assert rel_score_error(s.cpu().numpy(), ref, rbf_error_scale(x64, sv64, a, b, 0.3)) <= 1e-5
    assert (lab.cpu().numpy() == s.cpu().numpy().argmax(1)).all()


@pytest.mark.parametrize("crop", [8, 9, 50, 131, 255])
@pytest.mark.parametrize("flags", [0, 1, 2, 3])
def test_face_histogram_256_sizes_and_rules(B, ctx, orc, crop, flags):
    """The 0-255 histogram at the smallest and largest side and at every number of pixels in a row's
    last word, under every neighbour rule: rects inside and outside frames of even and odd width
    (one frame all holes), pre-cut crops and a general affine map, bit-exact with the oracle."""
    fl = flags | B.LBP_FACE_HIST256
    for W in (200, 203):
        g, d, r = synth.frames_with_rects(crop + flags + W, 3, 3, 20, 160, H=120, W=W)
        d[2] = 0
        want = orc.features_batch(g, d, r, crop, cell=crop, nbins=256, flags=flags)
        f, x, q = B.lbp_fused_features(ctx, dev_u8(g), dev_u16(d), B.rects_tensor(r), crop=crop, flags=fl,
                                       x_dtype="bf16")
        assert (host_u16(f) == want).all(), W
        x32 = orc.normalize_f32(want, nbins=256)
        assert (host_u16(x.view(torch.int16))[:, :256] == orc.f32_to_bf16(x32)).all()
    gc, dc = synth.crops(crop, 2, crop)
    want = orc.features_batch(gc, dc, None, crop, cell=crop, nbins=256, flags=flags)
    f, _, _ = B.lbp_fused_features(ctx, dev_u8(gc), dev_u16(dc), None, crop=crop, flags=fl)
    assert (host_u16(f) == want).all()
    n = r.shape[0]
    aff = np.zeros((n, 6), np.int32)
    for k in range(n):
        sc = r[k]["w"] / float(crop)
        aff[k] = [int(0.9 * sc * 65536), int(-0.3 * sc * 65536), int(r[k]["x"] * 65536),
                  int(0.3 * sc * 65536), int(0.9 * sc * 65536), int(r[k]["y"] * 65536)]
    want = orc.features_batch(g, d, r, crop, cell=crop, nbins=256, flags=flags, affine=aff)
    f, _, _ = B.lbp_fused_features(ctx, dev_u8(g), dev_u16(d), B.rects_tensor(r), crop=crop, flags=fl,
                                   affine=torch.from_numpy(aff).cuda())
    assert (host_u16(f) == want).all()
    assert ctx.status() == 0


@pytest.mark.parametrize("crop", [32, 64, 96, 128])
@pytest.mark.parametrize("dt", ["bf16", "fp8"])
def test_rows_with_and_without_the_quotient_table(B, ctx, orc, crop, dt):
    """Few faces (quotients computed) and more faces than SMs (bf16 quotients from the table at 96 and
    128): the same faces give the same rows and norms, and the rows are the oracle's."""
    g, d, r = synth.frames_with_rects(crop, 2, 5, 30, 160, H=160, W=200)
    many = np.concatenate([r] * 40)  # 400 faces
    f, x, q = B.lbp_fused_features(ctx, dev_u8(g), dev_u16(d), B.rects_tensor(r), crop=crop, x_dtype=dt)
    fm, xm, qm = B.lbp_fused_features(ctx, dev_u8(g), dev_u16(d), B.rects_tensor(many), crop=crop, x_dtype=dt)
    want = orc.features_batch(g, d, r, crop)
    assert (host_u16(f) == want).all()
    x32 = orc.normalize_f32(want)
    rows = orc.f32_to_bf16(x32) if dt == "bf16" else orc.f32_to_e4m3((x32 * np.float32(448.0)).astype(np.float32))
    got = host_u16(x.view(torch.int16)) if dt == "bf16" else x.cpu().numpy()
    assert (got[:, :want.shape[1]] == rows).all()
    for k in range(0, 400, 10):
        assert torch.equal(fm[k:k + 10], f) and torch.equal(xm[k:k + 10], x) and torch.equal(qm[k:k + 10], q)


@pytest.mark.parametrize("dt,C", [("bf16", 64), ("bf16", 3), ("fp8", 128)])
def test_split_combines_agree(B, ctx, orc, dt, C):
    """Up to 1024 rows are combined by a thread per output, more rows by a warp per row: the same
    terms in the same order, so the same rows give the same bits in a batch of 129, 1024 and 1025
    rows (one layout of the splits), and they are the fp64 scores within the type's bound."""
    rng = synth.rng_for(C)
    n_sv, dim = 5 * 256 + 40, 9 * 59
    X, SV = synth.poisson_counts(rng, 1025, dim), synth.poisson_counts(rng, n_sv, dim)
    a, _ = synth.rbf_coefficients(rng, C, n_sv)
    b = rng.normal(0, 0.01, C).astype(np.float32)
    model = B.svm_train_data_pack(ctx, dev_u16(SV), dev_f32(a), dev_f32(b), gamma=1.0 / dim, dtype=dt)
    got = {}
    ctx.set_tuning(B.TUNE_TC_SPLITS, 3)
    try:
        for n in (129, 1024, 1025):
            x, q = B.lbp_normalize_features(ctx, dev_u16(X[:n]), dt)
            got[n] = B.svm_score(ctx, model, x, q)
    finally:
        ctx.set_tuning(B.TUNE_TC_SPLITS, 0)
    assert ctx.status() == 0
    for n in (129, 1024):
        assert torch.equal(got[n][0], got[1025][0][:n]) and torch.equal(got[n][1], got[1025][1][:n])
    x64, sv64 = orc.normalize_f64(X[:129]), orc.normalize_f64(SV)
    ref = orc.svm_rbf(x64, sv64, a, b, 1.0 / dim)
    err = rel_score_error(got[129][0].cpu().numpy(), ref, rbf_error_scale(x64, sv64, a, b, 1.0 / dim))
    assert err <= {"bf16": 5e-5, "fp8": 1e-3}[dt]  # the types' stated bounds


@pytest.mark.parametrize("dt", ["bf16", "fp8", "bf16x3", "f32"])
@pytest.mark.parametrize("faces", [1, 7, 40])
def test_scores_right_behind_their_features(B, ctx, orc, faces, dt):
    """The scoring kernels of few rows start before the feature kernel in front of them has finished:
    frame after frame without a pause gives the same bits as with the GPU waited for in between."""
    rng = synth.rng_for(faces)
    H, W, n_sv, C, frames = 240, 320, 700, 12, 12
    grey = dev_u8(rng.integers(0, 256, (frames, H, W), np.uint8))
    depth = dev_u16(rng.integers(700, 1300, (frames, H, W)).astype(np.uint16))
    sv = dev_u16(rng.poisson(1.1, (n_sv, 64 * 59)).clip(0, 64).astype(np.uint16))
    coef = dev_f32(rng.normal(size=(C, n_sv)).astype(np.float32))
    model = B.svm_train_data_pack(ctx, sv, coef, gamma=0.02, dtype=dt)
    rects = []
    for f in range(frames):
        r = np.zeros(faces, orc.RECT_DTYPE)
        r["frame"], r["w"], r["h"] = f, rng.integers(30, 120, faces), rng.integers(30, 120, faces)
        r["x"], r["y"] = rng.integers(0, 200, faces), rng.integers(0, 120, faces)
        rects.append(B.rects_tensor(r))
    # one buffer for all frames' rows: rows read too early would be the frame before's
    _, x, xsq = B.lbp_fused_features(ctx, grey, depth, rects[0], crop=64, feats=False, x_dtype=dt)

    def scores(pause):
        out = []
        for r in rects:
            B.lbp_fused_features(ctx, grey, depth, r, crop=64, feats=False, x_dtype=dt, out={"x": x, "xsq": xsq})
            if pause:
                torch.cuda.synchronize()
            out.append(B.svm_score(ctx, model, x, xsq))
        return out

    for (s0, l0), (s1, l1) in zip(scores(True), scores(False)):
        assert torch.equal(s0, s1) and torch.equal(l0, l1)
    assert ctx.status() == 0


@pytest.mark.parametrize("crop", [64, 96])
@pytest.mark.parametrize("dt,flags", [("bf16", 0), ("fp8", 3), ("f32", 1), ("bf16x3", 2)])
def test_few_faces_give_the_bits_of_a_batch(B, ctx, orc, crop, dt, flags):
    """Up to a face per SM takes four threads per cell, a larger batch two: the same counts, rows and
    norms to the bit, and counts as the oracle's."""
    grey, depth, r = synth.frames_with_rects(crop, 10, 17, 20, 110, H=120, W=160)
    g, d = dev_u8(grey), dev_u16(depth)
    fb, xb, qb = B.lbp_fused_features(ctx, g, d, B.rects_tensor(r), crop=crop, flags=flags, x_dtype=dt)
    for k in (1, 40, 152):
        f, x, q = B.lbp_fused_features(ctx, g, d, B.rects_tensor(r[:k]), crop=crop, flags=flags, x_dtype=dt)
        whole = xb[:, :k] if dt == "bf16x3" else xb[:k]
        assert torch.equal(f, fb[:k]) and torch.equal(x, whole) and torch.equal(q, qb[:k])
    want = orc.features_batch(grey, depth, r[:40], crop, flags=flags)
    assert (host_u16(fb[:40]) == want).all()


@pytest.mark.parametrize("crop", [32, 64, 96, 128])
@pytest.mark.parametrize("W", [8, 60, 200])
def test_rects_around_the_crop_width(B, ctx, orc, crop, W):
    """Rects up to the crop's width read the grey taps of four pixels from one window, wider ones those
    of two: widths on both sides of the line, partly outside the frame, down to the narrowest frame."""
    rng = synth.rng_for(crop + W)
    H = 50
    grey = rng.integers(0, 256, (2, H, W)).astype(np.uint8)
    depth = rng.integers(800, 1200, (2, H, W)).astype(np.uint16)
    widths = [1, 2, crop // 2, crop - 1, crop, crop + 1, 2 * crop, 2 * crop + 1]
    r = np.zeros(4 * len(widths), orc.RECT_DTYPE)
    r["frame"], r["w"] = rng.integers(0, 2, len(r)), np.repeat(widths, 4)
    r["h"], r["y"] = rng.integers(1, 60, len(r)), rng.integers(-20, 40, len(r))
    r["x"] = np.tile([-3, 0, W // 2, W - 2], len(widths)) + rng.integers(0, 4, len(r))
    f, _, _ = B.lbp_fused_features(ctx, dev_u8(grey), dev_u16(depth), B.rects_tensor(r), crop=crop)
    assert (host_u16(f) == orc.features_batch(grey, depth, r, crop)).all()


@pytest.mark.parametrize("mask_mm", [1, 2, 150, 32768, 65535, 65536, 1 << 20])
@pytest.mark.parametrize("centre", [1, 140, 1000, 40000, 65535])
def test_depth_mask_at_the_ends_of_its_range(B, ctx, orc, mask_mm, centre):
    """The mask takes two depths at a time modulo 2^16: medians and windows at both ends of the range,
    holes, and depths one inside and one outside the window."""
    rng = synth.rng_for(centre + mask_mm % 1009)
    near = np.array([centre] * 8 + [centre + k for k in (-mask_mm, 1 - mask_mm, mask_mm - 1, mask_mm, -1, 1)])
    pool = np.concatenate([near, [0, 0, 1, 2, 65534, 65535]])
    depth = rng.choice(pool[(pool >= 0) & (pool <= 65535)], (6, 64, 64)).astype(np.uint16)
    depth[5] = 0
    grey = rng.integers(0, 256, (6, 64, 64)).astype(np.uint8)
    for flags in (0, 3):
        f, _, _ = B.lbp_fused_features(ctx, dev_u8(grey), dev_u16(depth), crop=64, mask_mm=mask_mm, flags=flags)
        assert (host_u16(f) == orc.features_batch(grey, depth, None, 64, mask_mm=mask_mm, flags=flags)).all()


@pytest.mark.parametrize("gamma", [0.3, 5.0, 20.0, 200.0])
@pytest.mark.parametrize("dt,n", [("f32", 1), ("f32", 3), ("f32", 8), ("bf16", 7), ("bf16", 40)])
def test_few_row_scores_at_any_gamma(B, ctx, orc, gamma, dt, n):
    """Scores of few rows where the distances of a model spread far over 1 / gamma: rows that are support
    vectors of the first and of the last SV tile, rows near no support vector, tiles 250 apart in mean
    distance.  Against fp64; exact fp32 rows also against the same rows in a batch of nine, which another
    kernel scores."""
    rng = synth.rng_for(int(10 * gamma) + n)
    cells, n_sv, C = 256, 700, 6
    SV = synth.poisson_counts(rng, n_sv, cells * 59)
    one = np.zeros((257, cells, 59), np.uint16)  # rows with one bin per cell: far from all others
    np.put_along_axis(one, rng.integers(0, 59, (257, cells, 1)), 64, 2)
    SV[:256] = one[:256].reshape(256, -1)
    rows = max(n, 9)
    X = synth.poisson_counts(rng, rows, cells * 59)
    X[0], X[1], X[2] = SV[600], SV[3], one[256].reshape(-1)
    a = rng.normal(0, 1, (C, n_sv)).astype(np.float32)
    b = rng.normal(0, 0.01, C).astype(np.float32)
    model = B.svm_train_data_pack(ctx, dev_u16(SV), dev_f32(a), dev_f32(b), gamma=gamma, dtype=dt)
    x, q = B.lbp_normalize_features(ctx, dev_u16(X[:n]), dt)
    s, lab = B.svm_score(ctx, model, x, q)
    s, lab = s.cpu().numpy(), lab.cpu().numpy()
    assert ctx.status() == 0

    def held(counts):  # the values a row holds, in fp64
        v = orc.normalize_f64(counts)
        return v if dt == "f32" else torch.from_numpy(v.astype(np.float32)).bfloat16().double().numpy()

    x64, sv64 = held(X), held(SV)
    xx, ss, g = (x64 ** 2).sum(1)[:, None], (sv64 ** 2).sum(1)[None, :], x64 @ sv64.T
    K = np.exp(-gamma * np.maximum(xx + ss - 2 * g, 0))
    ref = K @ a.astype(np.float64).T + b
    # a distance is off by the fp32 rounding of two norms and a product: chains of at most 80 additions
    # (tensor cores: 15104 products in any order, taken as 1024), a kernel value by gamma times that,
    # the sums by the path's 1e-5 of the score's scale and of the largest kernel value
    off = gamma * (96 if dt == "f32" else 1024) * 2.0 ** -24 * (xx + ss + 2 * g)
    absa = np.abs(a.astype(np.float64)).T
    tol = (K * np.expm1(np.minimum(off, 50))) @ absa + 1e-5 * (K @ absa + np.abs(b)) + 1e-6 * K.max(1, keepdims=True) * absa.sum(0)
    assert (np.abs(s - ref[:n]) <= tol[:n]).all()
    assert (lab == s.argmax(1)).all()
    if dt == "f32":
        x9, q9 = B.lbp_normalize_features(ctx, dev_u16(X), dt)
        s9, _ = B.svm_score(ctx, model, x9, q9)
        assert (np.abs(s - s9.cpu().numpy()[:n]) <= 2 * tol[:n] + 1e-6 * absa.sum(0)).all()


def _waits(tiles, stages, sms):
    """CTAs whose range of the even split begins inside a tile, and that tile."""
    starts = [tiles * stages * g // sms for g in range(sms)]
    return {g: u // stages for g, u in enumerate(starts) if u % stages}


def test_fp32_rows_of_a_lost_handover_are_zero(B, ctx, orc):
    """A CTA waits in vain for the first part of a tile: the status says so, the rows of that tile get zero
    scores and label 0, the other rows their bits, and the next call is whole again."""
    rng = synth.rng_for(11)
    n, n_sv, C, dim = 1300, 2100, 7, 9 * 59
    X, SV = synth.poisson_counts(rng, n, dim), synth.poisson_counts(rng, n_sv, dim)
    a = rng.normal(0, 1, (C, n_sv)).astype(np.float32)
    model = B.svm_train_data_pack(ctx, dev_u16(SV), dev_f32(a), dev_f32(np.ones(C, np.float32)), gamma=0.3, dtype="f32")
    x, q = B.lbp_normalize_features(ctx, dev_u16(X), "f32")
    want, labels = B.svm_score(ctx, model, x, q)
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    mt, nt = -(-n // 128), -(-n_sv // 128)
    waits = _waits(mt * nt, model.k_pad // 16, sms)
    ctx.status(clear=True)
    for cta in list(waits)[3::40]:
        B.rgbd_debug_drop_handover(ctx, cta - 1)
        try:
            s, lab = B.svm_score(ctx, model, x, q)
        finally:
            B.rgbd_debug_drop_handover(ctx, -1)
        assert ctx.status(clear=True) == B.STATUS_WAIT_TIMEOUT
        lost = slice(128 * (waits[cta] % mt), min(n, 128 * (waits[cta] % mt + 1)))
        assert not s[lost].any() and not lab[lost].any()
        s[lost], lab[lost] = want[lost], labels[lost]
        assert torch.equal(s, want) and torch.equal(lab, labels)
    s, lab = B.svm_score(ctx, model, x, q)
    assert torch.equal(s, want) and torch.equal(lab, labels) and ctx.status() == 0


def test_training_of_a_lost_handover_gives_zeros(B, ctx):
    """The same in the kernel matrix, on which every class hangs."""
    rng = synth.rng_for(12)
    n, k_pad = 2100, 48
    x = rng.normal(0, 0.4, (n, k_pad)).astype(np.float32)
    q = (x.astype(np.float64) ** 2).sum(1).astype(np.float32)
    args = (dev_f32(x), dev_f32(q), torch.from_numpy(rng.integers(0, 3, n).astype(np.int32)).cuda(), 3, 1.0, 1.0, 1e-3)
    want = B.svm_train_rbf(ctx, *args, max_iter=60)
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    t = -(-n // 128)
    cta = list(_waits(t * (t + 1) // 2, k_pad // 16, sms))[20]
    ctx.status(clear=True)
    B.rgbd_debug_drop_handover(ctx, cta - 1)
    try:
        got = B.svm_train_rbf(ctx, *args, max_iter=60)
    finally:
        B.rgbd_debug_drop_handover(ctx, -1)
    assert ctx.status(clear=True) == B.STATUS_WAIT_TIMEOUT
    assert not any(t.any() for t in got)
    assert all(torch.equal(u, v) for u, v in zip(B.svm_train_rbf(ctx, *args, max_iter=60), want))
    assert ctx.status() == 0


@pytest.mark.parametrize("call", ["crop", "normalise", "face256"])
def test_threads_with_different_sizes(B, call):
    """Two threads, each with a context and a stream, make calls that take different amounts of shared
    memory: a limit that one sets must not be lowered by the other before the launch."""
    import threading
    rects = torch.zeros((1000, 5), dtype=torch.int32, device="cuda")
    rects[:, 3:] = 16
    grey = torch.zeros((1, 16, 16), dtype=torch.uint8, device="cuda")
    depth = torch.ones((1, 16, 16), dtype=torch.int16, device="cuda")
    rows = {d: torch.ones((2, d), dtype=torch.int16, device="cuda") for d in (59 * 450, 59 * 1100)}
    work = {"crop": lambda c, s, big: B.rgbd_crop_affine(c, grey, depth, rects, 4096 if big else 3100, 4, stream=s),
            "normalise": lambda c, s, big: B.lbp_normalize_features(c, rows[59 * (1100 if big else 450)], "bf16", stream=s),
            "face256": lambda c, s, big: B.lbp_fused_features(c, grey, depth, rects[:2], crop=255 if big else 40,
                                                              flags=B.LBP_FACE_HIST256, stream=s)}[call]
    torch.cuda.synchronize()
    errors, start = [], threading.Barrier(2)

    def loop(big):
        c, s = B.Context(0), torch.cuda.Stream()
        try:
            start.wait()
            with torch.cuda.stream(s):
                for _ in range(400):
                    work(c, s, big)
        except B.RgbdError as e:
            errors.append(str(e))
        finally:
            s.synchronize()
            c.close()

    threads = [threading.Thread(target=loop, args=(big,)) for big in (False, True)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors[0]


@pytest.mark.parametrize("crop", [32, 64, 96])
def test_two_ctas_per_sm_are_those_of_a_128_crop(B, ctx, crop):
    """A context tuned for 128 x 128 batches (two CTAs per SM, all that fit) keeps the occupancy of smaller
    crops, of which 4 to 16 fit: as fast as untuned (at two, 32 x 32 crops take several times as long), and
    the same counts; one means half of what fits."""
    grey, depth, r = synth.frames_with_rects(crop, 8, 20, 30, 110, H=240, W=320)
    g, d, rects = dev_u8(grey), dev_u16(depth), B.rects_tensor(np.concatenate([r] * 25))  # 4000 faces

    def run():
        best = []
        for _ in range(12):
            e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            e0.record()
            f, _, _ = B.lbp_fused_features(ctx, g, d, rects, crop=crop)
            e1.record()
            torch.cuda.synchronize()
            best.append(e0.elapsed_time(e1))
        return min(best), f

    t0, f0 = run()
    times = {}
    for ctas in (2, 1):
        ctx.set_tuning(B.TUNE_LBP_CTAS_PER_SM, ctas)
        try:
            times[ctas], f = run()
        finally:
            ctx.set_tuning(B.TUNE_LBP_CTAS_PER_SM, 0)
        assert torch.equal(f, f0)
    assert times[2] < 1.25 * t0, (t0, times)


@pytest.mark.parametrize("n_sv", [65536, 65537, 132000])
@pytest.mark.parametrize("n,gamma", [(1, 0.3), (8, 0.3), (3, 20.0)])
def test_few_rows_against_more_than_256_tiles(B, ctx, orc, n_sv, n, gamma):
    """Up to eight fp32 rows against models around and beyond 65536 support vectors, which the few-row
    epilogue combines in pieces of 256 tiles: scores within the path's bound of fp64."""
    rng = synth.rng_for(n_sv + n)
    dim, C = 4 * 59, 5
    X, SV = synth.poisson_counts(rng, n, dim), synth.poisson_counts(rng, n_sv, dim)
    X[0] = SV[n_sv - 1]
    a = rng.normal(0, 1, (C, n_sv)).astype(np.float32)
    b = rng.normal(0, 0.01, C).astype(np.float32)
    model = B.svm_train_data_pack(ctx, dev_u16(SV), dev_f32(a), dev_f32(b), gamma=gamma, dtype="f32")
    x, q = B.lbp_normalize_features(ctx, dev_u16(X), "f32")
    s, lab = B.svm_score(ctx, model, x, q)
    assert ctx.status() == 0
    x64, sv64 = orc.normalize_f64(X), orc.normalize_f64(SV)
    d2 = (x64 ** 2).sum(1)[:, None] + (sv64 ** 2).sum(1)[None, :] - 2.0 * x64 @ sv64.T
    ref = np.exp(-gamma * np.maximum(d2, 0.0)) @ a.astype(np.float64).T + b
    # the path's stated bound (1e-5 of the score scale)
    assert rel_score_error(s.cpu().numpy(), ref, rbf_error_scale(x64, sv64, a, b, gamma)) <= 1e-5
    assert (lab.cpu().numpy() == s.cpu().numpy().argmax(1)).all()


def test_server_of_a_large_model_and_batch_is_created_quickly(B, ctx):
    """The workspace of the largest batch is found from the few batch sizes that can hold the maximum; asking
    for all 65536 of them against 300000 fp32 support vectors took 1.2 s of host time."""
    import time
    n_sv, dim, C = 300000, 16 * 59, 5
    sv = torch.ones((n_sv, dim), dtype=torch.int16, device="cuda")
    model = B.svm_train_data_pack(ctx, sv, torch.ones((C, n_sv), device="cuda"), gamma=0.01, dtype="f32")

    def create(faces):
        t = time.monotonic()
        server = B.NativeServer(model, 64, 64, 4, n_slots=2, max_batch_faces=faces, crop=32)
        t = time.monotonic() - t
        server.close()
        return t

    create(64)
    assert min(create(65536) for _ in range(3)) < 0.6


@pytest.mark.parametrize("per_sm", [1, 2, 4, 8, 9])
@pytest.mark.parametrize("dim,C", [(59, 1), (944, 2), (59, 3), (944, 4), (944, 5), (59, 8), (944, 9), (59, 33),
                                   (12036, 5), (12036, 3)])
def test_linear_scores_by_rows_per_sm(B, ctx, per_sm, dim, C):
    """Linear scores around the row counts where the threads per row change (a row, two, four and eight per
    SM), with class counts on both sides of the two, four and eight taken at a time."""
    rng = synth.rng_for(per_sm + dim + C)
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    w, b = synth.linear_model(rng, C, dim)
    model = B.svm_train_data_pack(ctx, None, dev_f32(w), dev_f32(b), kernel=B.KERNEL_LINEAR, dim=dim)
    for n in {per_sm * sms, (per_sm - 1) * sms + 1, per_sm * sms - 2}:
        x = rng.uniform(0, 0.1, (n, B.k_pad_for(dim))).astype(np.float32)
        x[:, dim:] = 0
        s, lab = B.svm_score(ctx, model, dev_f32(x))
        x64 = x[:, :dim].astype(np.float64)
        ref = x64 @ w.astype(np.float64).T + b
        scale = np.abs(x64) @ np.abs(w.astype(np.float64)).T + np.abs(b)
        # fp32 chains of at most 12036 / 128 products and sums over 128 threads, well inside 1e-5
        assert np.all(np.abs(s.cpu().numpy() - ref) <= 1e-5 * scale)
        assert (lab.cpu().numpy() == s.cpu().numpy().argmax(1)).all()


@pytest.mark.parametrize("H", [1, 8, 15, 16, 17, 33, 40])
def test_face_roi_of_a_single_pixel(B, ctx, orc, H):
    """The scans from the top and from the bottom meet in the middle of the window: one pixel in each row in
    turn, and none."""
    W = 70
    depth = np.zeros((H + 1, H, W), np.uint16)  # frame H has none
    rng = synth.rng_for(H)
    for i in range(H):
        depth[i, i, rng.integers(0, W)] = 1000
    boxes = np.zeros(H + 1, orc.RECT_DTYPE)
    boxes["frame"], boxes["w"], boxes["h"] = np.arange(H + 1), W + 80, H
    cal = synth.calibration(rng, W + 80, H)
    cal["a"][:] = [65536, 0, 0, 0, 65536, 0]
    want = orc.face_roi(depth, cal, boxes)
    got = B.rgbd_face_roi(ctx, dev_u16(depth), B.Calib.from_record(cal), B.rects_tensor(boxes)).cpu().numpy()
    for i, f in enumerate(["frame", "x", "y", "w", "h"]):
        assert (got[:, i] == want[f]).all(), f
    assert (want["h"][:H] == 1).all() and want["h"][H] == 0


@pytest.mark.parametrize("n,out_h,out_w", [(1, 300, 518), (1, 300, 520), (1, 9, 131072 // 32), (2, 1100, 300), (800, 20, 39),
                                           (3, 1030, 256), (400, 300, 5), (400, 301, 7), (6000, 16, 16), (6000, 16, 17)])
def test_crops_of_few_and_of_many_pixels(B, ctx, orc, n, out_h, out_w):
    """Crops around the sizes where a thread makes one pixel or a group of four, by rect and by affine map, rows
    of whole warps of groups and others: the oracle's pixels, and zeros for a bad rect."""
    rng = synth.rng_for(n + out_h + out_w)
    H, W = 60, 80
    g = rng.integers(0, 256, (2, H, W)).astype(np.uint8)
    d = rng.integers(0, 65536, (2, H, W)).astype(np.uint16)
    r = np.zeros(n, orc.RECT_DTYPE)
    r["frame"] = rng.integers(0, 2, n)
    r["x"], r["y"] = rng.integers(-20, W, n), rng.integers(-20, H, n)
    r["w"], r["h"] = rng.integers(1, 90, n), rng.integers(1, 90, n)
    if n > 1:
        r["w"][n - 1] = 0
    aff = rng.integers(-70000, 70000, (n, 6)).astype(np.int32)
    aff[:, [2, 5]] *= 30
    gd, dd, rd = dev_u8(g), dev_u16(d), B.rects_tensor(r)
    for a in (None, aff):
        og, od = B.rgbd_crop_affine(ctx, gd, dd, rd, out_h, out_w, affine=None if a is None else torch.from_numpy(a).cuda())
        for k in {0, n // 2, n - 1}:
            kg, kd = og[k].cpu().numpy(), host_u16(od[k])
            if r[k]["w"] == 0:
                assert not kg.any() and not kd.any()
                continue
            wg, wd = orc.crop(g[r[k]["frame"]], d[r[k]["frame"]], tuple(r[k][f] for f in ("x", "y", "w", "h")), out_h, out_w,
                              affine=None if a is None else a[k])
            assert (kg == wg).all() and (kd == wd).all(), (k, a is None)
    assert bool(ctx.status(clear=True) & B.STATUS_BAD_RECT) == (n > 1)


def _training_rows(n, k_pad, C, spread):
    rng = synth.rng_for(n + k_pad)
    lab = rng.integers(0, C, n).astype(np.int32)
    x = ((rng.normal(0, 1, (C, k_pad))[lab] + rng.normal(0, spread, (n, k_pad))) / np.sqrt(k_pad)).astype(np.float32)
    q = (x.astype(np.float64) ** 2).sum(1).astype(np.float32)
    return lab, x, q


def _ascent(x, lab, c, a):
    """-y G of class c's dual at coefficients a, in fp64 (from the rows with a coefficient alone), y, and how far
    fp32 may be from it after `steps` steps."""
    x64 = x.astype(np.float64)
    y = np.where(lab == c, 1.0, -1.0)
    sv = np.flatnonzero(a)
    d2 = (x64 ** 2).sum(1)[:, None] + (x64[sv] ** 2).sum(1)[None, :] - 2 * x64 @ x64[sv].T
    v = y - np.exp(-np.maximum(d2, 0)) @ a[sv]
    # every step rounds a row's value once; a kernel value is off by the fp32 rounding of its distance (norms and
    # a chain of k_pad products) and of its exponential
    off_k = (x.shape[1] + 4) * 2.0 ** -24 * 4 * (x64 ** 2).sum(1).max() + 4 * 2.0 ** -24
    return v, y, lambda steps: steps * 2.0 ** -24 * 4 + np.abs(a).sum() * off_k


@pytest.mark.parametrize("n,k_pad", [(300, 48), (2100, 48), (2300, 50)])
def test_training_converges_to_the_optimum(B, ctx, n, k_pad):
    """Trained to the stopping gap, in tiles of a CTA each and in tiles handed from CTA to CTA: the optimality
    conditions hold in fp64 for every row of every class, which takes the kernel values between all support
    vectors and all rows; the bias is the mean over the free vectors."""
    C, eps = 3, 1e-2
    lab, x, q = _training_rows(n, k_pad, C, 0.9)
    coef, bias, iters = B.svm_train_rbf(ctx, dev_f32(x), dev_f32(q), torch.from_numpy(lab).cuda(), C, 1.0, 1.0, eps,
                                        max_iter=200000)
    assert ctx.status() == 0
    for c in range(C):
        a, it = coef[c].cpu().numpy().astype(np.float64), int(iters[c])
        assert 10 < it < 200000
        v, y, off = _ascent(x, lab, c, a)
        alpha, tol = a * y, off(it)
        assert (alpha >= 0).all() and (alpha <= 1).all() and abs(a.sum()) <= it * 2.0 ** -23
        up = np.where(y > 0, alpha < 1, alpha > 0)
        low = np.where(y > 0, alpha > 0, alpha < 1)
        assert v[up].max() - v[low].min() <= eps + 2 * tol, (c, tol)
        free = (alpha > 0) & (alpha < 1)
        assert free.any() and abs(float(bias[c]) - v[free].mean()) <= tol + 1e-6


@pytest.mark.parametrize("n", [256, 257, 1024, 1025, 2048, 2049, 4096, 4097, 8192, 8193])
def test_training_steps_take_the_most_violating_pair(B, ctx, n):
    """Around the row counts where the threads and the rows per thread change: the pair that step s + 1 moves
    (the coefficients after s + 1 steps against those after s) is the most violating one after s, in fp64."""
    C, k_pad = 2, 32
    lab, x, q = _training_rows(n, k_pad, C, 0.9)
    lab[-1], lab[0] = 0, 1
    args = (dev_f32(x), dev_f32(q), torch.from_numpy(lab).cuda(), C, 1.0, 1.0, 1e-6)
    for s in (0, 1, 2, 7, 40):
        a0, _, i0 = B.svm_train_rbf(ctx, *args, max_iter=s)
        a1, _, i1 = B.svm_train_rbf(ctx, *args, max_iter=s + 1)
        assert (i0 == s).all() and (i1 == s + 1).all()
        for c in range(C):
            a, b = a0[c].cpu().numpy().astype(np.float64), a1[c].cpu().numpy().astype(np.float64)
            v, y, off = _ascent(x, lab, c, a)
            up = np.where(y > 0, a < 1, a < 0)
            low = np.where(y > 0, a > 0, a > -1)
            moved = np.flatnonzero(a != b)
            assert len(moved) == 2 and (b[moved] - a[moved]).sum() <= 2.0 ** -22
            i, j = moved if b[moved[0]] > a[moved[0]] else moved[::-1]  # a grows by i's step, falls by j's
            assert up[i] and low[j]
            assert v[i] >= v[up].max() - 2 * off(s) and v[j] <= v[low].min() + 2 * off(s)
    assert ctx.status() == 0


def test_epilogue_expm1_up_to_its_switch(B):
    """The series of the epilogue's e^z - 1 reaches to 1/2: within 2 ulp of the exact value (3 of CUDA's expm1f)
    densely from 1/32 to 1/2 and on both sides of the switch."""
    rng = np.random.default_rng(6)
    half = np.float32(0.5)
    z = np.concatenate([rng.uniform(0.03, 0.5, 300000), np.linspace(0.499, 0.501, 4001),
                        [half, np.nextafter(half, np.float32(0)), np.nextafter(half, np.float32(1))]]).astype(np.float32)
    z = np.concatenate([z, -z])
    zt = torch.from_numpy(z).cuda()
    ours, cuda = B.rgbd_debug_expm1(zt).cpu().numpy().astype(np.float64), torch.expm1(zt).cpu().numpy().astype(np.float64)
    exact = np.expm1(z.astype(np.float64))
    ulp = np.spacing(np.abs(exact).astype(np.float32)).astype(np.float64)
    assert np.max(np.abs(ours - exact) / ulp) <= 2.0
    assert np.max(np.abs(ours - cuda) / ulp) <= 3.0


@pytest.mark.parametrize("C", [1, 2, 63, 64, 65, 128])
@pytest.mark.parametrize("n", [129, 130, 131, 132])
def test_split_combine_of_few_and_many_classes(B, ctx, orc, C, n):
    """The combine takes up to four rows to a block, fewer for more classes: a last block of one to four rows,
    against fp64, and the same bits as a warp per row gives (a batch of more than 1024 rows)."""
    rng = synth.rng_for(C + n)
    n_sv, dim = 700, 9 * 59
    X, SV = synth.poisson_counts(rng, 1025, dim), synth.poisson_counts(rng, n_sv, dim)
    a = rng.normal(0, 1, (C, n_sv)).astype(np.float32)
    b = rng.normal(0, 0.01, C).astype(np.float32)
    model = B.svm_train_data_pack(ctx, dev_u16(SV), dev_f32(a), dev_f32(b), gamma=1.0 / dim, dtype="bf16")
    ctx.set_tuning(B.TUNE_TC_SPLITS, 3)
    try:
        x, q = B.lbp_normalize_features(ctx, dev_u16(X), "bf16")
        big, lbig = B.svm_score(ctx, model, x, q)
        s, lab = B.svm_score(ctx, model, x[:n].contiguous(), q[:n].contiguous())
    finally:
        ctx.set_tuning(B.TUNE_TC_SPLITS, 0)
    assert ctx.status() == 0 and torch.equal(s, big[:n]) and torch.equal(lab, lbig[:n])
    x64, sv64 = orc.normalize_f64(X[:n]), orc.normalize_f64(SV)
    ref = orc.svm_rbf(x64, sv64, a, b, 1.0 / dim)
    assert rel_score_error(s.cpu().numpy(), ref, rbf_error_scale(x64, sv64, a, b, 1.0 / dim)) <= 5e-5


@pytest.mark.parametrize("gamma", [0.02, 0.06, 0.12, 0.3, 1.0])
@pytest.mark.parametrize("dt", ["bf16", "bf16x3"])
def test_tile_scores_on_both_sides_of_the_series(B, ctx, orc, gamma, dt):
    """The tile kernel's e^z - 1 is a polynomial up to |z| = 0.35: gammas for which all, some and few of the
    arguments lie below, against fp64 of the stored values.  F and the coefficients are rounded to bf16 (to pairs
    of them), relative to the mean distance of the split."""
    rng = synth.rng_for(int(100 * gamma))
    n, n_sv, dim, C = 150, 500, 64 * 59, 9
    X, SV = rng.poisson(2, (n, dim)).astype(np.uint16), rng.poisson(2, (n_sv, dim)).astype(np.uint16)
    SV[::3] = (SV[::3] * rng.integers(0, 2, (len(SV[::3]), dim))).astype(np.uint16)  # distances of several kinds
    a = rng.normal(0, 1, (C, n_sv)).astype(np.float32)
    b = rng.normal(0, 0.01, C).astype(np.float32)
    model = B.svm_train_data_pack(ctx, dev_u16(SV), dev_f32(a), dev_f32(b), gamma=gamma, dtype=dt)
    x, q = B.lbp_normalize_features(ctx, dev_u16(X), dt)
    s, lab = B.svm_score(ctx, model, x, q)
    assert ctx.status() == 0

    def held(counts):
        v = torch.from_numpy(orc.normalize_f32(counts))
        hi = v.bfloat16()
        return (hi.double() + ((v - hi.float()).bfloat16().double() if dt == "bf16x3" else 0)).numpy()

    x64, sv64 = held(X), held(SV)
    xx, ss, g = (x64 ** 2).sum(1)[:, None], (sv64 ** 2).sum(1)[None, :], x64 @ sv64.T
    d2 = np.maximum(xx + ss - 2 * g, 0)
    K = np.exp(-gamma * d2)
    ref = K @ a.astype(np.float64).T + b
    z = gamma * np.abs(d2 - d2.mean(1, keepdims=True)).max(1, keepdims=True)
    # F and the coefficient are each rounded to u = 2^-9 (2^-17 as pairs) of themselves, F at most e^z - 1; a
    # distance is off by the products' fp32 sums (taken as 256 roundings; a pair's lo * lo product, 2^-18 of g, is left
    # out), the rest by fp32
    u = 2.0 ** -9 if dt == "bf16" else 2.0 ** -17
    off = gamma * (256 * 2.0 ** -24 * (xx + ss + 2 * g) + (2.0 ** -16 * g if dt == "bf16x3" else 0))
    absa = np.abs(a.astype(np.float64)).T
    tol = np.exp(-gamma * d2.min(1, keepdims=True)) * (2.1 * u * np.expm1(z) + 1e-6) * absa.sum(0) + (K * np.expm1(off)) @ absa
    assert (np.abs(s.cpu().numpy() - ref) <= tol).all()
    assert (lab.cpu().numpy() == s.cpu().numpy().argmax(1)).all()


@pytest.mark.parametrize("w,h", [(1, 90), (90, 1), (13, 17), (59, 60), (60, 60), (61, 59), (60, 61), (90, 91), (30, 129)])
@pytest.mark.parametrize("density", [0.001, 0.1, 1.0])
def test_face_roi_of_small_and_large_windows(B, ctx, orc, w, h, density):
    """Windows around the size up to which every pixel is read (4096, with the margins at the sides), down to
    single rows and columns, nearly empty to full."""
    rng = synth.rng_for(100 * w + h + int(1000 * density))
    H, W, n = 140, 150, 24
    depth = rng.integers(700, 1300, (3, H, W)).astype(np.uint16)
    depth[rng.random((3, H, W)) >= density] = 0
    boxes = np.zeros(n, orc.RECT_DTYPE)
    boxes["frame"], boxes["w"], boxes["h"] = rng.integers(0, 3, n), w, h
    boxes["x"], boxes["y"] = rng.integers(0, W - w + 1, n), rng.integers(0, H - h + 1, n)
    cal = synth.calibration(rng, W, H)
    cal["a"][:] = [65536, 0, 0, 0, 65536, 0]
    cal["parallax"] = 0
    want = orc.face_roi(depth, cal, boxes)
    got = B.rgbd_face_roi(ctx, dev_u16(depth), B.Calib.from_record(cal), B.rects_tensor(boxes)).cpu().numpy()
    for i, f in enumerate(["frame", "x", "y", "w", "h"]):
        assert (got[:, i] == want[f]).all(), f
