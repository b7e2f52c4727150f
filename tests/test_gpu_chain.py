"""The chain (one-pass band FHT, DP tiles, read-back) at the edges of its rules:
window modes, tile and block widths, edge columns, unaligned rows, batches of
several tile widths.  Integer results and decisions equal the oracle's exactly,
float Hough values bit for bit."""
import numpy as np
import pytest

import oracle
from helpers import hough_from_oracle, to_device

pytestmark = pytest.mark.gpu


def _img(h, w, dtype, seed):
    rng = np.random.default_rng(seed)
    if dtype == "u8":
        return rng.integers(0, 256, (h, w)).astype(np.uint8)
    if dtype == "i32":
        return rng.integers(-3000, 3000, (h, w)).astype(np.int32)
    return np.abs(rng.standard_normal((h, w))).astype(np.float32)


def _detect(img, k, B):
    return oracle.detect_f32(img, k, B) if img.dtype == np.float32 else oracle.detect(img, k, B)


def _same(got, want):
    x, d, s = (t.cpu().numpy() for t in got)
    xo, do, so = want
    assert list(x) == list(xo) and list(d) == list(do)
    assert s.reshape(-1)[0] == s.dtype.type(so)


# Scanned windows (B <= 3), padded ones (up to 32; not a multiple of the run of
# 8, one run, several), clipped ones (33 and on), for the tile widths 256 .. 16.
@pytest.mark.parametrize("n,B", [(1, 0), (2, 1), (4, 3), (4, 6), (8, 2), (8, 3), (8, 4), (8, 14),
                                 (16, 7), (16, 8), (32, 9), (32, 31), (64, 16), (64, 32), (64, 33),
                                 (128, 5), (128, 24), (128, 32), (128, 33), (128, 100), (128, 254),
                                 (256, 3), (256, 32), (256, 40), (256, 510)])
def test_detect_every_window_mode_matches_oracle(lib, n, B):
    for dtype, w in (("u8", 333), ("i32", 260), ("f32", 301)):
        k = 4 if n > 64 else 6
        img = _img(k * n, w, dtype, 13 * n + B)
        _same(lib.detect_polyline(to_device(img), k, B), _detect(img, k, B))


# Shortest windows of 1 (scanned), 8 / 9 / 10 around the rule, and long ones.
@pytest.mark.parametrize("n,gamma", [(8, 0.3), (32, 0.12), (32, 0.14), (32, 0.16), (64, 0.07),
                                     (128, 0.02), (128, 0.035), (128, 0.04), (128, 0.5),
                                     (256, 0.0175), (256, 0.3)])
def test_angle_windows_around_the_run_length(lib, n, gamma):
    k = 4
    for dtype in ("u8", "f32"):
        img = _img(k * n, 290, dtype, n)
        want = (oracle.detect_angle_f32 if dtype == "f32" else oracle.detect_angle)(img, k, 1, gamma)
        _same(lib.detect_polyline_angle(to_device(img), k, 1, gamma), want)


# Widths at the edges of the FHT's columns (multiples of 16), rows that cannot
# be read four pixels at a time, images narrower than a band.
@pytest.mark.parametrize("n", [4, 8, 16, 128, 256])
@pytest.mark.parametrize("w", [1, 15, 16, 17, 255, 256, 257, 512, 530])
def test_fht_block_widths_match_oracle(lib, n, w):
    for dtype in ("u8", "f32"):
        img = _img(2 * n, w, dtype, n + w)
        H = lib.fht_bands(to_device(img), 2).cpu().numpy()
        if dtype == "f32":
            want = hough_from_oracle(img, 2, float32=True)
            assert np.array_equal(H.view(np.uint32), want.view(np.uint32))
        else:
            assert np.array_equal(H.astype(np.float64), hough_from_oracle(img, 2))


# Bands so short that the four pixels at the image's right edge reach past the
# cyclic width (n = 2, w = 1 mod 4: column w - 1 + 3 is column 0 again).
@pytest.mark.parametrize("n", [1, 2])
@pytest.mark.parametrize("w", [1, 2, 3, 4, 5, 8, 33, 34, 255, 257])
def test_fht_of_short_bands_wraps_at_the_padded_width(lib, n, w):
    for dtype in ("u8", "i32", "f32"):
        img = _img(6 * n, w, dtype, 7 * n + w)
        H = lib.fht_bands(to_device(img), 6).cpu().numpy()
        if dtype == "f32":
            want = hough_from_oracle(img, 6, float32=True)
            assert np.array_equal(H.view(np.uint32), want.view(np.uint32))
        else:
            assert np.array_equal(H.astype(np.float64), hough_from_oracle(img, 6))


# Bands of at most 16 rows: blocks of several bands (narrow images), bands left
# over, blocks inside the image and at its edges, rows of a wider array.
@pytest.mark.parametrize("n", [1, 2, 4, 8, 16])
@pytest.mark.parametrize("k,w", [(1, 1), (3, 5), (37, 7), (9, 33), (5, 131), (2, 1030)])
def test_fht_of_short_bands_matches_oracle(lib, n, k, w):
    for dtype in ("u8", "i32", "f32"):
        wide = _img(k * n, w + 3, dtype, n + k + w)
        H = lib.fht_bands(to_device(wide)[:, 1:w + 1], k).cpu().numpy()
        img = np.ascontiguousarray(wide[:, 1:w + 1])
        if dtype == "f32":
            want = hough_from_oracle(img, k, float32=True)
            assert np.array_equal(H.view(np.uint32), want.view(np.uint32))
        else:
            assert np.array_equal(H.astype(np.float64), hough_from_oracle(img, k))


# Rows split among the warps that search V_0 (fewer rows than 256), parts of odd
# lengths and parts past the last column.
@pytest.mark.parametrize("n,k,w", [(1, 3, 1), (1, 2, 5000), (2, 3, 77), (2, 2, 9001), (16, 2, 2049),
                                   (64, 2, 700), (128, 2, 259), (256, 2, 65)])
def test_backtrack_of_split_rows_matches_oracle(lib, n, k, w):
    for dtype in ("i32", "f32"):
        img = _img(n * k, w, dtype, n + w)
        B = max(1, n // 4)
        V = lib.polyline_dp(lib.fht_bands(to_device(img), k), n * k, w, k, B)
        _same(lib.backtrack(V, n * k, w, k, B), _detect(img, k, B))


# The layer calls on arrays of the caller's own: d = 0 is read in the "+" half,
# whatever the copy in the "-" half holds.
@pytest.mark.parametrize("n,k,w", [(1, 3, 40), (4, 3, 1100), (64, 3, 90), (128, 2, 2050)])
def test_layer_calls_read_d0_in_the_plus_half(lib, n, k, w):
    for dtype in ("i32", "f32"):
        img = _img(n * k, w, dtype, n + w + 2)
        B = n // 2
        H = lib.fht_bands(to_device(img), k)
        H[:, 1, 0, :] = 1 << 20
        V = lib.polyline_dp(H, n * k, w, k, B)
        if k > 1:
            import torch
            assert torch.equal(V[:, 0, 0, :w], V[:, 1, 0, :w])
        V[:, 1, 0, :] = 1 << 20
        _same(lib.backtrack(V, n * k, w, k, B), _detect(img, k, B))


def test_backtrack_passes_over_nan(lib):
    """NaN values lose against every number, in the top band and in the windows;
    a window of nothing but NaN is followed at its first value."""
    import torch
    n, k, w, B = 8, 3, 50, 2
    rng = np.random.default_rng(0)
    V = rng.standard_normal((k, 2, n, w + n)).astype(np.float32)
    V[:, 1, 0] = V[:, 0, 0]
    x = np.arange(w)
    for s in range(n):
        V[:, 0, s, :w][:, x + s >= w] = -np.inf
        V[:, 1, s, :w][:, x - s < 0] = -np.inf
    V[..., w:] = -np.inf
    dead = np.isneginf(V)
    V[rng.random(V.shape) < 0.3] = np.nan
    V[1, :, :, 20:30] = np.nan          # whole windows
    V[dead] = -np.inf
    V[0, 0, 3, 22] = 9.0                # the optimum's link leads there
    at = lambda b, x, d: V[b, 0, d, x] if d >= 0 else V[b, 1, -d, x]
    best, xs, ds = None, [], []
    for xx in range(w):
        for d in range(-(n - 1), n):
            v = at(0, xx, d)
            if v == v and not np.isneginf(v) and (best is None or v > best):
                best, xs, ds = v, [xx], [d]
    for b in range(1, k):
        xs.append(xs[-1] + ds[-1])
        win = [d for d in range(max(ds[-1] - B, 1 - n), min(ds[-1] + B, n - 1) + 1)
               if not np.isneginf(at(b, xs[-1], d))]
        real = [d for d in win if at(b, xs[-1], d) == at(b, xs[-1], d)]
        ds.append(max(real, key=lambda d: (at(b, xs[-1], d), -d)) if real else win[0])
    xs.append(xs[-1] + ds[-1])
    gx, gd, gs = lib.backtrack(torch.from_numpy(V).cuda(), n * k, w, k, B)
    assert gx.tolist() == xs and gd.tolist() == ds and gs.item() == best


@pytest.mark.parametrize("dtype", ["i32", "f32"])
def test_batch_of_every_band_height(lib, dtype):
    shapes = [(256, 333, 128, 16), (512, 70, 128, 40), (256, 500, 64, 3), (320, 201, 32, 5),
              (128, 640, 16, 2), (64, 300, 8, 4), (64, 19, 4, 1), (40, 33, 2, 2), (17, 50, 1, 0),
              (512, 90, 256, 20)]
    imgs = [_img(h, w, dtype, h + w) for h, w, n, B in shapes]
    plan = lib.BatchPlan([to_device(im) for im in imgs], [h // n for h, w, n, B in shapes],
                         [B for h, w, n, B in shapes])
    for _ in range(2):   # the second run finds the first one's counters
        plan.run()
        plan.status()
        for i, (h, w, n, B) in enumerate(shapes):
            _same((plan.x[i], plan.d[i], plan.score[i]), _detect(imgs[i], h // n, B))


def test_detect_runs_in_the_engine_workspace_too(lib):
    """A uint8 image whose workspace is too small for the chain runs on the
    fused engine, with the same results."""
    import torch
    img = _img(1024, 700, "u8", 5)
    dimg = to_device(img)
    need = lib.workspace_bytes(0, 1024, 700, 8, 12)
    want = _detect(img, 8, 12)
    for size in (need, need - 4096):
        _same(lib.detect_polyline(dimg, 8, 12, ws=torch.empty(size, dtype=torch.uint8, device="cuda")),
              want)


@pytest.mark.parametrize("r", [0, 1, 4, 5])
@pytest.mark.parametrize("w,pitch", [(1, 1), (7, 8), (64, 64), (130, 131), (1025, 1028)])
def test_gauss_rows_edges(lib, r, w, pitch):
    import torch
    for dtype in ("u8", "i32", "f32"):
        img = _img(5, w, dtype, w + r)
        big = torch.zeros((5, pitch), dtype=to_device(img).dtype, device="cuda")
        big[:, :w] = to_device(img)
        got = lib.gauss_rows(big[:, :w], r).cpu().numpy()
        want = (oracle.gauss_rows_f32 if dtype == "f32" else oracle.gauss_rows)(img, r)
        assert np.array_equal(got, want)


def test_missing_producer_of_a_middle_band_times_out(lib):
    import torch
    img = to_device(_img(512, 384, "f32", 3))
    ws = torch.empty(lib.workspace_bytes(2, 512, 384, 4, 8), dtype=torch.uint8, device="cuda")
    lib.lib().fhtdp_debug_inject(2, 5, 2_000_000)
    lib.detect_polyline(img, 4, 8, ws=ws)
    with pytest.raises(lib.FhtdpError) as e:
        lib.workspace_status(ws)
    assert e.value.code == 4
    _same(lib.detect_polyline(img, 4, 8, ws=ws), _detect(img.cpu().numpy(), 4, 8))
    lib.workspace_status(ws)


@pytest.mark.parametrize("w", [197, 244, 255])
def test_noalloc_takes_256_row_bands_up_to_its_scratch(lib, w):
    """int32 rows of eight bands of 256 rows: 14.8, 16.4 and 16.7 of 16.8 MB, the
    last two only with rows that are not padded to whole lines."""
    import ctypes

    import torch
    img = _img(2048, w, "i32", w)
    src = to_device(img)
    x = torch.empty(9, dtype=torch.int32, device="cuda")
    d = torch.empty(8, dtype=torch.int32, device="cuda")
    s = torch.empty(1, dtype=torch.int32, device="cuda")
    p = [ctypes.c_void_p(t.data_ptr()) for t in (src, x, d, s)]
    rc = lib.lib().fhtdp_detect_polyline_noalloc(
        p[0], 1, 2048, w, w, 8, 20, p[1], p[2], p[3],
        ctypes.c_void_p(torch.cuda.current_stream().cuda_stream))
    assert rc == 0, lib.lib().fhtdp_last_error().decode()
    _same((x, d, s), oracle.detect(img, 8, 20))


def test_batch_status_reports_a_wait_of_a_256_row_image_that_gave_up(lib):
    """Those images run by themselves beside the batch's launch: the plan's
    status covers them."""
    import torch
    img = _img(1024, 300, "i32", 5)
    plan = lib.BatchPlan([to_device(img)] * 2, [4, 4], [9, 9])
    lib.lib().fhtdp_debug_inject(3, 1, 2_000_000)   # waits of about 1 ms
    plan.run()
    torch.cuda.synchronize()
    with pytest.raises(lib.FhtdpError) as e:
        plan.status()
    assert e.value.code == 4
    plan.run()
    torch.cuda.synchronize()
    assert plan.status() == 0
    for i in range(2):
        _same((plan.x[i], plan.d[i], plan.score[i]), oracle.detect(img, 4, 9))


# Every single-image call in the least workspace that it accepts (one byte less is
# refused), the bytes after it untouched.
@pytest.mark.parametrize("n,k,w", [(1, 5, 9), (2, 3, 1), (8, 4, 33), (64, 3, 101), (128, 2, 257),
                                   (256, 1, 65), (256, 3, 130)])
def test_calls_in_the_least_workspace(lib, n, k, w):
    import torch
    L = lib.lib()
    for dtype, code in (("u8", 0), ("i32", 1), ("f32", 2)):
        img = _img(n * k, w, dtype, n + k + w)
        dev, h, B = to_device(img), n * k, max(1, n // 8)
        f = dtype == "f32"
        at = lambda t: t.data_ptr()
        cases = [
            (L.fhtdp_detect_polyline, (B,), 1, [_detect(img, k, B)]),
            (L.fhtdp_detect_through_point, (B, 0, w // 2), 1,
             [(oracle.detect_through_f32 if f else oracle.detect_through)(img, k, B, 0, w // 2)]),
            (L.fhtdp_detect_polyline_padded, (B,), 1,
             [(oracle.detect_padded_f32 if f else oracle.detect_padded)(img, k, B)]),
            (L.fhtdp_detect_two_polylines, (B, 2), 2,
             list(zip(*(oracle.detect_two_f32 if f else oracle.detect_two)(img, k, B, 2)))),
        ]
        for r in (0, 2):
            cases.append((L.fhtdp_detect_polyline_angle, (r, 0.3), 1,
                          [(oracle.detect_angle_f32 if f else oracle.detect_angle)(img, k, r, 0.3)]))
        for fn, args, count, want in cases:
            x = torch.empty((count, k + 1), dtype=torch.int32, device="cuda")
            d = torch.empty((count, k), dtype=torch.int32, device="cuda")
            s = torch.empty(count, dtype=torch.float32 if f else torch.int32, device="cuda")
            ws = torch.full((1 << 22,), 0x5a, dtype=torch.uint8, device="cuda")
            call = lambda b: fn(at(dev), code, h, w, w, k, *args, at(x), at(d), at(s), at(ws), b,
                                torch.cuda.current_stream().cuda_stream)
            assert call(1) == 2
            need = int(L.fhtdp_last_error().decode().split("needs ")[1].split()[0])
            assert call(need - 1) == 2 and call(need) == 0
            for i in range(count):
                _same((x[i], d[i], s[i]), want[i])
            assert bool((ws[need:] == 0x5a).all())


def test_batch_of_256_row_bands_in_the_least_workspace(lib):
    """int32 images that run one by one: the workspace that the plan offers, and
    the smaller one of their two Hough arrays each."""
    import torch
    L = lib.lib()
    shapes = [(256, 65, 1), (512, 130, 2), (768, 33, 3), (256, 64, 1), (512, 31, 2)]
    imgs = [_img(h, w, "i32", w) for h, w, _ in shapes]
    dev = [to_device(i) for i in imgs]
    ks, Bs = [k for _, _, k in shapes], [20] * len(shapes)
    plan = lib.BatchPlan(dev, ks, Bs)
    least = 4 * max(256 + 2 * (k * 2 * 256 * (w + 256) * 4) for _, w, k in shapes) + 4096
    offered = plan.ws.numel()
    assert least < offered
    for size in (offered, least):
        ws = torch.full((offered + 4096,), 0x5a, dtype=torch.uint8, device="cuda")
        small = lib.BatchPlan(dev, ks, Bs, ws=ws[:size])
        small.run()
        assert small.status() == 0
        for i, img in enumerate(imgs):
            _same((small.x[i], small.d[i], small.score[i]), _detect(img, ks[i], Bs[i]))
        assert bool((ws[size:] == 0x5a).all())
    with pytest.raises(ValueError):
        lib.BatchPlan(dev, ks, Bs, ws=ws[:4096])


@pytest.mark.parametrize("dtype", ["i32", "f32"])
def test_tuning_calls_on_int32_and_float_batches(lib, dtype):
    """autotune leaves the outputs of a run, choice reports what the queue is, and
    configure takes the one width that there is."""
    shapes = [(256, 300, 64), (64, 90, 8), (256, 41, 128)]
    imgs = [_img(h, w, dtype, w) for h, w, _ in shapes]
    ks, Bs = [h // n for h, _, n in shapes], [n // 8 for _, _, n in shapes]
    plan = lib.BatchPlan([to_device(i) for i in imgs], ks, Bs)
    tiles = {64: 32, 8: 256, 128: 16}
    width = sum(-(-w // tiles[n]) for _, w, n in shapes)
    assert plan.autotune(reps=1) == width

    def right():
        for i, img in enumerate(imgs):
            _same((plan.x[i], plan.d[i], plan.score[i]), _detect(img, ks[i], Bs[i]))
            plan.x[i].fill_(-7)
    right()
    for n, tile in tiles.items():
        c = plan.choice(n)
        assert c["schedule"] == "groups" and c["width"] == width and c["tile"] == tile
        plan.configure(n, tile, c["depth"])
        plan.configure(n, 16, 2)
        for bad in ((tile + 1, 2), (tile, 4), (tile, 1)):
            with pytest.raises(lib.FhtdpError):
                plan.configure(n, *bad)
    with pytest.raises(lib.FhtdpError):
        plan.configure(32, 16, 2)          # no image of 32-row bands
    plan.run()
    right()
