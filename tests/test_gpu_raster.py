"""gs_raster_fwd / gs_raster_bwd against the FP64 oracle on identical FP32 records.

The oracle projects in FP64; its records rounded to FP32 are the input of both the
CUDA path (gs_bin_sort + gs_raster_*) and the oracle compositing (evaluated in FP64).
Pixels where a cut-off decision (alpha vs 1/255, T vs 1e-4) lies within rounding
distance of its threshold are flagged by the oracle and excluded from the 1e-4
bound; their number is asserted to be tiny and their error bounded.
"""
import numpy as np
import pytest
import torch

from oracle import raster as oras
from paper_2507_20239_gb300 import rasterizer as R
from paper_2507_20239_gb300 import synth
from tests.gs_fixtures import oracle_lists, oracle_records_fp32, records_to_gpu, rel_l2, scene

pytestmark = pytest.mark.gpu
IMG_TOL = 1e-4
GRAD_TOL = 1e-3


def _oracle_fwd(rec, cam, tile, bg, tiles=None, d_image=None):
    lists = oracle_lists(rec)
    if d_image is None:
        rt = oras.records_to_torch(rec["mean2d"], rec["conic_f"], rec["opacity"], rec["rgb"])
        with torch.no_grad():
            return oras.rasterize(rt, lists, cam.width, cam.height, tile[0], tile[1], bg, tiles), None
    return oras.raster_vjp(rec["mean2d"], rec["conic_f"], rec["opacity"], rec["rgb"], lists, cam.width,
                           cam.height, d_image, tile[0], tile[1], bg, tiles)


def _gpu(recs, cams, tile, bg, store_stop=True):
    frame = R.Frame(cams, tile=tile)
    proj = records_to_gpu(recs)
    bins = R.bin_sort(proj, frame)
    img, T, stop = R.raster_fwd(proj, bins, frame, bg, store_stop=store_stop)
    torch.cuda.synchronize()
    return frame, proj, bins, img, T, stop


def _tile_mask(cam, tile, tiles):
    gx = (cam.width + tile[0] - 1) // tile[0]
    m = np.zeros((cam.height, cam.width), bool)
    for t in tiles:
        tx, ty = t % gx, t // gx
        m[ty * tile[1]:(ty + 1) * tile[1], tx * tile[0]:(tx + 1) * tile[0]] = True
    return m


def _compare_fwd(o, img, T, stop, mask=None, counts=None, max_flag_frac=2e-3):
    """Image and T within 1e-4, stop index and per-pixel work counts exact, on every
    pixel the oracle does not flag. A flagged pixel (an alpha-floor or cut-off
    decision within the derived FP32 error bound of its threshold, see
    oracle.raster.composite) whose GPU stop index and work counts still equal the
    oracle's took the same decisions and is held to 1e-4 too; the others (a decision
    flipped inside the bound) to 1/255 + 1e-4. Flagged pixels must be rare: the
    derived window predicts ~0.02% on the 60k-Gaussian view and ~0.2% on the dense
    tiles of the full-size views."""
    flag = o["flag"]
    sel = ~flag if mask is None else (~flag & mask)
    err = np.abs(img - o["image"]).max(0)
    errT = np.abs(T - o["T_final"])
    assert err[sel].max(initial=0) < IMG_TOL, err[sel].max()
    assert errT[sel].max(initial=0) < IMG_TOL
    assert np.array_equal(stop[sel], o["stop"][sel])
    if counts is not None:
        assert np.array_equal(counts[..., 0][sel], o["n_examined"][sel])
        assert np.array_equal(counts[..., 1][sel], o["n_contrib"][sel])
    fl = flag if mask is None else (flag & mask)
    n_fl = int(fl.sum())
    print(f"flagged {n_fl} of {int(sel.sum()) + n_fl} pixels")
    assert n_fl <= max(2, max_flag_frac * (sel.sum() + n_fl)), n_fl
    if n_fl:
        same = fl & (stop == o["stop"])
        if counts is not None:
            same &= (counts[..., 0] == o["n_examined"]) & (counts[..., 1] == o["n_contrib"])
        else:
            same[:] = False
        assert err[same].max(initial=0) < IMG_TOL and errT[same].max(initial=0) < IMG_TOL
        assert err[fl].max() < 1 / 255 + IMG_TOL
    return n_fl


@pytest.mark.parametrize("name,tile,bg", [("small", (16, 16), (0, 0, 0)), ("small", (8, 8), (0.2, 0.5, 1.0)),
                                          ("orbit_small", (16, 16), (0, 0, 0)),
                                          ("orbit_small", (16, 32), (0.3, 0.1, 0.7))])
def test_raster_fwd_matches_oracle(name, tile, bg):
    sc = scene(name)
    cam = sc.cameras[0]
    rec = oracle_records_fp32(sc.params(), sc.sh_degree, cam, tile)
    frame, proj, bins, img, T, stop = _gpu([rec], [cam], tile, bg)
    o, _ = _oracle_fwd(rec, cam, tile, bg)
    counts = R.raster_count(proj, bins, frame).cpu().numpy().reshape(cam.height, cam.width, 2)
    _compare_fwd(o, frame.view_image(img, 0).cpu().numpy(), frame.view_pixels(T, 0).cpu().numpy(),
                 frame.view_pixels(stop, 0).cpu().numpy(), counts=counts)


def test_raster_fwd_ragged_image_and_empty_tiles():
    # a 37x23 image (ragged last tile row/column) where most tiles are empty
    from paper_2507_20239_gb300 import synth
    sc = synth.small_scene(3, n=40, width=37, height=23)
    cam = sc.cameras[0]
    rec = oracle_records_fp32(sc.params(), 0, cam)
    frame, proj, bins, img, T, stop = _gpu([rec], [cam], (16, 16), (0.1, 0.1, 0.1))
    o, _ = _oracle_fwd(rec, cam, (16, 16), (0.1, 0.1, 0.1))
    _compare_fwd(o, frame.view_image(img, 0).cpu().numpy(), frame.view_pixels(T, 0).cpu().numpy(),
                 frame.view_pixels(stop, 0).cpu().numpy())


@pytest.mark.parametrize("use_stop", [False, True])
@pytest.mark.parametrize("name,tile,bg", [("small", (16, 16), (0, 0, 0)), ("small", (8, 8), (0.2, 0.5, 1.0)),
                                          ("orbit_small", (16, 16), (0.1, 0.2, 0.3))])
def test_raster_bwd_matches_oracle(name, tile, bg, use_stop):
    # use_stop: the walk is bounded by the forward's stop indices instead of
    # re-deriving the cut-off; the gradients are the same
    sc = scene(name)
    cam = sc.cameras[0]
    rec = oracle_records_fp32(sc.params(), sc.sh_degree, cam, tile)
    frame, proj, bins, img, T, stop = _gpu([rec], [cam], tile, bg)
    rng = np.random.default_rng(7)
    d_image = rng.normal(0, 1, (3, cam.height, cam.width)).astype(np.float32)
    o, g = _oracle_fwd(rec, cam, tile, bg, d_image=d_image)
    assert o["flag"].sum() <= max(2, 2e-3 * o["flag"].size)
    dg = torch.as_tensor(d_image.reshape(-1)).cuda()
    rg = R.raster_bwd(proj, bins, frame, img, dg, bg, stop=stop if use_stop else None)
    torch.cuda.synchronize()
    got = dict(d_mean2d=rg.d_mean2d.cpu().numpy(), d_conic=rg.d_conic_opacity[:, :3].cpu().numpy(),
               d_opacity=rg.d_conic_opacity[:, 3].cpu().numpy(), d_rgb=rg.d_rgb[:, :3].cpu().numpy())
    assert np.all(rg.d_rgb[:, 3].cpu().numpy() == 0)
    for k in got:
        e = rel_l2(got[k], g[k])
        assert e < GRAD_TOL, (k, e)
    # culled records receive nothing
    cul = rec["radius"] == 0
    assert np.all(got["d_mean2d"][cul] == 0)


def test_raster_full_size_sampled_tiles():
    """1.5M Gaussians at 1246x826 in the benchmark's launch configuration; the
    oracle composites 24 sampled tiles (plus the 4 longest lists) and back-propagates
    a d_image that is zero outside them."""
    sc = scene("orbit")
    cam = sc.cameras[0]
    tile = (16, 16)
    rec = oracle_records_fp32(sc.params(), sc.sh_degree, cam, tile)
    frame, proj, bins, img, T, stop = _gpu([rec], [cam], tile, (0, 0, 0))
    ranges = bins.ranges.cpu().numpy()
    lens = ranges[:, 1] - ranges[:, 0]
    rng = np.random.default_rng(11)
    busy = np.nonzero(lens > 0)[0]
    tiles = sorted(set(rng.choice(busy, 24, replace=False).tolist()) | set(np.argsort(lens)[-4:].tolist()))
    mask = _tile_mask(cam, tile, tiles)
    d_image = np.where(mask[None], rng.normal(0, 1, (3, cam.height, cam.width)), 0).astype(np.float32)
    o, g = _oracle_fwd(rec, cam, tile, (0, 0, 0), tiles=tiles, d_image=d_image)
    counts = R.raster_count(proj, bins, frame).cpu().numpy().reshape(cam.height, cam.width, 2)
    _compare_fwd(o, frame.view_image(img, 0).cpu().numpy(), frame.view_pixels(T, 0).cpu().numpy(),
                 frame.view_pixels(stop, 0).cpu().numpy(), mask=mask, counts=counts, max_flag_frac=5e-3)
    for st in (None, stop):   # recomputed cut-off, and the forward's stop indices (the bench's path)
        rg = R.raster_bwd(proj, bins, frame, img, torch.as_tensor(d_image.reshape(-1)).cuda(), stop=st)
        torch.cuda.synchronize()
        got = dict(d_mean2d=rg.d_mean2d.cpu().numpy(), d_conic=rg.d_conic_opacity[:, :3].cpu().numpy(),
                   d_opacity=rg.d_conic_opacity[:, 3].cpu().numpy(), d_rgb=rg.d_rgb[:, :3].cpu().numpy())
        for k in got:
            e = rel_l2(got[k], g[k])
            assert e < GRAD_TOL, (k, e, st is not None)


@pytest.mark.parametrize("use_stop", [False, True])
@pytest.mark.parametrize("depth", [0, 1])
@pytest.mark.parametrize("n,size,tile", [
    (190, (64, 64), (16, 16)),       # 16 tiles: a quarter of a tile per CTA; one short window
    (2500, (61, 50), (16, 16)),      # lists over several windows, ragged edges
    (300, (250, 183), (16, 16)),     # 192 tiles: half a tile per CTA; too few records a tile below
    (2600, (250, 183), (16, 16)),
    (5000, (333, 301), (16, 16)),    # 399 tiles: whole tiles, four-warp CTAs
    (900, (37, 64), (8, 8)), (3000, (200, 190), (8, 8)),
    (3000, (130, 70), (16, 32)), (3000, (70, 130), (32, 16))])
def test_tile_backward_matches_per_splat_backward(n, size, tile, depth, use_stop):
    """gs_raster_bwd's paths by frame size against gs_raster_bwd_splat on the same lists:
    FP32 on both sides, the sums in another order (1e-4, as between the two backwards
    elsewhere). A wide camera puts 60 to 700 entries in a tile's list: one window and several,
    with bucket counts that are no multiple of the warps'."""
    sc = synth.small_scene(n, n=n, width=size[0], height=size[1])
    frame = R.Frame(sc.cameras, tile=tile)
    P = R.to_device_params(sc.params())
    proj = R.project(P, 0, frame)
    bins = R.bin_sort(proj, frame)
    ckpt = R.alloc_ckpt(frame, bins)
    bg = (0.2, 0.1, 0.4)
    img, _, stop = R.raster_fwd_ckpt(proj, bins, frame, ckpt, bg)
    d_image = torch.randn(img.shape, generator=torch.Generator("cuda").manual_seed(n), device="cuda")
    want = R.raster_bwd_splat(proj, bins, frame, img, d_image, stop, ckpt)
    got = R.raster_bwd(proj, bins, frame, img, d_image, bg, stop=stop if use_stop else None, stage_depth=depth)
    for k in ("d_mean2d", "d_conic_opacity", "d_rgb"):
        a, b = getattr(got, k).cpu().numpy(), getattr(want, k).cpu().numpy()
        assert np.linalg.norm(b) > 0 and rel_l2(a, b) < 1e-4, k


@pytest.mark.parametrize("use_stop", [False, True])
@pytest.mark.parametrize("depth", [0, 1])
@pytest.mark.parametrize("n,size,tile,zoom", [
    (200, (64, 64), (16, 16), 3.0), (2500, (61, 50), (16, 16), 1.0),     # quarters of tiles; short, and several windows
    (2400, (250, 183), (16, 16), 5.0), (9000, (250, 183), (16, 16), 2.5),   # halves; short, and mixed
    (9000, (333, 301), (16, 16), 4.0), (60_000, (333, 301), (16, 16), 4.0),   # whole tiles, four-warp CTAs
    (3000, (120, 120), (8, 8), 4.0), (20_000, (200, 190), (8, 8), 2.0), (3000, (130, 70), (16, 32), 3.0),
    (4000, (70, 130), (32, 16), 1.0)])
def test_tile_backward_matches_per_pixel_backward(n, size, tile, zoom, depth, use_stop):
    """raster_bwd_tile_kernel, its short lists, its split tiles and its windows included, against
    raster_bwd_kernel, which shares neither walk nor reduction with it: a large second view beside the
    small one takes the frame beyond the line between them. FP32 on both sides, the sums in another
    order: 1e-4, as between the backwards elsewhere."""
    sc = synth.small_scene(n, n=n, width=size[0], height=size[1])
    cam = sc.cameras[0]
    cam = synth.Camera(cam.R, cam.t, cam.fx * zoom, cam.fy * zoom, cam.cx, cam.cy, cam.width, cam.height)
    big = synth.Camera(cam.R, cam.t, 1000., 1000., 640., 480., 1280, 960)
    P = R.to_device_params(sc.params())
    got = {}
    for name, cams in (("tile", [cam]), ("pixel", [cam, big])):
        frame = R.Frame(cams, tile=tile)
        proj = R.project(P, 0, frame)
        bins = R.bin_sort(proj, frame)
        img, _, stop = R.raster_fwd(proj, bins, frame, store_stop=True)
        d_image = torch.zeros_like(img)
        d_image[:3 * size[0] * size[1]] = torch.randn(3 * size[0] * size[1], device="cuda",
                                                      generator=torch.Generator("cuda").manual_seed(n))
        rg = R.raster_bwd(proj, bins, frame, img, d_image, stop=stop if use_stop else None, stage_depth=depth)
        got[name] = {k: getattr(rg, k)[:n].cpu().numpy() for k in ("d_mean2d", "d_conic_opacity", "d_rgb")}
        if name == "tile":
            lens = (bins.ranges[:, 1] - bins.ranges[:, 0]).cpu().numpy()
            print(f"lists of {lens.min()} to {lens.max()} entries, {(lens <= 32).mean():.2f} of them up to 32")
    for k, b in got["pixel"].items():
        assert np.linalg.norm(b) > 0 and rel_l2(got["tile"][k], b) < 1e-4, k


@pytest.mark.parametrize("bad", [np.nan, np.inf])
@pytest.mark.parametrize("backward", ["tile", "tile, cut-off recomputed", "splat"])
def test_backwards_agree_on_records_that_are_no_numbers(backward, bad):
    """An opacity that is NaN or infinite counts as 0.99 in the forward (min(0.99, sigma)), and so for the
    transmittance of what lies behind it (here a record over every block of the view, in the middle of
    the scene): the other records' gradients against raster_bwd_kernel's (a large second view beside the
    small one), tolerance as above."""
    n, w, h = 2500, 120, 90
    sc = synth.small_scene(3, n=n, width=w, height=h)
    cam = sc.cameras[0]
    big = synth.Camera(cam.R, cam.t, 1000., 1000., 640., 480., 1280, 960)
    P = R.to_device_params(sc.params())
    rest = torch.arange(n, device="cuda") != 5
    got = {}
    for name, cams in ((backward, [cam]), ("pixel", [cam, big])):
        frame = R.Frame(cams)
        proj = R.project(P, 0, frame)
        proj.mean2d[5] = torch.tensor([60.0, 45.0])
        proj.conic_opacity[5] = torch.tensor([1e-5, 0.0, 1e-5, float(bad)])
        proj.rgb[5] = torch.tensor([0.2, 0.9, 0.5, 9.0])
        proj.depth[5], proj.radius[5] = 4.0, 900
        proj.rect[5] = torch.tensor([0, 0, 8, 6], dtype=torch.int16)
        bins = R.bin_sort(proj, frame)
        ckpt = R.alloc_ckpt(frame, bins)
        img, _, stop = R.raster_fwd_ckpt(proj, bins, frame, ckpt)
        d_image = torch.zeros_like(img)
        d_image[:3 * w * h] = torch.randn(3 * w * h, generator=torch.Generator("cuda").manual_seed(1), device="cuda")
        if name == "splat":
            rg = R.raster_bwd_splat(proj, bins, frame, img, d_image, stop, ckpt)
        else:
            rg = R.raster_bwd(proj, bins, frame, img, d_image, stop=None if "recomputed" in name else stop)
        got[name] = {k: getattr(rg, k)[:n][rest].cpu().numpy() for k in ("d_mean2d", "d_conic_opacity", "d_rgb")}
        assert torch.isfinite(img).all()
    for k, b in got["pixel"].items():
        assert np.linalg.norm(b) > 0 and rel_l2(got[backward][k], b) < 1e-4, k
