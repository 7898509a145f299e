"""gs_bin_sort: keys, order and per-tile ranges bit-exact against the oracle's
definition (sort by tile, FP32 depth bits, record index) on the same FP32 records."""
import numpy as np
import pytest
import torch

from oracle import project as oproj
from oracle import raster as oras
from paper_2507_20239_gb300 import rasterizer as R
from paper_2507_20239_gb300 import synth
from tests.gs_fixtures import bins_pairs, dev_params, exact_list_check, oracle_records_fp32, records_to_gpu, scene

pytestmark = pytest.mark.gpu


def _synthetic_records(seed, n, cams, tile):
    recs = []
    rng = np.random.default_rng(1000 + seed)
    for v, cam in enumerate(cams):
        m2, dep, rad = synth.random_records(seed + v, n, cam.width, cam.height)
        sx = rng.uniform(0.6, 14, n)
        sy = rng.uniform(0.6, 14, n)
        conic_f = np.stack([1 / sx ** 2, rng.normal(0, 0.5, n), 1 / sy ** 2], 1).astype(np.float32)
        o = rng.uniform(0.01, 0.99, n)
        q_max = (2 * np.log(255 * o)).astype(np.float32)
        half = oproj.footprint_half(conic_f.astype(np.float64), q_max.astype(np.float64)).astype(np.float32)
        half[rad == 0] = -1
        gx, gy = oproj.tile_grid(cam.width, cam.height, *tile)
        rect = oproj.tile_rect(m2, half, tile[0], tile[1], gx, gy)
        area = (rect[:, 2] - rect[:, 0]) * (rect[:, 3] - rect[:, 1])
        rad = np.where(area > 0, np.maximum(rad, 1), 0).astype(np.int32)
        rect[area <= 0] = 0
        z3 = np.zeros((n, 3), np.float32)
        recs.append(dict(mean2d=m2, depth=np.where(rad > 0, dep, 0).astype(np.float32), radius=rad, rect=rect,
                         conic_f=conic_f, q_max=q_max, opacity=o.astype(np.float32), rgb=z3, grid=(gx, gy),
                         width=cam.width, height=cam.height, tile=tuple(tile)))
    return recs


def _oracle_bins(recs, frame):
    cat = lambda k: np.concatenate([r[k] for r in recs])
    n = recs[0]["rect"].shape[0]
    V = len(recs)
    arr = dict(mean2d=cat("mean2d"), conic_f=cat("conic_f"), q_max=cat("q_max"), rect=cat("rect"),
               depth=cat("depth"))
    per = lambda i: np.repeat([frame.views[v][i] for v in range(V)], n).astype(np.int64)
    return oras.bin_and_sort(arr, per(3), per(4), per(0), per(1), frame.tile[0], frame.tile[1], frame.n_tiles)


def _check(recs, cams, tile, capacity=None, fused_bits=0):
    frame = R.Frame(cams, tile=tile, sort_fused_bits=fused_bits)
    proj = records_to_gpu(recs)
    keys, vals, ranges = _oracle_bins(recs, frame)
    bins = R.bin_sort(proj, frame, capacity=capacity, want_keys=True)
    torch.cuda.synchronize()
    M = int(bins.count.item())
    assert M == len(vals)
    assert np.array_equal(bins.vals[:M].cpu().numpy().view(np.uint32), vals)
    assert np.array_equal(bins.keys[:M].cpu().numpy().view(np.uint64), keys)
    assert np.array_equal(bins.ranges.cpu().numpy().view(np.uint32), ranges)
    return M


@pytest.mark.parametrize("tile", [(16, 16), (8, 8), (16, 32)])
def test_bin_sort_synthetic_records_single_view(tile):
    cam = synth.Camera(np.eye(3, dtype=np.float32), np.zeros(3, np.float32), 100., 100., 150., 100., 300, 200)
    recs = _synthetic_records(0, 20000, [cam], tile)
    assert _check(recs, [cam], tile) > 20000


def test_bin_sort_mixed_resolution_views():
    cams, _ = synth.mixed_resolution_cameras(6)
    recs = _synthetic_records(10, 30000, cams, (16, 16))
    _check(recs, cams, (16, 16))


@pytest.mark.parametrize("fused_bits", [1, 3, 8])
def test_bin_sort_fused_bits_override(fused_bits):
    # the number of tile-id bits sorted during emission is a tuning knob: every
    # choice gives the same keys, order and ranges
    cams, _ = synth.mixed_resolution_cameras(6)
    recs = _synthetic_records(11, 20000, cams, (16, 16))
    _check(recs, cams, (16, 16), fused_bits=fused_bits)


def test_bin_sort_rejects_fused_bits_beyond_tile_id_width():
    cam = synth.Camera(np.eye(3, dtype=np.float32), np.zeros(3, np.float32), 50., 50., 17., 9., 35, 19)
    recs = _synthetic_records(3, 500, [cam], (16, 16))      # 6 tiles: 3-bit tile ids
    frame = R.Frame([cam], tile=(16, 16), sort_fused_bits=4)
    with pytest.raises(RuntimeError):
        R.bin_sort(records_to_gpu(recs), frame)


def test_bin_sort_edge_cases():
    cam = synth.Camera(np.eye(3, dtype=np.float32), np.zeros(3, np.float32), 50., 50., 17., 9., 35, 19)
    # all culled -> empty lists
    recs = _synthetic_records(3, 500, [cam], (16, 16))
    for k in ("radius", "depth"):
        recs[0][k][:] = 0
    recs[0]["rect"][:] = 0
    assert _check(recs, [cam], (16, 16)) == 0
    # a single record whose footprint covers all 6 tiles of its rectangle
    recs = _synthetic_records(4, 1, [cam], (16, 16))
    recs[0]["radius"][:] = 50
    recs[0]["rect"][0] = [0, 0, 3, 2]
    recs[0]["depth"][:] = 1.0
    recs[0]["mean2d"][0] = [17.0, 9.0]
    recs[0]["conic_f"][0] = [1e-4, 0.0, 1e-4]
    assert _check(recs, [cam], (16, 16)) == 6
    # a thin diagonal footprint inside a large rectangle: only the tiles it crosses
    recs[0]["conic_f"][0] = [1.0, -1.0, 1e-4]
    recs[0]["q_max"][0] = 4.0
    assert 0 < _check(recs, [cam], (16, 16)) < 6
    # all records at exactly the same depth (ties -> record order)
    recs = _synthetic_records(5, 5000, [cam], (16, 16))
    recs[0]["depth"][recs[0]["radius"] > 0] = 2.5
    _check(recs, [cam], (16, 16))


def test_bin_sort_capacity_overflow_reports_and_retries():
    cam = synth.Camera(np.eye(3, dtype=np.float32), np.zeros(3, np.float32), 100., 100., 150., 100., 300, 200)
    recs = _synthetic_records(7, 3000, [cam], (16, 16))
    frame = R.Frame([cam])
    proj = records_to_gpu(recs)
    _, vals, _ = _oracle_bins(recs, frame)
    bins = R.alloc_bins(frame, proj.mean2d.shape[0], capacity=len(vals) // 2)
    R.bin_sort_into(proj, frame, bins)
    torch.cuda.synchronize()
    assert int(bins.error.item()) == 2                # GS_ERR_CAPACITY
    # the required size is reported: the capacity also holds one entry per tile row
    # of each visible record's rectangle while the lists are built
    assert int(bins.count.item()) == max(len(vals), _rect_rows(recs))
    assert np.all(bins.ranges.cpu().numpy() == 0)     # and every list is empty
    # the binding grows the buffer and redoes the sort
    _check(recs, [cam], (16, 16), capacity=len(vals) // 2)


def _rect_rows(recs):
    rows = 0
    for r in recs:
        x0, y0, x1, y1 = (r["rect"][:, i].astype(np.int64) for i in range(4))
        live = (r["radius"] > 0) & (x1 > x0) & (y1 > y0)
        rows += int(((y1 - y0) * live).sum())
    return rows


def test_bin_sort_rectangle_rows_beyond_the_entry_count():
    """Tall one-column rectangles around small footprints: the rows the binning
    visits (13 per record) outnumber the entries (about one per record), so the
    first capacity (8 entries per record) overflows on the rows alone; the reported
    size covers them and the retry gives the exact lists."""
    cam = synth.Camera(np.eye(3, dtype=np.float32), np.zeros(3, np.float32), 100., 100., 150., 100., 300, 200)
    n = 20000
    recs = _synthetic_records(9, n, [cam], (16, 16))
    rng = np.random.default_rng(99)
    r = recs[0]
    tx, ty = rng.integers(0, 19, n), rng.integers(0, 13, n)
    r["mean2d"][:] = np.stack([16 * tx + 8, 16 * ty + 8], 1).astype(np.float32)
    r["conic_f"][:] = [1.0, 0.0, 1.0]
    r["q_max"][:] = np.float32(2 * np.log(255 * 0.5))
    r["rect"][:] = np.stack([tx, np.zeros(n), tx + 1, np.full(n, 13)], 1).astype(r["rect"].dtype)
    r["radius"][:] = 3
    r["depth"][:] = rng.uniform(1.0, 5.0, n).astype(np.float32)
    assert _rect_rows(recs) == 13 * n
    frame = R.Frame([cam])
    bins = R.alloc_bins(frame, n, capacity=8 * n)
    R.bin_sort_into(records_to_gpu(recs), frame, bins)
    torch.cuda.synchronize()
    assert int(bins.error.item()) == 2 and int(bins.count.item()) == 13 * n
    assert _check(recs, [cam], (16, 16), capacity=8 * n) == n


def test_bin_sort_full_size_orbit_scene():
    sc = scene("orbit")                       # 1.5M Gaussians, 1246x826, 16x16 tiles
    cam = sc.cameras[0]
    rec = oracle_records_fp32(sc.params(), sc.sh_degree, cam)
    M = _check([rec], [cam], (16, 16))
    assert M > 1_000_000


def test_full_view_lists_hold_every_exact_fp64_pair():
    """The benchmark view's lists, made by the GPU path end to end (gs_project then
    gs_bin_sort), against the exact FP64 geometry of the footprint ellipse on the
    GPU's own FP32 records: every (tile, record) pair the exact test keeps beyond the
    derived FP32 margin is listed, and every listed pair lies within it."""
    sc = scene("orbit")
    cam = sc.cameras[0]
    frame = R.Frame([cam])
    proj = R.project(dev_params(sc), sc.sh_degree, frame)
    bins = R.bin_sort(proj, frame)
    torch.cuda.synchronize()
    co = proj.conic_opacity.cpu().numpy()
    tiles, recs = bins_pairs(bins, frame.n_tiles)
    listed, must, between = exact_list_check(proj.mean2d.cpu().numpy(), co[:, :3], proj.rgb[:, 3].cpu().numpy(),
                                             proj.radius.cpu().numpy(), cam.width, cam.height, (16, 16), tiles, recs)
    print(f"listed {listed}, exact-with-margin {must}, within the margin {between}")
    assert listed > 10_000_000 and must > 0.99 * listed and between < 1e-3 * listed


def _wide(seed, n, width, height, tile=(16, 16), footprint=1.0):
    cam = synth.Camera(np.eye(3, dtype=np.float32), np.zeros(3, np.float32), 100., 100., width / 2, height / 2,
                       width, height)
    return _synthetic_records(seed, n, [cam], tile), cam


@pytest.mark.parametrize("n,size,tile", [
    (1, (16, 16), (16, 16)), (63, (33, 17), (16, 16)), (2047, (300, 200), (16, 16)), (2049, (300, 200), (16, 16)),
    (70_001, (100, 60), (8, 8)),            # few tiles, long lists: records of one chunk share every tile
    (320_000, (640, 480), (16, 16)),        # chunks of equal weight instead of equal counts
    (400_000, (1250, 830), (8, 8)),         # 16328 tiles: one mask word per tile
    (20_000, (1700, 1300), (8, 8))])        # 34,669 tiles in a view: emitted pairs and radix passes
def test_bin_sort_paths_by_frame_size(n, size, tile):
    """Counting and pair paths at the edges of their batches (32 and 256 records), sort
    partitions (2048), chunks and tables."""
    recs, cam = _wide(n, n, *size, tile=tile)
    _check(recs, [cam], tile)


def test_bin_sort_many_records_in_one_place():
    """Every record over the same few tiles, of depths in few values, in a view whose other
    tiles stay empty: full masks in the emission, one chunk's weight in one place, ties kept in
    record order; and a view in which nothing is visible beside it."""
    recs, cam = _wide(21, 330_000, 400, 300)
    r = recs[0]
    n = len(r["radius"])
    rng = np.random.default_rng(5)
    r["mean2d"][:] = np.stack([rng.uniform(100, 130, n), rng.uniform(90, 120, n)], 1).astype(np.float32)
    r["conic_f"][:] = [1 / 36.0, 0.0, 1 / 36.0]
    r["q_max"][:] = np.float32(2 * np.log(255 * 0.5))
    half = oproj.footprint_half(r["conic_f"].astype(np.float64), r["q_max"].astype(np.float64)).astype(np.float32)
    r["rect"][:] = oproj.tile_rect(r["mean2d"], half, 16, 16, *r["grid"])
    r["radius"][:] = 20
    r["depth"][:] = rng.choice(np.float32([0.5, 1.0, 1.0000001, 7.25, 3e7]), n)
    empty = {k: (v.copy() if isinstance(v, np.ndarray) else v) for k, v in r.items()}
    for k in ("radius", "depth", "rect"):
        empty[k][:] = 0
    _check([r, empty], [cam, cam], (16, 16))


# ---- the general path (emitted pairs and radix passes): views of more than 20000 tiles, or more than
# 1024 views, with the cases that smaller frames give the counting path

def _large_views(seed, n, views=1):
    """8 x 8 tiles: 34,669 of a view, with smaller ones beside it."""
    sizes = [(1700, 1300), (425, 325), (850, 650)][:views]
    cams = [synth.Camera(np.eye(3, dtype=np.float32), np.zeros(3, np.float32), 100., 100., w / 2, h / 2, w, h)
            for w, h in sizes]
    return _synthetic_records(seed, n, cams, (8, 8)), cams


@pytest.mark.parametrize("fused_bits", [0, 1, 3, 8])
def test_pair_path_fused_bits_and_views(fused_bits):
    recs, cams = _large_views(31, 6000, views=3)
    _check(recs, cams, (8, 8), fused_bits=fused_bits)


def test_pair_path_capacity_overflow_reports_and_retries():
    recs, cams = _large_views(32, 3000)
    frame, proj = R.Frame(cams, tile=(8, 8)), records_to_gpu(recs)
    _, vals, _ = _oracle_bins(recs, frame)
    bins = R.alloc_bins(frame, proj.mean2d.shape[0], capacity=len(vals) // 2)
    R.bin_sort_into(proj, frame, bins)
    torch.cuda.synchronize()
    assert int(bins.error.item()) == 2 and int(bins.count.item()) == max(len(vals), _rect_rows(recs))
    assert np.all(bins.ranges.cpu().numpy() == 0)
    _check(recs, cams, (8, 8), capacity=len(vals) // 2)


def test_pair_path_rectangle_rows_beyond_the_entry_count():
    recs, cams = _large_views(33, 2000)
    r, n = recs[0], 2000
    rng = np.random.default_rng(98)
    tx, ty = rng.integers(0, 212, n), rng.integers(0, 162, n)
    r["mean2d"][:] = np.stack([8 * tx + 4, 8 * ty + 4], 1).astype(np.float32)
    r["conic_f"][:] = [4.0, 0.0, 4.0]
    r["q_max"][:] = np.float32(2 * np.log(255 * 0.5))
    r["rect"][:] = np.stack([tx, np.zeros(n), tx + 1, np.full(n, 163)], 1).astype(r["rect"].dtype)
    r["radius"][:] = 2
    r["depth"][:] = rng.uniform(1.0, 5.0, n).astype(np.float32)
    frame = R.Frame(cams, tile=(8, 8))
    bins = R.alloc_bins(frame, n, capacity=8 * n)
    R.bin_sort_into(records_to_gpu(recs), frame, bins)
    torch.cuda.synchronize()
    assert int(bins.error.item()) == 2 and int(bins.count.item()) == _rect_rows(recs) == 163 * n
    assert _check(recs, cams, (8, 8), capacity=8 * n) >= n


def test_pair_path_ties_and_empty_views():
    recs, cams = _large_views(34, 4000, views=2)
    for r in recs:
        r["depth"][r["radius"] > 0] = 2.5
    _check(recs, cams, (8, 8))                       # ties: record order
    for k in ("radius", "depth", "rect"):
        recs[0][k][:] = 0
    _check(recs, cams, (8, 8))                       # nothing visible in one view
    for k in ("radius", "depth", "rect"):
        recs[1][k][:] = 0
    assert _check(recs, cams, (8, 8)) == 0           # nor in the other


@pytest.mark.parametrize("views", [1024, 1025])      # the counting path's most views, and one more
def test_bin_sort_of_many_small_views(views):
    cams = [synth.Camera(np.eye(3, dtype=np.float32), np.zeros(3, np.float32), 30., 30., w / 2, 9., w, 17)
            for w in (15 + v % 20 for v in range(views))]
    recs = _synthetic_records(40, 40, cams, (16, 16))
    assert _check(recs, cams, (16, 16)) > views


@pytest.mark.parametrize("n,sizes", [
    (3000, [(1000, 700)] * 2),                              # 11,000 tiles each: blocks of 512 threads
    (60_000, [(700, 660)]),                                 # 7304 tiles: one word of mask, two blocks an SM
    (9_900, [(1000, 700), (500, 350), (250, 175)]),         # unequal views, counted
    (10_100, [(1000, 700), (500, 350), (250, 175)]),        # unequal views of more records: pairs
    (700, [(840, 800)] * 7), (120_100, [(840, 800)] * 7)])  # 73,500 tiles in all: pairs; counted from 12 records a tile
def test_bin_sort_on_both_sides_of_the_plans_lines(n, sizes):
    cams = [synth.Camera(np.eye(3, dtype=np.float32), np.zeros(3, np.float32), 100., 100., w / 2, h / 2, w, h)
            for w, h in sizes]
    _check(_synthetic_records(50, n, cams, (8, 8)), cams, (8, 8))


@pytest.mark.parametrize("sizes,tile,counts", [
    ([(1246, 826)], (16, 16), [75_777, 75_776, 40_000, 1, 0]),
    ([(1000, 700), (500, 350)], (8, 8), [10_001, 10_000, 9_999, 300, 0]),   # pairs, then counted
    ([(1700, 1300)], (8, 8), [3000, 1, 0])])
def test_bins_sized_for_more_records_hold_fewer(sizes, tile, counts):
    cams = [synth.Camera(np.eye(3, dtype=np.float32), np.zeros(3, np.float32), 100., 100., w / 2, h / 2, w, h)
            for w, h in sizes]
    frame = R.Frame(cams, tile=tile)
    bins = R.alloc_bins(frame, counts[0] * len(cams), capacity=1_500_000)
    for n in counts:
        recs = _synthetic_records(60, n, cams, tile)
        proj = records_to_gpu(recs)
        R.bin_sort_into(proj, frame, bins)
        assert int(bins.error.item()) == 0
        M, ranges = int(bins.count.item()), bins.ranges.cpu().numpy().view(np.uint32)
        if n == 0:
            assert M == 0 and not ranges.any()
            continue
        _, vals, want = _oracle_bins(recs, frame)
        assert M == len(vals) and np.array_equal(ranges, want)
        assert np.array_equal(bins.vals[:M].cpu().numpy().view(np.uint32), vals)
