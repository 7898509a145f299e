"""gs_downscale / gs_spectrum_l1 and the energy-guided schedule built on them,
against the FP64 oracle (oracle/schedule.py) on the same FP32 images."""
import numpy as np
import pytest
import torch

from oracle import schedule as osch
from paper_2507_20239_gb300 import schedule as S

pytestmark = pytest.mark.gpu


def _image(seed, C, H, W):
    rng = np.random.default_rng(seed)
    y, x = np.mgrid[0:H, 0:W]
    base = 0.5 + 0.3 * np.sin(x / 7.0 + seed) * np.cos(y / 11.0)
    return np.stack([base + 0.1 * rng.normal(size=(H, W)) for _ in range(C)]).astype(np.float32)


@pytest.mark.parametrize("r", [1, 2, 3, 4, 8])
def test_downscale_matches_oracle(r):
    img = _image(0, 3, 207, 311)
    got = S.downscale(torch.as_tensor(img).cuda(), r).cpu().numpy()
    want = osch.downscale(img, r)
    assert got.shape == want.shape == (3, osch.downscaled_size(207, r), osch.downscaled_size(311, r))
    assert np.abs(got - want).max() < 1e-5


@pytest.mark.parametrize("shape", [(3, 413, 623), (1, 37, 53), (2, 1, 1)])
def test_spectrum_l1_matches_oracle(shape):
    img = _image(1, *shape)
    got = S.spectrum_l1(torch.as_tensor(img).cuda())
    want = osch.spectrum_l1(img)
    assert abs(got - want) <= 1e-5 * want


@pytest.mark.parametrize("shape", [(1, 2, 2), (5, 3, 3), (1, 63, 64), (1, 65, 127), (2, 128, 130), (3, 129, 14),
                                   (17, 16, 257)])
def test_spectrum_l1_at_tile_edges(shape):
    """Line, frequency and column counts around the DFT passes' tiles (16 rows, 8 columns,
    64-position chunks, 128 frequencies), odd and even widths (the folded half spectrum).
    A coefficient's FP32 error (at most N roundings of partial sums below 0.8 N) has no
    preferred sign, so the sum of the magnitudes holds 1e-5."""
    img = _image(3, *shape)
    got = S.spectrum_l1(torch.as_tensor(img).cuda())
    want = osch.spectrum_l1(img)
    assert abs(got - want) <= 1e-5 * want


@pytest.mark.parametrize("shape", [(8, 397, 333), (9, 259, 515), (3, 530, 255)])
def test_spectrum_l1_larger_tiles(shape):
    """Images of blocks enough for the passes' larger tiles (16 rows, two frequencies a
    thread), with ragged last tiles; tolerance as above."""
    test_spectrum_l1_at_tile_edges(shape)


@pytest.mark.parametrize("shape,r", [((3, 207, 311), 16), ((2, 207, 311), 17), ((1, 207, 311), 40), ((2, 5, 33), 2),
                                     ((1, 9, 64), 2), ((1, 40, 3), 8)])
def test_downscale_filter_widths(shape, r):
    """The tabulated filters up to 36 taps and the general kernel beyond, ragged output tiles."""
    img = _image(4, *shape)
    got = S.downscale(torch.as_tensor(img).cuda(), r).cpu().numpy()
    want = osch.downscale(img, r)
    assert got.shape == want.shape and np.abs(got - want).max() < 1e-5


def test_energy_schedule_matches_oracle():
    imgs = [_image(s, 3, 413, 623) for s in (2, 3)]
    E, T, st = S.energy_schedule(imgs, K=8, T_densify=25000)
    Eo = osch.energies(imgs, 8)
    assert np.all(np.abs(E - Eo) <= 1e-5 * Eo)
    To = osch.iterations(Eo, 25000)
    # a T_r may differ by one only where E_r / E_1 T_densify lies within the FP32
    # error of a rounding boundary
    frac = Eo / Eo[0] * 25000 + 0.5
    near = np.abs(frac - np.round(frac)) < 1e-5 * 25000
    assert np.all((T == To) | (near & (np.abs(T - To) == 1)))
    assert st == osch.stages(To) or near.any()
    assert T[0] == 25000 and all(T[i] >= T[i + 1] for i in range(7))


def test_spectrum_rejects_oversized_images():
    assert S.lib().gs_spectrum_workspace_size(3, 4097, 100) == 0
    with pytest.raises(RuntimeError):
        S.spectrum_l1(torch.zeros(1, 4097, 8, device="cuda"))


def test_energy_schedule_drives_training():
    from paper_2507_20239_gb300 import rasterizer as R, synth
    from paper_2507_20239_gb300.train import Schedule, Trainer, energy_stages, orbit_views, render_targets
    full = orbit_views(2, 320, 212, 320.0, divisors=(1,))[1]
    gt = synth.surface_scene(13, 60_000, 3)
    targets = render_targets(gt.params(), 3, full)
    stages, views, (E, T) = energy_stages(full, targets, 4, 300)
    assert stages[0][0] == 0 and stages[-1][1] == 1
    assert [s[1] for s in stages] == sorted((s[1] for s in stages), reverse=True)      # coarse to fine
    assert all(m == R.DENSIFY_SPLIT_ONLY for _, r, m in stages if r > 1)
    for r, (cams, imgs) in views.items():
        assert imgs[0].shape == (3, S.downscaled_size(212, r), S.downscaled_size(320, r))
        assert cams[0].width == imgs[0].shape[2]
    sched = Schedule(stages=stages, total=400, densify_until=300, sh_every=100)
    tr = Trainer(synth.surface_scene(3, 10_000, 3).params(), views, sched, extent=4.4)
    hist = tr.run(log_every=100)
    assert tr.event == 3 and hist[-1][2] < hist[0][2]


def _column_spectrum(x0, x1):
    """||E||_1 of the one-column image (x0, x1, 0, 0), whose DFT takes one rounding per coefficient: the
    twiddles are 1, -i, -1 and i, so Y = (x0 + x1, x0 - i x1, x0 - x1, x0 + i x1) in FP32."""
    a, b = np.float32(x0), np.float32(x1)
    with np.errstate(all="ignore"):
        return abs(np.float64(a + b)) + abs(np.float64(a - b)) + 2 * np.hypot(np.float64(a), np.float64(b))


@pytest.mark.parametrize("seed", range(8))
def test_spectrum_magnitudes_beyond_fp32(seed):
    """The sum of exactly known coefficients: each magnitude within 2^-46 of its value and the sums in
    pairs of 2^-47 and FP64, so 2^-43 with room for 16 terms; an FP32 root would be off by 2^-25."""
    rng = np.random.default_rng(seed)
    x = (rng.uniform(0.5, 1.0, (4, 2)) * 2.0 ** rng.integers(-3, 3, (4, 2))).astype(np.float32)
    for c in (1, 4):
        img = np.zeros((c, 4, 1), np.float32)
        img[:, :2, 0] = x[:c]
        want = sum(_column_spectrum(*v) for v in x[:c])
        got = S.spectrum_l1(torch.as_tensor(img).cuda())
        assert abs(got - want) <= 2.0 ** -43 * want, (c, got, want)


@pytest.mark.parametrize("x0,x1", [(3e-13, 4e-13), (3e-20, 4e-20), (1.5e-30, 1e-31), (1e-12, 3e-25), (3e16, 4e16),
                                   (2e30, 1.25e31), (1e15, 1e-3), (3.0, 4e-20), (0.0, 2e-15), (0.0, 0.0)])
def test_spectrum_magnitudes_over_the_range(x0, x1):
    """Magnitudes around and outside the range that the FP32 pairs take (1e-12 to 1e15)."""
    img = np.array([x0, x1, 0, 0], np.float32).reshape(1, 4, 1)
    got, want = S.spectrum_l1(torch.as_tensor(img).cuda()), _column_spectrum(x0, x1)
    assert abs(got - want) <= 2.0 ** -43 * want, (got, want)


@pytest.mark.parametrize("bad", [np.nan, np.inf, -np.inf])
def test_spectrum_of_images_with_non_finite_values(bad):
    img = np.ones((1, 8, 8), np.float32)
    img[0, 3, 5] = bad
    assert np.isnan(S.spectrum_l1(torch.as_tensor(img).cuda()))


def test_downscale_of_an_image_wider_than_fp32_positions():
    """2^28 columns at scale 17: the positions' FP32 rounding widens some filters to 37 taps, one more
    than the tabulated kernel has room for. Sampled columns against the filter's definition in FP32,
    whose position (j + 1/2) s - 1/2 may be one or two roundings."""
    n, r, f = 1 << 28, 17, np.float32
    x = torch.rand(1, 1, n, generator=torch.Generator("cuda").manual_seed(5), device="cuda")
    got = S.downscale(x, r)[0, 0]
    m = got.shape[0]
    rng = np.random.default_rng(6)
    s = f(n) / f(m)
    widest = 0
    for j in np.concatenate([rng.integers(0, m, 300), np.arange(m - 100, m)]):
        err = []
        for c in ((f(j) + f(0.5)) * s - f(0.5), f(np.float64(f(j) + f(0.5)) * np.float64(s) - 0.5)):
            k0, k1 = max(0, int(np.ceil(c - s))), min(n - 1, int(np.floor(c + s)))
            w = np.maximum(f(0), f(1) - np.abs(np.arange(k0, k1 + 1).astype(f) - c) / s).astype(np.float64)
            err.append(abs(float(got[j]) - (w * x[0, 0, k0:k1 + 1].cpu().numpy().astype(np.float64)).sum() / w.sum()))
            widest = max(widest, k1 - k0 + 1)
        assert min(err) < 1e-5, j
    assert widest == 37


@pytest.mark.parametrize("shape,r", [((1, 2600, 2688), 8), ((1, 2600, 2696), 8), ((2, 2650, 2650), 16)])
def test_downscale_of_large_images(shape, r):
    """Scales of whole 32-byte steps below and above seven million pixels (the tabulated and the general
    kernel); tolerance as above."""
    img = _image(9, *shape)
    got = S.downscale(torch.as_tensor(img).cuda(), r).cpu().numpy()
    want = osch.downscale(img, r)
    assert got.shape == want.shape and np.abs(got - want).max() < 1e-5
