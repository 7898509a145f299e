"""gs_project (EWA projection + SH colour) and gs_project_bwd against the FP64 oracle."""
import numpy as np
import pytest
import torch

from oracle import pipeline as opipe
from oracle import project as oproj
from paper_2507_20239_gb300 import rasterizer as R
from paper_2507_20239_gb300 import synth
from tests.gs_fixtures import dev_params, rel_l2, scene

pytestmark = pytest.mark.gpu


def _straddle_ok(pr, tile=16, tol=1e-4):
    """Records whose integer outputs (radius, rect, visibility) sit within rounding
    distance of a decision boundary in the FP64 oracle."""
    half = np.where(pr["half"] > 0, pr["half"], 0.0)
    hmax = half.max(1)
    near_int = np.abs(hmax - np.round(hmax)) < tol * np.maximum(hmax, 1)
    u, v = pr["mean2d"][:, 0], pr["mean2d"][:, 1]
    edges = np.stack([(u - half[:, 0]) / tile, (v - half[:, 1]) / tile, (u + half[:, 0]) / tile,
                      (v + half[:, 1]) / tile], 1)
    near_edge = (np.abs(edges - np.round(edges)) < tol).any(1)
    o = pr["opacity"]
    near_o = np.abs(o * 255 - 1) < 1e-5
    return near_int | near_edge | near_o


def _compare_projection(sc, cams, tile=(16, 16), sample=None):
    frame = R.Frame(cams, tile=tile)
    P = dev_params(sc)
    proj = R.project(P, sc.sh_degree, frame)
    torch.cuda.synchronize()
    n = sc.n
    idx = np.arange(n) if sample is None else sample
    sub = {k: v[idx] for k, v in sc.params().items()}
    for v, cam in enumerate(cams):
        pr = oproj.project_np(sub, sc.sh_degree, cam, tile[0], tile[1])
        rows = v * n + idx
        rad = proj.radius.cpu().numpy()[rows]
        rect = proj.rect_np()[rows]
        ok = _straddle_ok(pr, tile[0])
        vis_o = pr["visible"]
        vis_g = rad > 0
        bad = (vis_o != vis_g) & ~ok
        assert bad.sum() == 0, f"visibility differs on {bad.sum()} non-straddling records"
        both = vis_o & vis_g & ~ok
        assert np.array_equal(rad[both], pr["radius"][both])
        assert np.array_equal(rect[both], pr["rect"][both])
        assert both.sum() > 0.5 * vis_o.sum()
        vis = vis_o & vis_g
        m2 = proj.mean2d.cpu().numpy()[rows][vis]
        assert np.abs(m2 - pr["mean2d"][vis]).max() < 2e-3
        co = proj.conic_opacity.cpu().numpy()[rows][vis]
        cf = pr["conic_f"][vis]
        # the conic (A B; B C) = (A, A beta; A beta, gamma + A beta^2) implied by the
        # factored form, per record to a relative 1e-5 of its largest entry
        def mat(f):
            f = f.astype(np.float64)
            return np.stack([f[:, 0], f[:, 0] * f[:, 1], f[:, 2] + f[:, 0] * f[:, 1] ** 2], 1)
        mg, mo = mat(co[:, :3]), mat(cf)
        rel = np.abs(mg - mo).max(1) / np.abs(mo).max(1)
        assert rel.max() < 1e-5, rel.max()
        assert np.abs(co[:, 3] - pr["opacity"][vis]).max() < 1e-6
        dep = proj.depth.cpu().numpy()[rows][vis]
        assert np.abs(dep - pr["depth"][vis]).max() < 1e-5 * np.abs(pr["depth"][vis]).max()
        rgb = proj.rgb.cpu().numpy()[rows][vis]
        assert np.abs(rgb[:, :3] - pr["rgb"][vis]).max() < 2e-6
        assert np.abs(rgb[:, 3] - pr["q_max"][vis]).max() < 2e-5          # q_max = 2 ln(255 o)
        cl = proj.clamped.cpu().numpy()[rows][vis]
        want = (pr["clamped"][vis] * np.array([1, 2, 4])).sum(1)
        near0 = (np.abs(pr["rgb"][vis] - 0) < 1e-6).any(1)
        assert np.array_equal(cl[~near0], want[~near0])
        # culled rows are all zero
        cul = ~vis_g
        assert np.all(proj.conic_opacity.cpu().numpy()[rows][cul] == 0)


def test_project_small_scene():
    sc = scene("small")
    _compare_projection(sc, sc.cameras)


@pytest.mark.parametrize("tile", [(16, 16), (8, 8), (16, 32)])
def test_project_orbit_sh3_tiles(tile):
    sc = scene("orbit_small")
    _compare_projection(sc, sc.cameras, tile)


def test_project_multiview_mixed_resolution():
    sc = scene("batched_small")
    _compare_projection(sc, sc.cameras)


def test_project_full_size_sampled():
    sc = scene("orbit")                       # 1.5M Gaussians, SH degree 3, 1246x826
    rng = np.random.default_rng(0)
    sample = np.sort(rng.choice(sc.n, 20000, replace=False))
    _compare_projection(sc, sc.cameras, sample=sample)


def _rand_rec_grads(rng, R_, scale=1.0):
    return dict(d_mean2d=rng.normal(0, scale, (R_, 2)), d_conic=rng.normal(0, scale, (R_, 3)),
                d_opacity=rng.normal(0, scale, R_), d_rgb=rng.normal(0, scale, (R_, 3)))


def _rec_grads_gpu(gs):
    n = gs[0]["d_mean2d"].shape[0]
    V = len(gs)
    co = np.zeros((V * n, 4), np.float32)
    co[:, :3] = np.concatenate([g["d_conic"] for g in gs])
    co[:, 3] = np.concatenate([g["d_opacity"] for g in gs])
    rgb = np.zeros((V * n, 4), np.float32)
    rgb[:, :3] = np.concatenate([g["d_rgb"] for g in gs])
    t = lambda a: torch.as_tensor(np.ascontiguousarray(a, np.float32)).cuda()
    return R.RecGrads(t(np.concatenate([g["d_mean2d"] for g in gs])), t(co), t(rgb))


@pytest.mark.parametrize("name", ["small", "orbit_small", "batched_small"])
def test_project_vjp_matches_oracle(name):
    sc = scene(name)
    cams = sc.cameras
    n = min(sc.n, 4000)
    sub = {k: v[:n] for k, v in sc.params().items()}
    frame = R.Frame(cams)
    P = {k: torch.as_tensor(np.ascontiguousarray(v)).cuda() for k, v in sub.items()}
    proj = R.project(P, sc.sh_degree, frame)
    rng = np.random.default_rng(1)
    gs = [{k: v.astype(np.float32) for k, v in _rand_rec_grads(rng, n).items()} for _ in cams]
    rad = proj.radius.cpu().numpy().reshape(len(cams), n)
    # the oracle's gradient is zero for culled records; agree on visibility first
    vis = [oproj.project_np(sub, sc.sh_degree, c)["visible"] for c in cams]
    for v in range(len(cams)):
        assert np.array_equal(vis[v], rad[v] > 0)
    out = R.project_bwd(P, sc.sh_degree, frame, proj, _rec_grads_gpu(gs))
    torch.cuda.synchronize()
    want = opipe.project_vjp(sub, sc.sh_degree, cams, gs)
    for k in R.PARAM_KEYS:
        got = out[k].cpu().numpy()
        assert rel_l2(got, want[k]) < 1e-4, (k, rel_l2(got, want[k]))


def test_project_vjp_clamped_colour_and_fov_clamp():
    # a Gaussian far off to the side (J clamp active) and one with a clamped channel
    cam = synth.Camera(R=np.eye(3, dtype=np.float32), t=np.array([0, 0, 2], np.float32), fx=60.0, fy=60.0,
                       cx=32.0, cy=32.0, width=64, height=64)
    p = dict(means=np.array([[1.2, 0.0, 0.0], [0.05, 0.1, 0.3]], np.float32),
             log_scales=np.array([[-0.5, -0.8, -0.6], [-2.0, -2.2, -1.9]], np.float32),
             quats=np.array([[0.9, 0.1, 0.2, 0.3], [0.5, -0.5, 0.5, 0.5]], np.float32),
             opacity_logits=np.array([0.3, -0.2], np.float32),
             sh=np.array([[[0.2, -3.0, 0.5]], [[-4.0, 0.1, 0.9]]], np.float32))
    frame = R.Frame([cam])
    P = {k: torch.as_tensor(v).cuda() for k, v in p.items()}
    proj = R.project(P, 0, frame)
    assert (proj.radius.cpu().numpy() > 0).all()
    assert list(proj.clamped.cpu().numpy()) == [2, 1]
    rng = np.random.default_rng(3)
    g = {k: v.astype(np.float32) for k, v in _rand_rec_grads(rng, 2).items()}
    out = R.project_bwd(P, 0, frame, proj, _rec_grads_gpu([g]))
    want = opipe.project_vjp(p, 0, [cam], [g])
    for k in R.PARAM_KEYS:
        assert rel_l2(out[k].cpu().numpy(), want[k]) < 1e-4, k


@pytest.mark.parametrize("degree", [0, 1, 2])
@pytest.mark.parametrize("views", [1, 3])
@pytest.mark.parametrize("stored,shift", [(16, 0), (16, 1), (11, 0)])
@pytest.mark.parametrize("n", [1, 33, 1000])
def test_project_vjp_of_rows_wider_than_the_degree(n, stored, shift, views, degree):
    """SH rows that store more coefficients than the degree uses, on 16-byte boundaries or not
    (shift: one float off) and of widths that are no multiple of four: bit for bit the
    gradients of exact rows, and zeros beyond them. The exact rows against the oracle."""
    K = (degree + 1) ** 2
    sc = scene("orbit_small")
    cams = [synth.orbit_camera(4.0, 0.3 + 1.9 * v, 15.0, 200 - 40 * v, 150, 180.0) for v in range(views)]
    sub = {k: np.ascontiguousarray(v[:n]) for k, v in sc.params().items()}
    exact = dict(sub, sh=np.ascontiguousarray(sub["sh"][:, :K]))
    frame = R.Frame(cams)
    P = {k: torch.as_tensor(v).cuda() for k, v in exact.items()}
    proj = R.project(P, degree, frame)
    rng = np.random.default_rng(n + degree)
    gs = [{k: v.astype(np.float32) for k, v in _rand_rec_grads(rng, n).items()} for _ in cams]
    rec = _rec_grads_gpu(gs)
    want = R.project_bwd(P, degree, frame, proj, rec)
    oracle = opipe.project_vjp(exact, degree, cams, gs)
    for k in R.PARAM_KEYS:
        w = oracle[k]
        assert np.linalg.norm(want[k].cpu().numpy() - w) <= 1e-4 * np.linalg.norm(w) + 1e-30, k

    def placed(value):
        flat = torch.full((n * stored * 3 + 1,), value, device="cuda")
        return flat[shift:shift + n * stored * 3].view(n, stored, 3)

    wide = dict(P, sh=placed(7.0))
    wide["sh"][:, :K] = P["sh"]
    out = {k: torch.empty_like(P[k]) for k in R.PARAM_KEYS}
    out["sh"] = placed(5.0)
    R.project_bwd(wide, degree, frame, proj, rec, out=out)
    for k in R.PARAM_KEYS:
        got = out[k][:, :K] if k == "sh" else out[k]
        assert torch.equal(got, want[k]), k
    assert not out["sh"][:, K:].any()


@pytest.mark.parametrize("degree,stored", [(0, 1), (1, 4), (2, 9), (2, 16), (3, 16)])
@pytest.mark.parametrize("n", [1, 127, 3000])
def test_project_of_several_views_equals_each_view(n, degree, stored):
    """A frame of several views (of different sizes, some Gaussians behind or outside some of
    them) against frames of one view, bit for bit: both evaluate the same expressions."""
    sc = scene("orbit_small")
    sub = {k: np.ascontiguousarray(v[:n]) for k, v in sc.params().items()}
    sub["sh"] = np.ascontiguousarray(sub["sh"][:, :stored])
    P = {k: torch.as_tensor(v).cuda() for k, v in sub.items()}
    cams = [synth.orbit_camera(4.0 - v, 0.3 + 1.9 * v, 15.0, 200 - 40 * v, 150, 180.0) for v in range(4)]
    got = R.project(P, degree, R.Frame(cams))
    seen = 0
    for v, cam in enumerate(cams):
        want = R.project(P, degree, R.Frame([cam]))
        seen += int((want.radius > 0).sum())
        for k in ("mean2d", "conic_opacity", "rgb", "depth", "radius", "rect", "clamped"):
            assert torch.equal(getattr(got, k)[v * n:(v + 1) * n], getattr(want, k)), (v, k)
    assert n < 100 or n < seen < 4 * n


@pytest.mark.parametrize("degree,stored", [(0, 1), (1, 4), (2, 9), (3, 16)])
@pytest.mark.parametrize("more", [-1, 0, 129])
def test_project_of_several_views_around_the_line_between_its_kernels(degree, stored, more):
    """Counts on both sides of views_at_once's line, bit for bit the records of one-view frames."""
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    n = (256 if degree >= 2 else 1024) * sms + more
    g = torch.Generator("cuda").manual_seed(7)
    norm = lambda *s: torch.randn(*s, generator=g, device="cuda")   # noqa: E731
    P = dict(means=1.5 * norm(n, 3), log_scales=-4 + 0.7 * norm(n, 3), quats=norm(n, 4), opacity_logits=norm(n) - 2,
             sh=0.3 * norm(n, stored, 3))
    cams = [synth.orbit_camera(4.0 - v, 0.3 + 1.9 * v, 15.0, 200 - 40 * v, 150, 180.0) for v in range(3)]
    got = R.project(P, degree, R.Frame(cams))
    seen = 0
    for v, cam in enumerate(cams):
        want = R.project(P, degree, R.Frame([cam]))
        seen += int((want.radius > 0).sum())
        for k in ("mean2d", "conic_opacity", "rgb", "depth", "radius", "rect", "clamped"):
            assert torch.equal(getattr(got, k)[v * n:(v + 1) * n], getattr(want, k)), (v, k)
    assert 0.3 * n < seen < 2.9 * n


@pytest.mark.parametrize("stored,shift,degree", [(4, 1, 0), (9, 0, 0), (9, 0, 1), (10, 0, 2)])
@pytest.mark.parametrize("n", [1, 31, 1000])
def test_project_vjp_of_wide_rows_written_by_scalars(n, stored, shift, degree):
    """Gradient rows of 12 to 30 floats, several to a step of 32, that cannot be written as vectors."""
    test_project_vjp_of_rows_wider_than_the_degree(n, stored, shift, 1, degree)
