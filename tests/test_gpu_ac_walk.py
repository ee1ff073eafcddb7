"""The thread-per-ray alpha-compositing forward (whole images with many rays) against the
warp-per-ray kernel, which a ray batch listing the same pixels takes.  Both evaluate the
same depths, so that orders and ties are the same; the sums differ in their order only:
100 terms of 32 bits, 1e-5 of the sum at most."""

import numpy as np
import pytest
import torch

from paper_2308_14737_gb300 import fmb, synth

from gpu_util import dev_scene

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2308_14737_gb300 import build

    build.build()
    fmb.load_library()


@pytest.mark.parametrize("K,views,W,H,opts", [
    (1, 1, 601, 333, {}), (3, 1, 601, 333, dict(want_normals=1)), (4, 3, 333, 257, {}), (5, 1, 1021, 201, {}),
    (40, 5, 401, 303, dict(want_normals=1, n_flow=2)), (64, 3, 333, 257, dict(colors=1)),
    (65, 10, 1, 20011, {}), (100, 16, 320, 240, dict(n_flow=1)), (128, 2, 401, 303, dict(want_normals=1, colors=1)),
    (129, 2, 401, 303, dict(use_persistent=1)), (256, 1, 601, 333, dict(want_normals=1, n_flow=1))])
@pytest.mark.parametrize("ties", [False, True])
def test_walk_agrees_with_warp_per_ray(K, views, W, H, opts, ties):
    rng = np.random.default_rng(K)
    mu, ch, lam = synth.random_gaussians(rng, K)
    if ties:  # exact duplicates: equal depths on every ray
        n = K // 3
        mu[K - n:], ch[K - n:], lam[K - n:] = mu[:n], ch[:n], lam[:n]
    poses = [synth.look_at_pose(p) for p in synth.sphere_positions(rng, views)]
    vs = [dict(W=W, H=H, fx=300.0, fy=280.0, cx=W / 2.0, cy=H / 2.0, object=0, pose=i,
               flow_target=((i + 1) % views, i - 1)) for i in range(views)]
    s = synth.make_scene([(mu, ch, lam)], vs, poses)
    assert s.n_pixels >= 640 * 2 * 152
    kw = dict(dict(want_normals=0, n_flow=0), variant=1, keep_order=1, **{k: v for k, v in opts.items()})
    params = fmb.default_params(**kw)
    x = dev_scene(s)
    col = torch.rand(K, 3, device="cuda") if opts.get("colors") else None
    r = fmb.Renderer(s.obj_offsets, s.views, len(s.poses), params)
    a = {k: t.clone() for k, t in r.forward(*x, colors=col).items() if t is not None}
    assert fmb.fmb_read_device_status(r.ws) == 0
    listed = [dict(v, rays=np.arange(W * H)) for v in s.views]
    rb = fmb.Renderer(s.obj_offsets, listed, len(s.poses), params)
    b = rb.forward(*x, colors=col)
    seen = b["alpha"] >= 1e-2
    for k, t in a.items():
        u = b[k]
        if k in ("alpha", "saved"):
            if k == "saved" and opts.get("want_normals"):  # |N| below
                t, u = (q.view(views, 3, -1)[:, :2].reshape(-1) for q in (t, u))
            assert (t - u).abs().max() <= 1e-5 * max(1.0, float(u.abs().max())), k
        elif k == "depth":
            assert ((t - u).abs() / u.abs())[seen].max() <= 1e-5
        else:  # camera-plane vectors and pixels: per view [channels][P]
            c = t.numel() // s.n_pixels
            e = (t - u).view(views, c, -1).abs().amax(1).reshape(-1)
            if k == "normal":
                e = e * b["saved"].view(views, 3, -1)[:, 2].reshape(-1)
            assert e[seen].max() <= (2e-5 if k != "flow" else 1e-3), k
    # the stored orders: the same gradients from either forward's
    g = [torch.randn(s.n_pixels, device="cuda") * seen, torch.randn(s.n_pixels, device="cuda") * seen]
    gn = torch.randn(3 * s.n_pixels, device="cuda") * 0 if opts.get("want_normals") else None
    nf = opts.get("n_flow", 0)
    gf = torch.zeros(2 * nf * s.n_pixels, device="cuda") if nf else None
    gc = torch.randn(3 * s.n_pixels, device="cuda") if col is not None else None
    ga = r.backward(*x, g[0], g[1], gn, gf, colors=col, g_color=gc)
    gb = rb.backward(*x, g[0], g[1], gn, gf, colors=col, g_color=gc)
    for k in ga:
        assert (ga[k] - gb[k]).abs().max() <= 3e-5 * gb[k].abs().max(), k


def _coarse(K, views, W, H, f, kind="cholesky"):
    rng = np.random.default_rng(K)
    obj = synth.random_gaussians(rng, K, kind)
    pos = synth.sphere_positions(rng, min(views, 64))
    vs = [dict(W=W, H=H, fx=float(f), fy=float(f), cx=W / 2.0, cy=H / 2.0, object=0, pose=i % len(pos),
               flow_target=(-1, -1)) for i in range(views)]
    return synth.make_scene([obj], vs, [synth.look_at_pose(p) for p in pos])


def _both(s, params):
    """The scene's renderer and one that lists the same pixels as ray batches."""
    listed = [dict(v, rays=np.arange(v["W"] * v["H"])) for v in s.views]
    return [fmb.Renderer(s.obj_offsets, vs, len(s.poses), params) for vs in (s.views, listed)]


@pytest.mark.parametrize("K,views,W,H,f", [(256, 1, 631, 473, 60), (256, 16, 320, 240, 64), (200, 2, 801, 503, 100),
                                           (128, 16, 128, 96, 16), (100, 64, 64, 48, 10), (9, 64, 64, 48, 1)])
def test_orders_that_change_by_more_than_the_window(K, views, W, H, f):
    """Wide fields of view, where the order changes by many places from one pixel to the
    next: the warp-per-ray kernel's planes (1e-5, as above; of the scene's unit where hits in
    front of and behind the camera cancel in the depth) and depth orders."""
    s = _coarse(K, views, W, H, f)
    assert s.n_pixels >= 640 * 2 * 152
    x = dev_scene(s)
    r, rb = _both(s, fmb.default_params(variant=1, want_normals=0, n_flow=0, keep_order=1))
    a = {k: t.clone() for k, t in r.forward(*x).items() if t is not None}
    b = rb.forward(*x)
    seen = b["alpha"] >= 1e-2
    assert (a["alpha"] - b["alpha"]).abs().max() <= 1e-5
    assert ((a["depth"] - b["depth"]).abs() / b["depth"].abs().clamp(min=1.0))[seen].max() <= 1e-5
    torch.manual_seed(0)
    g = [torch.randn(s.n_pixels, device="cuda") * seen, torch.randn(s.n_pixels, device="cuda") * seen]
    ga, gb = r.backward(*x, *g, None, None), rb.backward(*x, *g, None, None)
    for k in ga:
        assert (ga[k] - gb[k]).abs().max() <= 3e-5 * gb[k].abs().max(), k


@pytest.mark.parametrize("K,views,W,H,f", [(256, 1, 631, 473, 631), (256, 16, 128, 96, 128), (100, 250, 32, 32, 32),
                                           (256, 100, 64, 48, 64), (100, 800, 16, 16, 16), (40, 3200, 8, 8, 2)])
@pytest.mark.parametrize("kind", ["cholesky", "diag"])
def test_no_slower_than_warp_per_ray(K, views, W, H, f, kind):
    """Whatever the planner takes for whole images is not slower than the warp-per-ray
    kernel that ray batches take (with a quarter to spare for the clock)."""
    s = _coarse(K, views, W, H, f, kind)
    x = dev_scene(s)
    ms = []
    for r in _both(s, fmb.default_params(variant=1, want_normals=0, n_flow=0)):
        best = np.inf
        for _ in range(5):
            a, b = (torch.cuda.Event(enable_timing=True) for _ in range(2))
            a.record()
            r.forward(*x)
            b.record()
            b.synchronize()
            best = min(best, a.elapsed_time(b))
        ms.append(best)
    assert ms[0] <= 1.25 * ms[1], ms
