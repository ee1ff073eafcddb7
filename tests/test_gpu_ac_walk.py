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
