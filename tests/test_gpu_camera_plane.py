"""The camera-plane form of the two-parameter render (batches of more than 131 072 rays)
where it can go wrong: records of two Gaussians with odd counts, cameras with unequal
focal lengths and an off-centre principal point, means off the image, behind the camera
and in its plane, normals that cancel, every option that it has; against the FP64 oracle
with the tolerances of gpu_util, and against the world-frame form, which calls of one
view of the same batch take."""

import numpy as np
import pytest
import torch

import oracle
from paper_2308_14737_gb300 import fmb, synth

from gpu_util import (compare_forward, compare_grads, dev_scene, gpu_backward, gpu_forward, masked_upstream,
                      nnorm_batched, plane_view)

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2308_14737_gb300 import build

    build.build()
    oracle.build()
    fmb.load_library()


WORLD_RAYS = 131072


def _scene(K, seed=3, W=301, H=239, outside=True, rays=0):
    """One object of K Gaussians seen by two skewed cameras (143 878 rays, or ``rays`` random
    ones); with ``outside`` some means are off the image, behind the camera or in its plane."""
    rng = np.random.default_rng(seed)
    mu, ch, lam = synth.random_gaussians(rng, K)
    if outside and K >= 3:
        mu[1::9] = [6.0, -5.0, 1.0]
        mu[1::9] += rng.normal(0, 0.5, mu[1::9].shape).astype(np.float32)
        mu[2::9] = [14.0, 9.0, -9.0]  # behind the first camera, off its image
        mu[5::9] = [3.0, 1.0, -4.0]   # in its plane
    poses = [synth.look_at_pose((0.0, 0.0, -4.0)), synth.look_at_pose((2.5, 1.0, 2.5))]
    q = lambda x: float(np.float32(x))  # what the library sees
    views = [dict(W=W, H=H, fx=q(1.09 * W), fy=q(0.83 * W), cx=q(0.36 * W), cy=q(0.65 * H), object=0, pose=0,
                  flow_target=(1, -1)),
             dict(W=H, H=W, fx=q(1.21 * H), fy=q(2.2 * H), cx=q(0.46 * H), cy=q(0.61 * W), object=0, pose=1,
                  flow_target=(0, 1))]
    s = synth.make_scene([(mu, ch, lam)], views, poses)
    return synth.ray_batch(s, rays, seed) if rays else s


def _upstream(s, nf, normals):
    ref = oracle.render_scene(s, n_flow=nf)
    ups = masked_upstream(s, ref["alpha"], nf, nnorm_ref=nnorm_batched(s, ref["saved"]))
    if not normals:
        ups["g_normal"] = np.zeros_like(ups["g_normal"])
    return ref, ups


@pytest.mark.parametrize("K", [1, 3, 65, 256, 257])
@pytest.mark.parametrize("normals,pose", [(1, True), (0, True), (1, False), (0, False)])
def test_odd_counts_skewed_cameras_and_outside_means(K, normals, pose):
    s = _scene(K)
    assert s.n_pixels > WORLD_RAYS
    gpu, r, dev = gpu_forward(s, fmb.default_params(n_flow=2, want_normals=normals))
    ref, ups = _upstream(s, 2, normals)
    compare_forward(s, gpu, ref, 2, bool(normals))
    g = gpu_backward(r, dev, ups, want_pose=pose)
    refg = oracle.backward_scene(s, ups["g_depth"], ups["g_alpha"], ups["g_normal"] if normals else None,
                                 ups["g_flow"], n_flow=2)
    compare_grads(g, refg, keys=("means", "chol", "weights") + (("poses",) if pose else ()))


@pytest.mark.parametrize("K,normals,rays,opts", [
    (75, 1, 0, {}), (75, 0, 0, dict(deterministic=1)), (129, 1, 0, dict(use_persistent=1, deterministic=1)),
    (129, 1, 0, dict(fwd_ksplit=3)), (33, 0, 0, dict(fwd_ksplit=8, fwd_rays_per_thread=4)),
    (33, 1, 0, dict(fwd_rays_per_thread=1, bwd_gblocks=4)), (75, 1, 0, dict(bwd_threads=96, bwd_ray_tile=1024)),
    (75, 1, 0, dict(colors=1)), (41, 0, 0, dict(colors=1, deterministic=1)), (101, 1, 140001, {}),
    (40, 0, 140001, dict(bwd_threads=32, bwd_ray_tile=33))])
def test_both_forms_agree(K, normals, rays, opts):
    """The whole batch (camera plane) against its views one by one (world frame): planes to
    1e-5, the summed gradients to 3e-5 of the largest entry (each form is within about 1e-5
    of FP64)."""
    s = _scene(K, outside=False, rays=rays)
    assert s.n_pixels > WORLD_RAYS and all(synth.view_entries(v) <= WORLD_RAYS for v in s.views)
    nf, colors = 1, opts.get("colors", 0)
    params = fmb.default_params(n_flow=nf, want_normals=normals, **opts)
    _, ups = _upstream(s, nf, normals)
    T = lambda a: None if a is None else torch.as_tensor(np.ascontiguousarray(a).reshape(-1), dtype=torch.float32,
                                                          device="cuda")
    u = [T(ups[k]) for k in ("g_depth", "g_alpha", "g_normal", "g_flow")]
    x = dev_scene(s)
    col = torch.rand(K, 3, device="cuda") if colors else None
    gc = torch.randn(3 * s.n_pixels, device="cuda") * (u[0] != 0).float().mean() if colors else None
    r = fmb.Renderer(s.obj_offsets, s.views, len(s.poses), params)
    out = r.forward(*x, colors=col)
    grads = r.backward(*x, *u, colors=col, g_color=gc)
    total = None
    for v in s.views:
        n, o = synth.view_entries(v), v["pix_offset"]
        r1 = fmb.Renderer(s.obj_offsets, [dict(v, pix_offset=0)], len(s.poses), params)
        one = r1.forward(*x, colors=col)
        seen = one["alpha"] >= 1e-2
        d = (out["depth"][o:o + n] - one["depth"]).abs()[seen]
        assert d.max() <= 1e-5 * one["depth"][seen].max()
        assert (out["alpha"][o:o + n] - one["alpha"]).abs().max() <= 2e-6
        if normals:
            e = (out["normal"][3 * o:3 * (o + n)] - one["normal"]).view(3, n).abs().amax(0)
            assert (e * one["saved"][2 * n:].clamp(min=1e-3))[seen].max() <= 2e-5
        if colors:
            assert (out["color"][3 * o:3 * (o + n)] - one["color"]).view(3, n)[:, seen].abs().max() <= 2e-5
        cut = lambda t, w: None if t is None else t[w * o:w * (o + n)].contiguous()
        g = r1.backward(*x, cut(u[0], 1), cut(u[1], 1), cut(u[2], 3), cut(u[3], 2 * nf), colors=col, g_color=cut(gc, 3))
        total = {k: t.double() + (total[k] if total else 0) for k, t in g.items()}
    for k, t in total.items():
        assert (grads[k].double() - t).abs().max() <= 3e-5 * t.abs().max(), k


@pytest.mark.parametrize("K,normals,colors", [(1, 1, 0), (75, 0, 0), (300, 1, 0), (33, 0, 1)])
def test_gradient_slots_around_their_count(K, normals, colors):
    """Gradients summed through the slots (views of 1, 2, 3, 7, 8, 9 and 281 tiles of 256
    rays) against the deterministic mode's one slot per tile: the same
    terms in another order, to 3e-5 of the largest entry as above."""
    s = _scene(K, outside=False)
    base = dict(s.views[0])
    for n in (1, 2, 3, 7, 8, 9):
        s.views.append(dict(base, W=16, H=16 * n, fx=30.0, fy=28.0, cx=8.25, cy=8.0 * n, pix_offset=s.n_pixels))
    assert s.n_pixels > WORLD_RAYS
    x = dev_scene(s)
    col = torch.rand(K, 3, device="cuda") if colors else None
    torch.manual_seed(K)
    P = s.n_pixels
    got = []
    for det in (0, 1):
        r = fmb.Renderer(s.obj_offsets, s.views, len(s.poses), fmb.default_params(
            n_flow=1, want_normals=normals, colors=colors, deterministic=det, bwd_ray_tile=256))
        out = r.forward(*x, colors=col)
        if det == 0:
            on = (out["alpha"] >= 1e-2).float()
            u = [torch.randn(P, device="cuda") * on, torch.randn(P, device="cuda") * on,
                 torch.zeros(3 * P, device="cuda"), torch.zeros(2 * P, device="cuda")]
            gc = torch.zeros(3 * P, device="cuda") if colors else None
        got.append(r.backward(*x, *u, colors=col, g_color=gc))
    for k, t in got[1].items():
        assert (got[0][k].double() - t.double()).abs().max() <= 3e-5 * t.abs().max(), k


def test_normals_that_cancel():
    """Two equal Gaussians side by side: their normals oppose each other between them, so
    |N| passes through 0 there.  N carries at most 5e-6 (the weights' 1e-5, Sec. 7's
    beta1 on a residual good to 1e-6), so its direction is good to 1e-5 / |N|."""
    mu = np.array([[-0.3, 0.0, 0.0], [0.3, 0.0, 0.0], [0.05, 0.9, 0.2]], dtype=np.float32)
    ch = np.tile(np.array([3.0, 0, 3.0, 0, 0, 3.0], dtype=np.float32), (3, 1))
    view = dict(W=801, H=200, fx=32000.0, fy=31000.0, cx=400.375, cy=99.25, object=0, pose=0)
    s = synth.make_scene([(mu, ch, np.ones(3, np.float32))], [view], [synth.look_at_pose((0.0, 0.0, -4.0))])
    gpu, _, _ = gpu_forward(s, fmb.default_params(n_flow=0))
    ref = oracle.render_scene(s, n_flow=0)
    nn = plane_view(ref["saved"], s.views[0], 3)[2]
    assert np.any(nn < 0.03) and np.any((nn > 0.03) & (nn < 0.1))
    err = np.abs(plane_view(gpu["normal"], s.views[0], 3) - plane_view(ref["normal"], s.views[0], 3)).max(0)
    assert np.all(err <= 1e-5 / np.maximum(nn, 1e-5) + 1e-5)
    assert np.all(np.abs(plane_view(gpu["saved"], s.views[0], 3)[2] - nn) <= 1e-5)


def test_noalloc_limit_counts_gaussians_not_padding():
    """A batch within the fixed scratch by its Gaussians (64 bytes each) is taken although
    every view's odd count is padded by a record."""
    K, n = 163, 100
    s = synth.object_orbit(K=K, n_views=n, W=3, H=2)
    assert 256 + 64 * K * n <= 1 << 20 < 256 + 64 * (K + 1) * n
    params = fmb.default_params(n_flow=1)
    want, r, dev = gpu_forward(s, params)
    out = r.new_planes()
    fmb.fmb_render_forward_noalloc(params, s.obj_offsets, *dev, r.c_views, out["depth"], out["alpha"], out["normal"],
                                   out["flow"], out["saved"])
    assert fmb.fmb_read_noalloc_status() == 0
    for k in ("depth", "alpha", "normal", "flow"):
        np.testing.assert_allclose(out[k].cpu().numpy(), want[k], rtol=2e-5, atol=2e-5)
