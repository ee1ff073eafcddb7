"""The camera-plane form of the two-parameter render at the edges of what the library
accepts: launch sizes, parameters and data that the scenes of test_gpu_camera_plane.py do
not have."""

import numpy as np
import pytest
import torch

import oracle
from paper_2308_14737_gb300 import fmb, synth

from gpu_util import (compare_forward, compare_grads, dev_scene, gpu_backward, gpu_forward, masked_upstream,
                      nnorm_batched, plane_view)

pytestmark = pytest.mark.gpu

WORLD_RAYS = 131072


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2308_14737_gb300 import build

    build.build()
    oracle.build()
    fmb.load_library()


def _two_views(mu, ch, lam, W=301, H=239):
    q = lambda x: float(np.float32(x))  # what the library sees
    poses = [synth.look_at_pose((0.0, 0.0, -4.0)), synth.look_at_pose((2.5, 1.0, 2.5))]
    views = [dict(W=W, H=H, fx=q(1.1 * W), fy=q(0.9 * W), cx=q(0.4 * W), cy=q(0.6 * H), object=0, pose=i,
                  flow_target=(1 - i, i)) for i in range(2)]
    s = synth.make_scene([(mu, ch, lam)], views, poses)
    assert s.n_pixels > WORLD_RAYS
    return s


@pytest.mark.parametrize("normals,colors,tile", [(1, 0, 430), (0, 0, 753), (0, 1, 502)])
def test_ray_tiles_whose_shared_memory_ends_at_48_kb(normals, colors, tile):
    """Dynamic shared memory of 48 160 to 48 192 bytes, which only the static part carries
    past 48 KB: the gradients of the default tile, whose sums have another order (3e-5)."""
    K = 40
    rng = np.random.default_rng(2)
    s = _two_views(*synth.random_gaussians(rng, K))
    x = dev_scene(s)
    P = s.n_pixels
    T = lambda a: torch.as_tensor(a.reshape(-1), device="cuda")
    col = torch.rand(K, 3, device="cuda") if colors else None
    got, ups = [], None
    for t in (0, tile):
        params = fmb.default_params(n_flow=2, want_normals=normals, colors=colors, bwd_ray_tile=t)
        r = fmb.Renderer(s.obj_offsets, s.views, len(s.poses), params)
        out = r.forward(*x, colors=col)
        if ups is None:
            on = (out["alpha"] >= 1e-2).cpu().numpy()
            gd, ga, gn, gf = synth.upstream_grads(rng, P, 2)
            ups = [T(gd * on), T(ga), torch.zeros(3 * P, device="cuda"), T(gf * on)]
        got.append(r.backward(*x, *ups, colors=col, g_color=T(gn * on) if colors else None))
    for k, t in got[0].items():
        assert (got[1][k].double() - t.double()).abs().max() <= 3e-5 * t.abs().max(), k


def _mild(K, seed):
    """Gaussians of 0.5 to 1 radius: whitened distances stay below about 10, so that 32-bit
    exponents are good to 1e-5 for any sign of beta1."""
    rng = np.random.default_rng(seed)
    mu = rng.uniform(-1, 1, (K, 3))
    d, o = rng.uniform(1.0, 2.0, (K, 3)), rng.normal(0, 0.3, (K, 3))
    ch = np.stack([d[:, 0], o[:, 0], d[:, 1], o[:, 1], o[:, 2], d[:, 2]], 1)
    return mu.astype(np.float32), ch.astype(np.float32), rng.uniform(0.5, 1.5, K).astype(np.float32)


@pytest.mark.parametrize("beta1", [0.0, -0.5, 0.3])
@pytest.mark.parametrize("K,opts", [(1, {}), (3, {}), (65, {}), (65, dict(fwd_ksplit=3)), (5, dict(fwd_rays_per_thread=1)),
                                    (257, dict(want_normals=0, fwd_rays_per_thread=4)), (64, {})])
def test_beta1_of_any_sign(beta1, K, opts):
    """beta1 may be any finite number: planes and gradients against the FP64 oracle."""
    s = _two_views(*_mild(K, K))
    params = fmb.default_params(n_flow=1, **opts)
    params.beta1 = beta1
    b1 = float(params.beta1)
    normals = bool(params.want_normals)
    gpu, r, dev = gpu_forward(s, params)
    ref = oracle.render_scene(s, n_flow=1, beta1=b1)
    compare_forward(s, gpu, ref, 1, normals)
    ups = masked_upstream(s, ref["alpha"], 1, nnorm_ref=nnorm_batched(s, ref["saved"]))
    if not normals:
        ups["g_normal"] = np.zeros_like(ups["g_normal"])
    g = gpu_backward(r, dev, ups)
    refg = oracle.backward_scene(s, ups["g_depth"], ups["g_alpha"], ups["g_normal"] if normals else None, ups["g_flow"],
                                 n_flow=1, beta1=b1)
    compare_grads(g, refg)


@pytest.mark.parametrize("zero", [(0,), (1,), (0, 1), (0, 1, 2, 3), (21, 22, 42, 43, 64)])
@pytest.mark.parametrize("opts", [{}, dict(fwd_ksplit=3), dict(want_normals=0)])
def test_weights_of_zero(zero, opts):
    """A Gaussian whose weight underflowed to 0 leaves the planes and the others' gradients
    what they are without it, wherever it stands (tolerances of two orders of summation)."""
    K = 65
    mu, ch, lam = synth.random_gaussians(np.random.default_rng(9), K)
    mu[32:40] = mu[24:32] + np.float32([0.0, 0.0, 0.3])  # normals that oppose each other
    keep = np.setdiff1d(np.arange(K), zero)
    lam0 = lam.copy()
    lam0[list(zero)] = 0.0
    params = fmb.default_params(n_flow=1, **opts)
    got, ups = [], None
    for s in (_two_views(mu[keep], ch[keep], lam[keep]), _two_views(mu, ch, lam0)):
        x = dev_scene(s)
        r = fmb.Renderer(s.obj_offsets, s.views, len(s.poses), params)
        out = {k: t.clone() for k, t in r.forward(*x).items() if t is not None}
        on = out["alpha"] >= 1e-2
        if ups is None:
            torch.manual_seed(1)
            ups = [torch.randn(n * s.n_pixels, device="cuda") for n in (1, 1, 3, 2)]
            ups = [ups[0] * on, ups[1], ups[2] * 0, 0.01 * ups[3] * on.view(2, 1, -1).expand(2, 2, -1).reshape(-1)]
        got.append((out, r.backward(*x, *ups), on))
    (a, ga, on), (b, gb, _) = got
    assert ((a["depth"] - b["depth"]).abs() / a["depth"])[on].max() <= 1e-5
    assert (a["alpha"] - b["alpha"]).abs().max() <= 2e-6
    if params.want_normals:
        nn = a["saved"].view(2, 3, -1)[:, 2]
        e = (a["normal"] - b["normal"]).view(2, 3, -1).abs().amax(1) * nn.clamp(min=1e-3)
        assert e.reshape(-1)[on].max() <= 2e-5
    assert torch.isfinite(b["normal"]).all() if params.want_normals else True
    idx = torch.as_tensor(keep, device="cuda")
    for k in ("means", "chol", "weights"):
        t = ga[k]
        assert (gb[k][idx].double() - t.double()).abs().max() <= 3e-5 * t.abs().max(), k


def test_flow_of_points_in_the_targets_camera_plane():
    """One flat Gaussian facing the camera, seen at depth 4 on every ray, and a target camera
    whose plane holds it: the flow is infinite, with the sign of the point's offset."""
    W, H = 401, 331
    mu, ch = np.array([[0.0, 0.0, 4.0]], np.float32), np.array([[1e-3, 0, 1e-3, 0, 0, 100.0]], np.float32)
    pose = np.concatenate([np.eye(3).reshape(-1), [0, 0, 0]])
    target = np.concatenate([np.eye(3).reshape(-1), [0, 0, -4.0]])
    view = dict(W=W, H=H, fx=300.0, fy=300.0, cx=200.25, cy=165.25, object=0, pose=0, flow_target=(1, -1))
    s = synth.make_scene([(mu, ch, np.ones(1, np.float32))], [view], [pose, target])
    assert s.n_pixels > WORLD_RAYS
    gpu, _, _ = gpu_forward(s, fmb.default_params(n_flow=1, want_normals=0))
    f = gpu["flow"].reshape(2, H, W)
    x, y = np.arange(W) + 0.5 - 200.25, np.arange(H) + 0.5 - 165.25
    np.testing.assert_array_equal(f[0], np.broadcast_to(np.copysign(np.inf, x), (H, W)))
    np.testing.assert_array_equal(f[1], np.broadcast_to(np.copysign(np.inf, y)[:, None], (H, W)))


def _thin(K, ratio, kind, seed):
    """Randomly turned discs (one short axis) or needles (two) of radius 0.4."""
    rng = np.random.default_rng(seed)
    mu = rng.uniform(-1, 1, (K, 3)) if K > 1 else rng.uniform(-0.2, 0.2, (K, 3))
    ch = np.zeros((K, 6))
    for k in range(K):
        q, _ = np.linalg.qr(rng.standard_normal((3, 3)))
        inv = np.array([1, 1, ratio] if kind == "disc" else [1, ratio, ratio]) / 0.4
        L = np.linalg.cholesky((q * inv ** 2) @ q.T)
        ch[k] = L[np.tril_indices(3)]
    return mu.astype(np.float32), ch.astype(np.float32), rng.uniform(0.5, 1.5, K).astype(np.float32)


@pytest.mark.parametrize("K,seed", [(1, 0), (1, 1), (1, 2), (24, 0), (25, 1)])
@pytest.mark.parametrize("ratio", [4, 6, 30, 100, 300])
def test_normals_of_thin_discs(K, seed, ratio):
    """The normal's error does not grow with the axis ratio: a pair's normal carries about
    eight roundings (5e-7), the blend its weights' 1e-6; 2e-6 rms over the rays that see
    the object, weighted by |N|."""
    s = _two_views(*_thin(K, ratio, "disc", seed))
    gpu, _, _ = gpu_forward(s, fmb.default_params(n_flow=0))
    ref = oracle.render_scene(s, n_flow=0)
    for v in s.views:
        nn = plane_view(ref["saved"], v, 3)[2]
        e = np.abs(plane_view(gpu["normal"], v, 3) - plane_view(ref["normal"], v, 3)).max(0) * nn
        e = e[ref["alpha"][v["pix_offset"]:][:len(e)] >= 1e-2]
        assert len(e) > 100 and np.sqrt(np.mean(e ** 2)) <= 2e-6


@pytest.mark.parametrize("kind,ratio", [("disc", 30), ("disc", 100), ("disc", 300), ("needle", 30)])
@pytest.mark.parametrize("K,seed", [(1, 0), (1, 1), (24, 0), (25, 1)])
def test_gradients_of_thin_gaussians(kind, ratio, K, seed):
    """With an upstream gradient of alpha alone the pairs' terms are well conditioned, so
    what the axis ratio costs shows in L's and the poses' gradients: 1e-5 of the largest
    entry, a tenth of the library's bound (sums of 32-bit terms carry about 1e-6)."""
    s = _two_views(*_thin(K, ratio, kind, seed))
    _, r, dev = gpu_forward(s, fmb.default_params(n_flow=1))
    ga = np.random.default_rng(seed).standard_normal(s.n_pixels).astype(np.float32)
    z = np.zeros(s.n_pixels, np.float32)
    ups = dict(g_depth=z, g_alpha=ga, g_normal=np.tile(z, 3), g_flow=np.tile(z, 2))
    g = gpu_backward(r, dev, ups)
    compare_grads(g, oracle.backward_scene(s, *(ups[k] for k in ("g_depth", "g_alpha", "g_normal", "g_flow")), n_flow=1),
                  rel=1e-5)


def _many_cancelling(zoom, W=401, H=331, K=2048):
    mu, ch, lam = synth.random_gaussians(np.random.default_rng(0), K, "diag")
    q = lambda x: float(np.float32(x))
    view = dict(W=W, H=H, fx=q(zoom * W), fy=q(zoom * W), cx=W / 2.0, cy=H / 2.0, object=0, pose=0, flow_target=(-1, -1))
    return synth.make_scene([(mu, ch, lam)], [view], [synth.look_at_pose((0.0, 0.0, -4.0))])


@pytest.mark.parametrize("rpt", [0, 4])
def test_scenes_whose_normals_all_nearly_cancel(rpt):
    """With beta1 = 0.1 and a narrow field of view |N| is below 0.06 on most rays.  N carries
    1e-6 per term's weight and direction, so err |N| stays below 5e-6, and the render takes
    at most three times as long as without normals (1.5 times the operations; seven times
    as long if every ray is summed again)."""
    s = _many_cancelling(8.0)
    assert s.n_pixels > WORLD_RAYS
    ms = {}
    for normals in (1, 0):
        params = fmb.default_params(n_flow=0, want_normals=normals, fwd_rays_per_thread=rpt)
        params.beta1, params.beta2 = 0.1, 0.3
        gpu, r, dev = gpu_forward(s, params)
        best = np.inf
        for _ in range(5):
            a, b = (torch.cuda.Event(enable_timing=True) for _ in range(2))
            a.record()
            r.forward(*dev)
            b.record()
            b.synchronize()
            best = min(best, a.elapsed_time(b))
        ms[normals] = best
        if normals:
            b1, b2 = float(params.beta1), float(params.beta2)
            pix = np.arange(0, s.n_pixels, 7)
            v = s.views[0]
            ref = oracle.render_view(s.means, s.chol, s.weights, s.poses[0], None,
                                     (v["W"], v["H"], v["fx"], v["fy"], v["cx"], v["cy"]), pixels=pix, beta1=b1, beta2=b2)
            nn = ref["saved"][:, 2]
            assert np.mean(nn < 0.06) > 0.5
            e = np.abs(plane_view(gpu["normal"], v, 3)[:, pix].T - ref["normal"]).max(1) * nn
            assert np.all(e <= 5e-6), e.max()
    assert ms[1] <= 3.0 * ms[0], ms


def _many_objects(n_obj, K, n_views, side, shown):
    """n_views square views, view i of object i mod shown of n_obj equal ones."""
    rng = np.random.default_rng(4)
    obj = synth.random_gaussians(rng, K)
    views = [dict(W=side, H=side, fx=float(side), fy=float(side), cx=side / 2.0, cy=side / 2.0, object=(7 * i) % shown,
                  pose=i, flow_target=((i + 1) % n_views, i - 1)) for i in range(n_views)]
    return synth.make_scene([obj] * n_obj, views, [synth.look_at_pose(p) for p in synth.sphere_positions(rng, n_views)])


@pytest.mark.parametrize("n_obj,K,n_views,side,shown,colors", [
    (5, 37, 11, 129, 3, 0), (40, 21, 70, 50, 33, 0), (300, 9, 300, 29, 299, 1), (3, 515, 5, 201, 2, 0)])
def test_slots_of_several_objects(n_obj, K, n_views, side, shown, colors):
    """Gradients of several objects (one to five launches' views, objects that no view
    shows) through the slots against the deterministic mode: the same terms in another
    order, 3e-5 of the largest entry."""
    s = _many_objects(n_obj, K, n_views, side, shown)
    assert s.n_pixels > WORLD_RAYS
    x = dev_scene(s)
    torch.manual_seed(n_obj)
    P = s.n_pixels
    col = torch.rand(n_obj * K, 3, device="cuda") if colors else None
    got, ups = [], None
    for det in (0, 1):
        r = fmb.Renderer(s.obj_offsets, s.views, len(s.poses), fmb.default_params(n_flow=2, colors=colors, deterministic=det))
        out = r.forward(*x, colors=col)
        if ups is None:
            on = out["alpha"] >= 1e-2
            planes = lambda n: torch.cat([torch.randn(n, side * side, device="cuda") *
                                          on[i * side * side:(i + 1) * side * side] for i in range(n_views)]).reshape(-1)
            nn = out["saved"].view(n_views, 3, -1)[:, 2:].expand(n_views, 3, -1).reshape(-1)
            ups = [planes(1), torch.randn(P, device="cuda"), planes(3) * (nn >= 0.05), 0.01 * planes(4)]
            gc = planes(3) if colors else None
        got.append(r.backward(*x, *ups, colors=col, g_color=gc))
    for k, t in got[1].items():
        assert (got[0][k].double() - t.double()).abs().max() <= 3e-5 * t.abs().max(), k
    for k in ("means", "chol", "weights"):
        assert not got[0][k].view(n_obj, -1)[shown:].any()


@pytest.mark.parametrize("n_obj,K,n_views,side,shown", [(256, 1024, 256, 64, 256), (4000, 1000, 64, 112, 64)])
def test_the_adjoint_of_many_objects_follows_what_is_rendered(n_obj, K, n_views, side, shown):
    """The time of the adjoint does not depend on how many objects the rays are spread
    over: twice one object's time at most, plus 1 ms for clearing the other gradients."""
    ms = []
    for obj, sh in ((n_obj, shown), (1, 1)):
        s = _many_objects(obj, K, n_views, side, sh)
        x = dev_scene(s)
        r = fmb.Renderer(s.obj_offsets, s.views, len(s.poses), fmb.default_params(n_flow=0, want_normals=0))
        on = (r.forward(*x)["alpha"] >= 1e-2).float()
        best = np.inf
        for _ in range(4):
            a, b = (torch.cuda.Event(enable_timing=True) for _ in range(2))
            a.record()
            r.backward(*x, on, on, None, None)
            b.record()
            b.synchronize()
            best = min(best, a.elapsed_time(b))
        ms.append(best)
    assert ms[0] <= 2.0 * ms[1] + 1.0, ms


@pytest.mark.parametrize("n_views,side,rays,K,normals", [(100, 200, 150000, 256, 0), (200, 32, 0, 256, 0),
                                                         (1, 448, 0, 160, 1), (16, 277, 0, 100, 1)])
def test_default_ray_tile_suits_the_call(n_views, side, rays, K, normals):
    """The planner's ray tile is not slower than three or four rays per thread asked for,
    whichever is better (with an eighth to spare for the clock): long tiles leave SMs idle
    in calls of a few hundred thousand rays."""
    s = _many_objects(1, K, n_views, side, 1)
    if rays:
        s = synth.ray_batch(s, rays, 0)
    assert s.n_pixels > WORLD_RAYS
    x = dev_scene(s)
    P, ms = s.n_pixels, {}
    for tile in (0, 384, 512):
        params = fmb.default_params(n_flow=0, want_normals=normals, bwd_threads=128, bwd_ray_tile=tile)
        r = fmb.Renderer(s.obj_offsets, s.views, len(s.poses), params)
        up = (r.forward(*x)["alpha"] >= 1e-2).float()
        gn = torch.zeros(3 * P, device="cuda") if normals else None
        best = np.inf
        for _ in range(4):
            a, b = (torch.cuda.Event(enable_timing=True) for _ in range(2))
            a.record()
            for _ in range(20):
                r.backward(*x, up, up, gn, None, want_pose=False)
            b.record()
            b.synchronize()
            best = min(best, a.elapsed_time(b))
        ms[tile] = best
    assert ms[0] <= 1.125 * min(ms[384], ms[512]), ms
