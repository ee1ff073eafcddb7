"""The kernels of large calls (more than 131 072 rays: camera-plane render and adjoint, the
alpha-compositing column walk) behind the entry points that the older tests call with
small scenes: no write outside any buffer, the workspace among them, the differentiable
render with its graph capture, and the adjoint of the stored depth orders with all
upstream gradients."""

import numpy as np
import pytest
import torch

import oracle
from paper_2308_14737_gb300 import fmb, synth

from gpu_util import compare_grads, dev_scene, masked_upstream, nnorm_batched
from test_gpu_guards import GUARD, SENTINEL, Arena

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


def _scene(Ks, sizes, seed=6):
    """One object per entry of Ks, seen by a view of each of the sizes."""
    rng = np.random.default_rng(seed)
    objs = [synth.random_gaussians(rng, K) for K in Ks]
    poses = [synth.look_at_pose(p) for p in synth.sphere_positions(rng, len(sizes))]
    q = lambda x: float(np.float32(x))
    views = [dict(W=W, H=H, fx=q(1.1 * max(W, H)), fy=q(0.9 * max(W, H)), cx=q(0.45 * W), cy=q(0.55 * H),
                  object=i % len(Ks), pose=i, flow_target=((i + 1) % len(sizes), -1)) for i, (W, H) in enumerate(sizes)]
    s = synth.make_scene(objs, views, poses)
    assert s.n_pixels > WORLD_RAYS
    return s


@pytest.mark.parametrize("Ks,sizes,opts", [
    ((1, 37, 259), [(301, 229), (1, 1), (255, 257), (7, 3)], {}),
    ((37, 2), [(511, 263), (3, 5)], dict(deterministic=1)),
    ((37, 260), [(301, 229), (255, 257)], dict(colors=1)),
    ((37, 131), [(301, 229), (255, 257)], dict(bwd_gblocks=2, fwd_ksplit=3)),
    ((37,), [(301, 229), (255, 257)], dict(use_persistent=1, want_normals=0, n_flow=2)),
    ((37, 200), [(631, 317), (17, 5)], dict(variant=1, keep_order=1)),
    ((63,), [(333, 601), (2, 1)], dict(variant=1, keep_order=1, want_normals=0, colors=1))])
def test_outputs_and_workspace_stay_inside_their_buffers(Ks, sizes, opts):
    s = _scene(Ks, sizes)
    params = fmb.default_params(**dict(dict(n_flow=1), **opts))
    nf, col = params.n_flow, bool(params.colors)
    G, P, NP = int(s.obj_offsets[-1]), s.n_pixels, len(s.poses)
    x = dev_scene(s)
    colors = torch.rand(G, 3, device="cuda") if col else None
    r = fmb.Renderer(s.obj_offsets, s.views, NP, params)
    # the workspace, of exactly the size asked for, between guards
    n = fmb.fmb_workspace_bytes(params, s.obj_offsets, r.c_views)
    raw = torch.full((n + 8 * GUARD,), 0xA5, dtype=torch.uint8, device="cuda")
    r.ws = raw[4 * GUARD:4 * GUARD + n]
    assert r.ws.data_ptr() % 256 == 0
    A = Arena()
    planes = dict(depth=A.take(P), alpha=A.take(P), normal=A.take(3 * P) if params.want_normals else None,
                  flow=A.take(2 * nf * P), saved=A.take(3 * P), color=A.take(3 * P) if col else None)
    grads = dict(means=A.take(3 * G).view(G, 3), chol=A.take(6 * G).view(G, 6), weights=A.take(G),
                 poses=A.take(12 * NP).view(NP, 12))
    if col:
        grads["colors"] = A.take(3 * G).view(G, 3)
    r.forward(*x, colors=colors, out=planes)
    on = (planes["alpha"] >= 1e-2).float()
    torch.manual_seed(0)
    r.backward(*x, torch.randn(P, device="cuda") * on, torch.randn(P, device="cuda"),
               torch.zeros(3 * P, device="cuda") if params.want_normals else None, torch.zeros(2 * nf * P, device="cuda"),
               colors=colors, g_color=torch.zeros(3 * P, device="cuda") if col else None, out=grads, planes=planes)
    assert fmb.fmb_read_device_status(r.ws) == 0
    assert A.intact() == []
    assert bool((raw[:4 * GUARD] == 0xA5).all()) and bool((raw[4 * GUARD + n:] == 0xA5).all())
    for k, t in list(planes.items()) + list(grads.items()):  # every entry was written
        if t is not None:
            assert not bool((t.reshape(-1).view(torch.int32) == SENTINEL).any()), k


@pytest.mark.parametrize("deterministic", [0, 1])
def test_differentiable_render_eager_and_captured(deterministic):
    """``render`` and its gradients against the oracle, and the same captured in a CUDA
    graph and replayed twice on other values (the slots start from 0 on every replay)."""
    s = _scene((41,), [(301, 229), (255, 257)])
    r = fmb.Renderer(s.obj_offsets, s.views, len(s.poses), fmb.default_params(n_flow=1, deterministic=deterministic))
    ref = oracle.render_scene(s, n_flow=1)
    ups = masked_upstream(s, ref["alpha"], 1, nnorm_ref=nnorm_batched(s, ref["saved"]))
    refg = oracle.backward_scene(s, ups["g_depth"], ups["g_alpha"], ups["g_normal"], ups["g_flow"], n_flow=1)
    u = [torch.as_tensor(ups[k].reshape(-1), dtype=torch.float32, device="cuda")
         for k in ("g_depth", "g_alpha", "g_normal", "g_flow")]
    leaves = [t.clone().requires_grad_() for t in dev_scene(s)]
    grads = lambda: torch.autograd.grad(fmb.render(r, *leaves), leaves, u)
    names = ("means", "chol", "weights", "poses")
    np64 = lambda g: {k: t.cpu().numpy().astype(np.float64) for k, t in zip(names, g)}
    compare_grads(np64(grads()), refg)
    side = torch.cuda.Stream()
    side.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(side):
        grads()
    torch.cuda.current_stream().wait_stream(side)
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        got = grads()
    with torch.no_grad():
        leaves[0].add_(1.0)
    graph.replay()
    with torch.no_grad():
        leaves[0].copy_(dev_scene(s)[0])
    graph.replay()
    torch.cuda.synchronize()
    compare_grads(np64(got), refg)


@pytest.mark.parametrize("K,normals,nf", [(40, 1, 2), (100, 1, 1), (129, 0, 2)])
def test_adjoint_of_stored_orders_with_all_upstreams(K, normals, nf):
    """Depth orders stored by the column walk, normal and flow upstreams among them: the
    gradients that the warp-per-ray forward's orders give (1e-4 of the largest entry, the
    library's bound; the normal's upstream where |N| >= 0.05)."""
    s = _scene((K,), [(401, 303), (333, 257)])
    x = dev_scene(s)
    params = fmb.default_params(variant=1, keep_order=1, want_normals=normals, n_flow=nf)
    listed = [dict(v, rays=np.arange(v["W"] * v["H"])) for v in s.views]
    got, u = [], None
    for vs in (s.views, listed):
        r = fmb.Renderer(s.obj_offsets, vs, len(s.poses), params)
        out = r.forward(*x)
        if u is None:
            torch.manual_seed(K)
            per = lambda c, w: torch.cat([(torch.randn(c, v["W"] * v["H"], device="cuda") *
                                           w[v["pix_offset"]:v["pix_offset"] + v["W"] * v["H"]]).reshape(-1)
                                          for v in s.views])
            on = (out["alpha"] >= 1e-2).float()
            nn = torch.cat([out["saved"][3 * v["pix_offset"]:][2 * v["W"] * v["H"]:3 * v["W"] * v["H"]] for v in s.views])
            u = [per(1, on), torch.randn(s.n_pixels, device="cuda"), per(3, on * (nn >= 0.05)) if normals else None,
                 0.01 * per(2 * nf, on)]
        got.append(r.backward(*x, *u))
    for k, t in got[1].items():
        assert float(t.abs().max()) > 0
        assert (got[0][k].double() - t.double()).abs().max() <= 1e-4 * t.abs().max(), k
