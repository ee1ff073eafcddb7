"""Timed cases of the renderer's public entry points, with their inputs, and the same results in 64 bits.

A case names one call pattern of a user's program ("kind") and its sizes:

* ``grad``         ``Renderer.forward`` then ``Renderer.backward`` (what a training step or a fit does);
* ``graph``        the differentiable ``render`` and its gradients, captured once in a CUDA graph and replayed;
* ``forward``      ``Renderer.forward`` alone (a viewer, an evaluation);
* ``points``       ``fmb_render_points``: points, screen-space normals (Eq. 16) and quality from a forward's planes
                   (the other normal's sign is undecided where one Gaussian alone is seen, so it is not asked for);
* ``attribution``  ``Renderer.attribution``, the per-Gaussian loss attribution of split / remove;
* ``step``         ``ReconstructionStep``: render, loss, adjoint and Adam in one captured graph.

Scenes, cameras and upstream gradients follow ``paper_2308_14737_gb300.synth``.  As the paper weights its
losses by the object mask, upstream gradients are zero where a ray misses the object (alpha < 1e-2).  The
normal's are weighted by how well its direction is defined: the blended normal must not cancel (weight |N|^2),
nor the ray pass through the centre of the Gaussian that it sees.  With alpha compositing, rays whose depth
order no 32-bit evaluation can decide have none.  The masks, the targets of the
reconstruction step and the planes that ``points`` and ``attribution`` read come from the plain torch
evaluation below, not from the library, so that inputs depend on the seed alone.
"""

import math

import numpy as np
import torch

from paper_2308_14737_gb300 import fmb, synth
from paper_2308_14737_gb300.step import ReconstructionStep

BETA1, BETA2 = 21.4, 3.14
DEV = "cuda"


def _case(name, kind, **kw):
    c = dict(name=name, kind=kind, scene="sphere", objects=1, views=1, width=64, height=64, K=40, variant=0, normals=1,
             n_flow=0, pose=0, colors=0, deterministic=0, keep_order=0, rays=0)
    c.update(kw)
    return c


def listed():
    return [
        # One 64x64 view of a 40-Gaussian object, differentiated: the smallest call, where latency and launches
        # count (a pose tracker or a small fit replays this as a graph).
        _case("view64_graph", "graph", scene="single", width=64, height=64, K=40, pose=1),
        # The paper's own fitting scale (40 Gaussians, images of about 250x130): a whole reconstruction iteration.
        _case("fit_step", "step", views=12, width=250, height=130, K=40, normals=0, n_flow=1),
        # A random ray minibatch across all frames, the stochastic form of the same fit.
        _case("minibatch_grad", "grad", views=100, width=640, height=480, K=256, normals=0, n_flow=2, rays=50000),
        # An orbit around one object, all four planes, gradients to the Gaussians and the camera poses.
        _case("orbit_grad", "grad", scene="orbit", views=16, width=320, height=240, K=100, n_flow=1, pose=1),
        # Many objects of uneven size in one call: uneven K, image sides from 64 to 512.
        _case("ragged_grad", "grad", scene="ragged", objects=24, views=4, K=400, width=512, height=512, pose=1),
        # A full reconstruction pass: 100 frames at 640x480, forward and backward flow, fixed cameras.
        _case("recon_grad", "grad", views=100, width=640, height=480, K=256, normals=0, n_flow=2),
        # A large scene of thousands of Gaussians, all planes, gradients to everything.
        _case("large_k_grad", "grad", scene="large_k", views=2, width=1024, height=768, K=4096, n_flow=1, pose=1),
        # A viewer's frame: one image of odd size, no gradients.
        _case("frame_forward", "forward", width=1023, height=767, K=333),
        # Appearance fit with per-Gaussian colours, bitwise reproducible gradients, odd sizes.
        _case("colour_grad", "grad", views=9, width=257, height=191, K=75, normals=0, colors=1, deterministic=1),
        # The alpha-compositing weights on the orbit, depth orders kept for the backward.
        _case("ac_orbit_grad", "grad", scene="orbit", views=16, width=320, height=240, K=100, variant=1, normals=0,
              n_flow=1, pose=1, keep_order=1),
        # An alpha-compositing frame without gradients, odd size.
        _case("ac_frame_forward", "forward", width=631, height=473, K=61, variant=1, normals=0),
        # Oriented points of an orbit for a surface reconstruction.
        _case("points_export", "points", scene="orbit", views=16, width=320, height=240, K=100),
    ]


def _log_int(rng, a, b):
    return int(round(math.exp(rng.uniform(math.log(a), math.log(b)))))


def draw(rng):
    kind = rng.choice(["grad", "grad", "grad", "grad", "graph", "forward", "points", "attribution", "step"])
    w = _log_int(rng, 33, 1100)
    h = max(17, int(w * rng.uniform(0.5, 1.0)))
    K = _log_int(rng, 20, 4096)
    variant = int(rng.random() < 0.25)
    c = dict(kind=kind, width=w, height=h, K=K, variant=variant, normals=int(not variant and rng.random() < 0.6))
    if kind == "step":
        c.update(variant=0, normals=0, n_flow=1, width=min(w, 320), height=min(h, 240))
    elif kind in ("grad", "graph", "forward"):
        c.update(n_flow=rng.choice([0, 1, 2]), pose=int(rng.random() < 0.5))
        if kind == "grad" and not c["variant"] and rng.random() < 0.2:
            c.update(colors=1)
        if kind == "grad" and rng.random() < 0.2:
            c.update(deterministic=1)
    else:
        c.update(normals=0, variant=0 if kind == "points" else variant)
    if c["variant"]:
        c.update(K=_log_int(rng, 20, 256), keep_order=int(kind == "grad" and rng.random() < 0.7))
    if kind in ("graph", "step"):
        c.update(K=min(c["K"], 400))
    # as many views as keep a pass below half of the largest listed one
    pairs = c["width"] * c["height"] * c["K"] * (8 if c["variant"] else 1)
    c["views"] = max(1, min(_log_int(rng, 1, 120), int(3.0e9 / pairs), 16 if kind == "graph" else 120))
    if kind == "grad" and not c["variant"] and not c.get("colors") and rng.random() < 0.25:
        c.update(views=max(20, c["views"]), width=640, height=480, K=min(c["K"], 600),
                 rays=_log_int(rng, 2000, 200000))
    c = _case("", **c)
    del c["name"]
    return c


# ------------------------------------------------------------------------------------------------- inputs
def _scene(c, seed):
    """The Gaussians, cameras and views of a case (numpy, float32)."""
    rng = np.random.default_rng(seed)
    K, n, W, H, nf = c["K"], c["views"], c["width"], c["height"], c["n_flow"]
    if c["scene"] == "single":
        s = synth.single_view(seed, K, W, H)
    elif c["scene"] == "orbit":
        s = synth.object_orbit(seed, K, n, W, H)
    elif c["scene"] == "ragged":
        # K from 20 up to c["K"]; sides 1, 1/2, 1/4 and 1/8 of the width; the same sizes whatever the seed
        sizes = np.random.default_rng(0)
        objs, views, poses = [], [], []
        for o in range(c["objects"]):
            side = W // int(sizes.choice((1, 2, 4, 8)))
            objs.append(synth.random_gaussians(rng, int(sizes.integers(20, K + 1)), "cholesky"))
            for p in synth.sphere_positions(rng, n):
                views.append(dict(W=side, H=side, fx=float(side), fy=float(side), cx=side / 2.0, cy=side / 2.0, object=o,
                                  pose=len(poses)))
                poses.append(synth.look_at_pose(p))
        s = synth.make_scene(objs, views, poses)
    elif c["scene"] == "large_k":
        s = synth.large_k(seed, K, n, W, H)
    else:
        obj = synth.random_gaussians(rng, K, "cholesky" if K <= 1024 else "diag")
        poses = [synth.look_at_pose(p) for p in synth.sphere_positions(rng, n)]
        views = [dict(W=W, H=H, fx=float(W), fy=float(W), cx=W / 2.0, cy=H / 2.0, object=0, pose=i,
                      flow_target=((i + 1 if i + 1 < n else -1) if nf > 0 else -1, i - 1 if nf > 1 else -1))
                 for i in range(n)]
        s = synth.make_scene([obj], views, poses)
    if c["kind"] == "step":  # a fit starts from faint Gaussians: no ray is saturated (log(1 - alpha) stays finite)
        s.weights *= np.float32(min(1.0, 10.0 / K))
    if c["rays"]:
        s = synth.ray_batch(s, c["rays"], seed)
    return s


def _params(c):
    return fmb.default_params(want_normals=c["normals"], n_flow=c["n_flow"], variant=c["variant"],
                              colors=c["colors"], deterministic=c["deterministic"], keep_order=c["keep_order"])


def _t(a, dtype=torch.float32):
    return torch.as_tensor(np.ascontiguousarray(a), device=DEV).to(dtype)


def _upstream(c, s, seed):
    """Upstream gradients of the planes, masked as described above."""
    g = torch.Generator(device=DEV)
    g.manual_seed(seed)
    P, nf = s.n_pixels, c["n_flow"]
    r = lambda n: torch.randn(n, generator=g, device=DEV)
    up = dict(depth=r(P), alpha=r(P), normal=r(3 * P) if c["normals"] else None,
              flow=0.01 * r(2 * nf * P) if nf else None, color=r(3 * P) if c["colors"] else None)
    pl = _planes(c, _as(s, torch.float32 if not c["variant"] else torch.float64), c["variant"], masks=True)
    for v in s.views:
        o, n = v["pix_offset"], synth.view_entries(v)
        m = pl["mask"][o:o + n].float()
        up["depth"][o:o + n] *= m
        if c["variant"]:
            up["alpha"][o:o + n] *= pl["decided"][o:o + n].float()
        if nf:
            up["flow"][2 * nf * o:2 * nf * (o + n)] *= m.repeat(2 * nf)
        if c["colors"]:
            up["color"][3 * o:3 * (o + n)] *= m.repeat(3)
        if c["normals"]:
            up["normal"][3 * o:3 * (o + n)] *= (m * pl["sure"][o:o + n].float()).repeat(3)
    return up


def _colors(s, seed):
    return np.random.default_rng(seed + 1).uniform(0.0, 1.0, (len(s.weights), 3)).astype(np.float32)


def _targets(c, seed):
    """Target planes of the reconstruction step: the same cameras, another object."""
    other = _as(_scene(c, seed + 1000003), torch.float32)
    other["poses"] = _t(_scene(c, seed).poses)
    pl = _planes(c, other, 0)
    return {k: pl[k].cpu().numpy() for k in ("depth", "alpha", "flow")}


def prepare(case, seed):
    c = case
    s = _scene(c, seed)
    if c["kind"] == "step":
        # silhouettes and flow of a video, no depth sensor
        st = ReconstructionStep(s, _targets(c, seed), params=_params(c), lr=1e-2, w_depth=0.0, device=DEV)
        st.capture(warmup=2)
        return dict(kind="step", step=st)
    r = fmb.Renderer(s.obj_offsets, s.views, len(s.poses), _params(c), device=DEV)
    st = dict(kind=c["kind"], r=r, x=(_t(s.means), _t(s.chol), _t(s.weights), _t(s.poses)), pose=bool(c["pose"]),
              colors=_t(_colors(s, seed)) if c["colors"] else None)
    if c["kind"] in ("points", "attribution"):  # the planes of a forward pass
        pl = _planes(c, _as(s, torch.float64), c["variant"], masks=True)
        r.depth.copy_(pl["depth"])
        r.saved.copy_(pl["saved"])
        if c["kind"] == "attribution":
            g = torch.Generator(device=DEV)
            g.manual_seed(seed)
            st["loss"] = torch.rand(s.n_pixels, generator=g, device=DEV) * pl["mask"]
        return st
    if c["kind"] == "forward":
        return st
    st["up"] = _upstream(c, s, seed)
    if c["kind"] == "graph":
        side = torch.cuda.Stream()
        side.wait_stream(torch.cuda.current_stream())
        with torch.cuda.stream(side):
            _differentiated(st)
        torch.cuda.current_stream().wait_stream(side)
        st["graph"] = torch.cuda.CUDAGraph()
        with torch.cuda.graph(st["graph"]):
            st["out"] = _differentiated(st)
    return st


def _differentiated(st):
    """The planes of ``fmb.render`` and the gradients of their product with the upstream planes."""
    x = [t.detach().requires_grad_(i < 3 or st["pose"]) for i, t in enumerate(st["x"])]
    planes = fmb.render(st["r"], *x)
    up = [st["up"][k] for k in ("depth", "alpha", "normal", "flow")]
    pairs = [(p, u) for p, u in zip(planes, up) if u is not None]
    wrt = [t for t in x if t.requires_grad]
    grads = torch.autograd.grad([p for p, _ in pairs], wrt, [u for _, u in pairs])
    return dict(planes=[p.detach() for p, _ in pairs], grads=list(grads))


def run(state):
    st = state
    if st["kind"] == "step":
        st["step"].replay()
        return dict(loss=st["step"].loss, grad=st["step"].grad, theta=st["step"].theta.detach())
    if st["kind"] == "graph":
        st["graph"].replay()
        return st["out"]
    r = st["r"]
    if st["kind"] == "points":
        new = lambda n: torch.empty(n, dtype=torch.float32, device=DEV)
        o = dict(points=new(3 * r.P), normal_screen=new(3 * r.P), quality=new(r.P))
        fmb.fmb_render_points(r.params, r.obj_offsets, *st["x"], r.c_views, r.depth, r.saved, o["points"], None,
                              o["normal_screen"], o["quality"], r.ws)
        return o
    if st["kind"] == "attribution":
        return r.attribution(*st["x"], st["loss"])
    out = r.forward(*st["x"], colors=st["colors"])
    planes = {k: out[k] for k in ("depth", "alpha", "normal", "flow", "color")}
    if st["kind"] == "forward":
        return dict(planes=planes)
    u = st["up"]
    g = r.backward(*st["x"], u["depth"], u["alpha"], u["normal"], u["flow"], want_pose=st["pose"], colors=st["colors"],
                   g_color=u["color"])
    return dict(planes=planes, grads=g)


def work(case):
    """Bytes: each input read once, each output written once.  Flops: the method's own operations per ray and
    Gaussian (docs/opcount.md without the compensation), an FMA as two."""
    c = case
    if c["scene"] == "ragged":
        s = _scene(c, 0)
        pairs, P, G, n = s.n_pairs, s.n_pixels, len(s.weights), len(s.poses)
    else:
        P = c["rays"] or c["views"] * c["width"] * c["height"]
        pairs, G, n = P * c["K"], c["K"], c["views"]
    fwd = (39 if c["normals"] else 26) + (3 if c["colors"] else 0)
    bwd = (90 if c["normals"] else 51) + (3 if c["pose"] else 0) + (6 if c["colors"] else 0)
    plane = 4 * (2 + 3 * c["normals"] + 2 * c["n_flow"] + 3 * c["colors"])
    scene = 4 * (G * (10 + 3 * c["colors"]) + 12 * n)
    if c["kind"] == "forward":
        return dict(bytes=scene + P * plane, flops=2.0 * pairs * fwd)
    if c["kind"] == "points":
        return dict(bytes=scene + P * 4 * (4 + 10), flops=2.0 * pairs * 45)
    if c["kind"] == "attribution":
        return dict(bytes=scene + P * 4 * 2 + 4 * G, flops=2.0 * pairs * 23)
    # the planes are written, the upstream planes read; gradients to every input
    return dict(bytes=2 * scene + 2 * P * plane, flops=2.0 * pairs * (fwd + bwd))


# ------------------------------------------------------------------------------- plain torch evaluation
def _as(s, dtype):
    return dict(means=_t(s.means, dtype), chol=_t(s.chol, dtype), weights=_t(s.weights, dtype), poses=_t(s.poses, dtype),
                views=s.views, offs=s.obj_offsets, P=s.n_pixels, dtype=dtype)


def _chunks(x, per):
    """(view, first entry, pixel indices) in pieces of about `per` ray-Gaussian pairs."""
    for v in x["views"]:
        n = synth.view_entries(v)
        K = int(x["offs"][v["object"] + 1] - x["offs"][v["object"]])
        pix = torch.arange(n, device=DEV) if v.get("rays") is None else _t(v["rays"], torch.int64)
        step = max(1, per // K)
        for a in range(0, n, step):
            yield v, a, pix[a:a + step]


def _rays(x, v, pix, normals, variant, colors=None, nf=0, masks=False):
    """One piece of one view: the planes at the given pixels, differentiable in the scene's tensors."""
    dt = x["dtype"]
    lo, hi = int(x["offs"][v["object"]]), int(x["offs"][v["object"] + 1])
    mu, ch, lam = x["means"][lo:hi], x["chol"][lo:hi], x["weights"][lo:hi]
    pose = x["poses"][v["pose"]]
    R, t0 = pose[:9].view(3, 3), pose[9:]
    px = (pix % v["W"]).to(dt) + 0.5
    py = torch.div(pix, v["W"], rounding_mode="floor").to(dt) + 0.5
    vc = torch.stack([(px - v["cx"]) / v["fx"], (py - v["cy"]) / v["fy"], torch.ones_like(px)], 1)
    vc = vc / vc.norm(dim=1, keepdim=True)
    vw = vc @ R  # world ray
    o = -(R.t() @ t0)
    m = mu - o
    l00, l10, l11, l20, l21, l22 = ch.unbind(1)
    v0, v1, v2 = (vw[:, i:i + 1] for i in range(3))
    a0, a1, a2 = l00 * v0 + l10 * v1 + l20 * v2, l11 * v1 + l21 * v2, l22 * v2
    b0 = l00 * m[:, 0] + l10 * m[:, 1] + l20 * m[:, 2]
    b1, b2 = l11 * m[:, 1] + l21 * m[:, 2], l22 * m[:, 2]
    t = (a0 * b0 + a1 * b1 + a2 * b2) / (a0 * a0 + a1 * a1 + a2 * a2)
    u0, u1, u2 = t * a0 - b0, t * a1 - b1, t * a2 - b2
    d = -0.5 * (u0 * u0 + u1 * u1 + u2 * u2) + torch.log(lam)
    delta = torch.exp(d)
    sd = delta.sum(1)
    out = dict(alpha=-torch.expm1(-sd), sd=sd)
    if variant:
        ts, idx = torch.sort(t, dim=1)
        ds = torch.gather(delta, 1, idx)
        w = torch.exp(-(torch.cumsum(ds, 1) - ds)) * -torch.expm1(-ds)
        W = w.sum(1, keepdim=True)
        out["first"] = W[:, 0]
        w = torch.zeros_like(w).scatter(1, idx, w / W)
        if masks:  # neighbours in depth too close for 32 bits, both of them seen
            wn = torch.gather(w, 1, idx)
            near = (ts[:, 1:] - ts[:, :-1]) < 4e-6 * ts[:, 1:].abs()
            seen = torch.minimum(ds[:, 1:], ds[:, :-1]) * torch.maximum(wn[:, 1:], wn[:, :-1]) > 1e-7
            out["decided"] = ~(near & seen).any(1)
    else:
        e = BETA1 * d - BETA2 * t
        lse = torch.logsumexp(e, 1)
        out["first"] = lse / math.log(2.0)
        w = torch.exp(e - lse[:, None])
    D = (w * t).sum(1)
    out["depth"], out["w"], out["t"] = D, w, t
    out["ray"], out["o"] = vw, o
    if normals:
        g0, g1, g2 = l00 * u0, l10 * u0 + l11 * u1, l20 * u0 + l21 * u1 + l22 * u2
        s = w / torch.sqrt(g0 * g0 + g1 * g1 + g2 * g2)
        N = torch.stack([(s * g0).sum(1), (s * g1).sum(1), (s * g2).sum(1)], 1)
        nl = N.norm(dim=1)
        if masks:
            q = u0 * u0 + u1 * u1 + u2 * u2
            out["sure"] = (nl * (w * (q / (q + 0.01))).sum(1)) ** 2
        out["normal"] = (N / nl[:, None]) @ R.t()
    if colors is not None:
        out["color"] = w @ colors[lo:hi]
    flows = []
    for j in range(nf):
        tg = v["flow_target"][j] if j < len(v["flow_target"]) else -1
        if tg < 0:
            flows.append(torch.zeros(len(pix), 2, dtype=dt, device=DEV))
            continue
        q = x["poses"][tg]
        X = (o + vw * D[:, None]) @ q[:9].view(3, 3).t() + q[9:]
        flows.append(torch.stack([v["fx"] * X[:, 0] / X[:, 2] + v["cx"] - px, v["fy"] * X[:, 1] / X[:, 2] + v["cy"] - py], 1))
    out["flow"] = flows
    return out


def _put(plane, v, a, n, parts, width):
    """Writes parts (width arrays of the piece) into a view's planar block."""
    P, off = synth.view_entries(v), width * v["pix_offset"]
    for k, x in enumerate(parts):
        plane[off + k * P + a:off + k * P + a + n] = x


@torch.no_grad()
def _planes(c, x, variant, masks=False, per=1 << 25):
    """The planes of a whole batch, laid out as the renderer does."""
    P, nf, dt = x["P"], c["n_flow"], x["dtype"]
    new = lambda n: torch.zeros(n, dtype=dt, device=DEV)
    out = dict(depth=new(P), alpha=new(P), saved=new(3 * P), mask=torch.zeros(P, dtype=torch.bool, device=DEV),
               sure=new(P), decided=torch.ones(P, dtype=torch.bool, device=DEV), normal=new(3 * P) if c["normals"] else None,
               flow=new(2 * nf * P) if nf else None)
    for v, a, pix in _chunks(x, per):
        q, n, o = _rays(x, v, pix, c["normals"], variant, nf=0 if masks else nf, masks=masks), len(pix), v["pix_offset"] + a
        out["depth"][o:o + n], out["alpha"][o:o + n] = q["depth"], q["alpha"]
        _put(out["saved"], v, a, n, [q["first"], q["sd"]], 3)
        out["mask"][o:o + n] = q["alpha"] >= 1e-2
        if c["normals"]:
            if masks:
                out["sure"][o:o + n] = q["sure"]
            _put(out["normal"], v, a, n, q["normal"].unbind(1), 3)
        if variant and masks:
            out["decided"][o:o + n] = q["decided"]
            out["mask"][o:o + n] &= q["decided"]
        if q["flow"]:
            _put(out["flow"], v, a, n, torch.cat(q["flow"], 1).unbind(1), 2 * nf)
    return out


def exact(case, seed):
    c = case
    s = _scene(c, seed)
    x = _as(s, torch.float64)
    if c["kind"] == "step":
        return _exact_step(c, s, x, seed)
    if c["kind"] == "points":
        return _exact_points(c, s, x)
    if c["kind"] == "attribution":
        g = torch.Generator(device=DEV)
        g.manual_seed(seed)
        loss = torch.rand(s.n_pixels, generator=g, device=DEV)
        out = torch.zeros(len(s.weights), dtype=torch.float64, device=DEV)
        mask = _planes(c, x, c["variant"], masks=True)["mask"]
        with torch.no_grad():
            for v, a, pix in _chunks(x, 1 << 24):
                q = _rays(x, v, pix, 0, c["variant"])
                o = v["pix_offset"] + a
                lo, hi = int(x["offs"][v["object"]]), int(x["offs"][v["object"] + 1])
                L = loss[o:o + len(pix)] * mask[o:o + len(pix)]
                out[lo:hi] += (L.double()[:, None] * q["w"]).sum(0)
        return out
    grad = c["kind"] in ("grad", "graph")
    if s.n_pairs > (9e9 if not grad else 7e9 if c["normals"] else 8e9):
        return None
    colors = _t(_colors(s, seed), torch.float64) if c["colors"] else None
    leaves = [x["means"], x["chol"], x["weights"]] + ([x["poses"]] if c["pose"] else []) + ([colors] if c["colors"] else [])
    up = _upstream(c, s, seed) if grad else None
    nf, P = c["n_flow"], s.n_pixels
    new = lambda n: torch.zeros(n, dtype=torch.float64, device=DEV)
    pl = dict(depth=new(P), alpha=new(P), normal=new(3 * P) if c["normals"] else None, flow=new(2 * nf * P) if nf else None,
              color=new(3 * P) if c["colors"] else None)
    for t in leaves:
        t.requires_grad_(grad)
    total = [torch.zeros_like(t) for t in leaves]
    for v, a, pix in _chunks(x, 1 << 24):
        with torch.set_grad_enabled(grad):
            q = _rays(x, v, pix, c["normals"], c["variant"], colors, nf)
            n, o, Pv = len(pix), v["pix_offset"] + a, synth.view_entries(v)
            cols = [("depth", q["depth"], o), ("alpha", q["alpha"], o)]
            if c["normals"]:
                cols += [("normal", q["normal"][:, k], 3 * v["pix_offset"] + k * Pv + a) for k in range(3)]
            if c["colors"]:
                cols += [("color", q["color"][:, k], 3 * v["pix_offset"] + k * Pv + a) for k in range(3)]
            for j in range(nf):
                cols += [("flow", q["flow"][j][:, k], 2 * nf * v["pix_offset"] + (2 * j + k) * Pv + a) for k in range(2)]
            if grad:
                scalar = sum((up[k][b:b + n].double() * y).sum() for k, y, b in cols)
        for k, y, b in cols:
            pl[k][b:b + n] = y.detach()
        if grad:
            for acc, g in zip(total, torch.autograd.grad(scalar, leaves)):
                acc += g
    if c["kind"] == "forward":
        return dict(planes=pl)
    if c["kind"] == "graph":
        return dict(planes=[pl[k] for k in ("depth", "alpha", "normal", "flow") if pl[k] is not None], grads=total)
    names = ["means", "chol", "weights"] + (["poses"] if c["pose"] else []) + (["colors"] if c["colors"] else [])
    return dict(planes=pl, grads=dict(zip(names, total)))


def _exact_points(c, s, x):
    """Points and normals from the 32-bit depth plane that the call reads."""
    P = s.n_pixels
    pl = _planes(c, x, c["variant"])
    depth = pl["depth"].float().double()
    out = {k: torch.zeros(3 * P, dtype=torch.float64, device=DEV) for k in ("points", "normal_screen")}
    out["quality"] = torch.zeros(P, dtype=torch.float64, device=DEV)

    def facing(n, v):
        n = n / n.norm(dim=1, keepdim=True)
        return torch.where((n * v).sum(1, keepdim=True) > 0, -n, n)

    with torch.no_grad():
        for v, a, pix in _chunks(x, 1 << 24):
            q, n, o = _rays(x, v, pix, 0, c["variant"]), len(pix), v["pix_offset"] + a
            _put(out["points"], v, a, n, (q["o"] + q["ray"] * depth[o:o + n, None]).unbind(1), 3)
            out["quality"][o:o + n] = q["w"].max(1).values
    for v in s.views:
        W, H, off = v["W"], v["H"], v["pix_offset"]
        R, t0 = x["poses"][v["pose"]][:9].view(3, 3), x["poses"][v["pose"]][9:]
        yy, xx = torch.meshgrid(torch.arange(H, device=DEV), torch.arange(W, device=DEV), indexing="ij")
        xx, yy = xx.double() + 0.5, yy.double() + 0.5
        d = torch.stack([(xx - v["cx"]) / v["fx"], (yy - v["cy"]) / v["fy"], torch.ones_like(xx)], -1)
        ray = (d / d.norm(dim=-1, keepdim=True)) @ R
        p = -(R.t() @ t0) + ray * depth[off:off + W * H].view(H, W, 1)
        px = torch.cat([p[:, 1:], p[:, -2:-1]], 1)
        py = torch.cat([p[1:], p[-2:-1]], 0)
        nrm = facing(torch.linalg.cross(p - px, p - py, dim=-1).reshape(-1, 3), ray.reshape(-1, 3))
        _put(out["normal_screen"], v, 0, W * H, nrm.unbind(1), 3)
    return out


def _exact_step(c, s, x, seed):
    """Three Adam iterations (the two warm-up steps of the capture, then the pass)."""
    if 3 * s.n_pairs > 4e9:
        return None
    tg = {k: _t(v, torch.float64) for k, v in _targets(c, seed).items()}
    G, P, nf = len(s.weights), s.n_pixels, c["n_flow"]
    theta = torch.cat([x["means"].reshape(-1), x["chol"].reshape(-1), x["weights"]])
    m, vv = torch.zeros_like(theta), torch.zeros_like(theta)
    for step in range(1, 4):
        th = theta.clone().requires_grad_(True)
        grad, loss = torch.zeros_like(theta), 0.0
        for v, a, pix in _chunks(x, 1 << 24):
            y = dict(x, means=th[:3 * G].view(G, 3), chol=th[3 * G:9 * G].view(G, 6), weights=th[9 * G:])
            q, n, o, Pv = _rays(y, v, pix, 0, 0, nf=nf), len(pix), v["pix_offset"] + a, synth.view_entries(v)
            ta, al = tg["alpha"][o:o + n], q["alpha"].clamp(1e-6, 1.0 - 1e-6)
            part = -(ta * torch.log(al) + (1.0 - ta) * torch.log1p(-al)).sum()
            for j in range(nf):
                for k in range(2):
                    b = 2 * nf * v["pix_offset"] + (2 * j + k) * Pv + a
                    f = (q["flow"][j][:, k] - tg["flow"][b:b + n]) * (2.0 / min(v["W"], v["H"]))
                    part = part + (ta * f * f).sum()
            grad += torch.autograd.grad(part / P, th)[0]
            loss += float(part.detach()) / P
        g = torch.cat([grad[:9 * G], grad[9 * G:] * theta[9 * G:]])  # the weights move in log space
        m = 0.9 * m + 0.1 * g
        vv = 0.999 * vv + 0.001 * g * g
        up = 1e-2 * (m / (1 - 0.9 ** step)) / ((vv / (1 - 0.999 ** step)).sqrt() + 1e-8)
        theta = torch.cat([theta[:9 * G] - up[:9 * G], theta[9 * G:] * torch.exp(-up[9 * G:])])
    return dict(loss=torch.tensor(loss, dtype=torch.float64), grad=grad, theta=theta)
