"""The adjoint kernels launched as clusters of two CTAs (every view in two Gaussian blocks)
write ray records into their peer's shared memory.  A peer's shared memory may only be
accessed once the peer runs: each kernel arrives at the cluster's barrier when it starts
and waits there before its first such store."""

import os
import re

import numpy as np
import pytest
import torch

import oracle
from paper_2308_14737_gb300 import fmb, synth

from gpu_util import compare_grads, gpu_backward, gpu_forward, masked_upstream, nnorm_batched

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2308_14737_gb300", "csrc")


@pytest.mark.parametrize("name", ["fmb_backward.cu", "fmb_world_bwd.cu"])
def test_remote_stores_wait_for_the_peers_start(name):
    src = re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, name)).read())
    body = src[src.index("__global__"):]
    arrive, wait, store = (body.find(f) for f in ("cluster_arrive()", "cluster_wait()", "st_cluster_f4("))
    assert 0 < arrive < wait < store
    # by every thread: the wait stands in front of the loop over the rays, not in it
    assert wait < body.index("for (int r = r_lo + tid;") < store
    # and before the work loop's first barrier of its own
    assert store < body.index("cluster_sync()")


@pytest.mark.gpu
@pytest.mark.parametrize("W,H", [(61, 43), (301, 239)])  # world-frame and camera-plane kernels
@pytest.mark.parametrize("K", [2, 41, 200])
@pytest.mark.parametrize("normals,pose", [(1, True), (0, False)])
def test_two_blocks_as_clusters(W, H, K, normals, pose):
    oracle.build()
    rng = np.random.default_rng(K)
    poses = [synth.look_at_pose((0.0, 0.0, -4.0)), synth.look_at_pose((2.5, 1.0, 2.5))]
    q = lambda x: float(np.float32(x))  # what the library sees
    views = [dict(W=W, H=H, fx=q(1.1 * W), fy=q(0.9 * W), cx=q(0.4 * W), cy=q(0.6 * H), object=0, pose=i,
                  flow_target=(1 - i, -1)) for i in range(2)]
    s = synth.make_scene([synth.random_gaussians(rng, K)], views, poses)
    assert (s.n_pixels > 131072) == (W > 100)
    _, r, dev = gpu_forward(s, fmb.default_params(n_flow=1, want_normals=normals, bwd_gblocks=2, bwd_ray_tile=256))
    ref = oracle.render_scene(s, n_flow=1)
    ups = masked_upstream(s, ref["alpha"], 1, nnorm_ref=nnorm_batched(s, ref["saved"]))
    if not normals:
        ups["g_normal"] = np.zeros_like(ups["g_normal"])
    g = gpu_backward(r, dev, ups, want_pose=pose)
    refg = oracle.backward_scene(s, ups["g_depth"], ups["g_alpha"], ups["g_normal"] if normals else None, ups["g_flow"],
                                 n_flow=1)
    compare_grads(g, refg, keys=("means", "chol", "weights") + (("poses",) if pose else ()))


@pytest.mark.gpu
@pytest.mark.parametrize("W,H", [(61, 43), (301, 239)])
@pytest.mark.parametrize("K", [2, 41, 200])
def test_clusters_change_no_bit(W, H, K):
    """The same blocks without clusters (persistent mode): the same records and sums in the
    same order, so the deterministic gradients of the Gaussians are the same bits."""
    rng = np.random.default_rng(K)
    poses = [synth.look_at_pose((0.0, 0.0, -4.0)), synth.look_at_pose((2.5, 1.0, 2.5))]
    views = [dict(W=W, H=H, fx=W, fy=W, cx=W / 2, cy=H / 2, object=0, pose=i, flow_target=(1 - i, -1)) for i in range(2)]
    s = synth.make_scene([synth.random_gaussians(rng, K)], views, poses)
    ups = dict(zip(("g_depth", "g_alpha", "g_normal", "g_flow"), synth.upstream_grads(rng, s.n_pixels, 1)))
    got = []
    for persistent in (0, 1):
        params = fmb.default_params(n_flow=1, bwd_gblocks=2, deterministic=1, use_persistent=persistent)
        _, r, dev = gpu_forward(s, params)
        got.append(gpu_backward(r, dev, ups))
    for k in ("means", "chol", "weights"):
        np.testing.assert_array_equal(got[0][k], got[1][k])
