"""The k-buffer kernels over every layout of a tile's pixels (whose warps cull the tile's list with a plane
or a ball of rays) and, backward, over the ways of summing a step's gradients: degrees 0 to 3, few
tiles and more than the chip has SMs, particles that cover a warp and particles that cover a few pixels."""
import numpy as np
import pytest
import torch

import oracle
from gpu_helpers import TOL, grad_compare, run_gpu, to_np
from paper_2412_12507_gb300 import render, synth

pytestmark = pytest.mark.gpu

TILES = [(8, 8), (16, 16), (8, 12), (12, 8), (20, 16), (16, 32), (64, 1)]


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__
    __graft_entry__.build()


@pytest.mark.parametrize("k", [1, 4, 16])
@pytest.mark.parametrize("rs", [0, 1])
def test_layouts_give_identical_images(rs, k):
    sc = synth.scene_cube(700, 5, log_s=(-3.0, 0.6), deg=2)
    kw = {}
    if rs:
        qe, te = synth.rs_end_pose(0.05, 2.0)
        kw = dict(q_end=qe, t_end=te, rolling_shutter=1)
    cam = synth.camera("fisheye", 101, 67, k=(0.02, -0.01, 0.0, 0.0), **kw)
    ref = None
    for tw, th in TILES:
        f = run_gpu(sc, cam, synth.options(tile_w=tw, tile_h=th, kbuffer=k))["frame"]
        img = [to_np(t) for t in (f.rgb, f.alpha, f.t_final)]
        ref = ref or img
        assert all(np.array_equal(a, b) for a, b in zip(img, ref)), (tw, th)


# the second size has 165 tiles of 16 x 16 and 660 of 8 x 8
@pytest.mark.parametrize("W,H,log_s,n", [(61, 45, -2.2, 250), (239, 175, -3.6, 1500)])
@pytest.mark.parametrize("deg", [0, 1, 2, 3])
def test_backward_matches_oracle(deg, W, H, log_s, n):
    sc = synth.scene_cube(n, 6 + deg, log_s=(log_s, 0.5), deg=deg)
    cam = synth.camera("pinhole", W, H, fx=0.9 * W, fy=0.9 * W)
    op = synth.options(kbuffer=4)
    proj = oracle.project(sc, cam, op, TOL)
    f = oracle.render(sc, cam, dict(op, eps_tau=1e-4), proj=proj, tol=TOL)
    ok = (f["flags"] & oracle.F_BACKWARD_TIES) == 0  # zero upstream where the decisions may differ
    rng = np.random.default_rng(deg)
    w_rgb, w_a = rng.standard_normal((H * W, 3)) * ok[:, None], rng.standard_normal(H * W) * ok
    ref = oracle.backward(sc, cam, op, proj, (f["px"], f["py"]), w_rgb, w_a, magnitudes=True)
    up = [torch.as_tensor(a.astype(np.float32)).cuda() for a in (w_rgb.T.reshape(3, H, W), w_a.reshape(H, W))]
    for tw, th in TILES if W < 100 else TILES[:2]:
        o = dict(op, tile_w=tw, tile_h=th)
        g = run_gpu(sc, cam, o)
        grads = render.composite_backward(g["scene"], cam, o, g["proj"], g["binning"], g["frame"], *up)
        for key in ("means", "log_scales", "quats", "opacity_logits", "sh"):
            grad_compare(to_np(grads[key]), ref[key], ref["mag"][key], key)
