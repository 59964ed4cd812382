"""The tile-order compositing kernels walk a tile with independent warps of 64 pixels: the edges of
that walk's chunks of list entries, of its pixel layouts and of its aligned copies."""
import numpy as np
import pytest
import torch

import oracle
from gpu_helpers import TOL, compare_frame, run_gpu, to_np
from paper_2412_12507_gb300 import render, synth

pytestmark = pytest.mark.gpu

# one warp (8x8), squares with a ragged image, two 8x4 blocks with an empty second half (8x12),
# row-major with an unfilled last warp (12x8), five warps in two blocks (20x16), eight in two (16x32)
TILES = [(8, 8), (16, 16), (8, 12), (12, 8), (20, 16), (16, 32), (64, 1)]


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__
    __graft_entry__.build()


def _list_case(n, deg, rs):
    """n broad, faint particles in front of a small ragged image: every tile lists all of them, and
    no pixel saturates."""
    sc = synth.scene_cube(n, 40 + n, log_s=(-0.7, 0.2), logit_std=0.1, deg=deg, lo=(-.5, -.5, 2.5), hi=(.5, .5, 3.5))
    sc["opacity_logits"] = sc["opacity_logits"] - np.float32(3.5)
    kw = {}
    if rs:
        qe, te = synth.rs_end_pose(0.05, 2.0)
        kw = dict(q_end=qe, t_end=te, rolling_shutter=1)
    return sc, synth.camera("fisheye" if rs else "pinhole", 37, 29, fx=30.0, fy=30.0, **kw)


@pytest.mark.parametrize("n", [1, 24, 25, 32, 33, 64, 65])
@pytest.mark.parametrize("deg,rs", [(0, 0), (2, 1), (3, 0)])
def test_chunk_edges_render_matches_oracle(n, deg, rs):
    sc, cam = _list_case(n, deg, rs)
    op = synth.options()
    ref = oracle.render(sc, cam, op, tol=TOL)
    g = run_gpu(sc, cam, op)
    r = compare_frame(g["frame"], ref)
    assert r["n_bad"] == 0, r
    assert g["K"] >= 4 * n  # four of the six tiles list every particle


@pytest.mark.parametrize("mode", [{}, dict(colour_mode=1), dict(kernel_degree=3)])
def test_pixel_layouts_give_identical_images(mode):
    """Every layout of the pixels over warps, and rows of SH coefficients without 16-byte alignment,
    give the bits of the 16 x 16 tiles."""
    sc = synth.scene_cube(700, 5, log_s=(-3.0, 0.6), deg=3)
    cam = synth.camera("fisheye", 101, 67, k=(0.02, -0.01, 0.0, 0.0))
    ref = None
    for tw, th in TILES:
        f = run_gpu(sc, cam, synth.options(tile_w=tw, tile_h=th, **mode))["frame"]
        img = [to_np(t) for t in (f.rgb, f.alpha, f.t_final)]
        if ref is None:
            ref = img
        assert all(np.array_equal(a, b) for a, b in zip(img, ref)), (tw, th)
    op = synth.options(**mode)
    g = run_gpu(sc, cam, op)
    s = g["scene"]
    sh = torch.empty(s.sh.numel() + 1, device="cuda")[1:].view_as(s.sh).copy_(s.sh)
    assert sh.data_ptr() % 16 == 4
    f = render.composite_forward(render.Scene(s.means, s.log_scales, s.quats, s.opacity_logits, sh, 3), cam, op,
                                 g["proj"], g["binning"])
    assert np.array_equal(to_np(f.rgb), ref[0])
