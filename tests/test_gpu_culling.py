"""The warps' culling of list entries (block_misses) drops only particles that every pixel of the warp
rejects: the counting variant of the forward walks every entry whose rectangle is near, and must give
the same bits, over the shapes that stress the bound's rounding slack."""
import numpy as np
import pytest
import torch

from gpu_helpers import run_gpu
from paper_2412_12507_gb300 import render, synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__
    __graft_entry__.build()


def _cam(model, rs, W=149, H=107):
    kw = {}
    if rs:  # a violent motion: 6 degrees and half a unit over the exposure
        qe, te = synth.rs_end_pose(0.5, 6.0)
        kw = dict(q_end=qe, t_end=te, rolling_shutter=1)
    if model == "fisheye":
        kw["k"] = (0.2, -0.1, 0.05, -0.01)
    if model == "pinhole_radial":
        kw["k"] = (-0.25, 0.08, 0.0, 0.0)
    return synth.camera(model, W, H, fx=0.5 * W, fy=0.5 * W, **kw)


def _scene(kind):
    sc = synth.scene_cube(6000, 11, log_s=(-3.0, 0.8), deg=1)
    rng = np.random.default_rng(3)
    if kind == "thin":  # needles and sheets, axes ratios up to 1e4
        sc["log_scales"] = (sc["log_scales"] - 4.6 * (rng.random((6000, 3)) < 0.5) -
                            4.6 * (rng.random((6000, 3)) < 0.3)).astype(np.float32)
    elif kind == "near":  # all around and right at the camera
        sc["means"] = (0.6 * rng.standard_normal((6000, 3)) + np.array([0, 0, 0.4])).astype(np.float32)
    elif kind == "far":  # the camera's offset dwarfs the particles' extent
        sc["means"] = (sc["means"] * 40).astype(np.float32)
        sc["log_scales"] = (sc["log_scales"] + 3.0).astype(np.float32)
    elif kind == "faint":
        sc["opacity_logits"] = (sc["opacity_logits"] - 4.0).astype(np.float32)
    return sc


@pytest.mark.parametrize("kind", ["plain", "thin", "near", "far", "faint"])
@pytest.mark.parametrize("model,rs", [("pinhole", 0), ("pinhole", 1), ("fisheye", 0), ("fisheye", 1),
                                      ("pinhole_radial", 1)])
def test_culled_walk_is_the_full_walk(kind, model, rs):
    sc, cam = _scene(kind), _cam(model, rs)
    for tw, th in ((16, 16), (8, 8), (8, 12), (12, 8), (64, 1)):
        for mode in ({}, dict(alpha_min=1e-6)) if (tw, th) == (16, 16) else ({},):
            op = synth.options(tile_w=tw, tile_h=th, **mode)
            g = run_gpu(sc, cam, op)
            stats = torch.zeros(2, dtype=torch.int64, device="cuda")
            f = render.composite_forward(g["scene"], cam, op, g["proj"], g["binning"], stats=stats)
            assert stats[1].item() > 1000
            for k in ("rgb", "alpha", "t_final", "n_used"):
                assert torch.equal(getattr(f, k), getattr(g["frame"], k)), (k, tw, th, mode)
