"""Particles so large that |d_g|^2 = |S^-1 R^T d|^2 is a subnormal number (scales above 1e19) are a uniform
veil of opacity sigma: their image and gradients are those of any other particle whose response is 1
everywhere in the image."""
import numpy as np
import pytest
import torch

from gpu_helpers import to_np
from paper_2412_12507_gb300 import render, synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__
    __graft_entry__.build()


def _step(log_s, cam, op):
    """Image and gradients of a particle of scale exp(log_s) in front of an ordinary one, both listed by
    every tile (the lists are given: the projection would cull the first)."""
    rng = np.random.default_rng(0)
    scene = render.Scene.from_arrays(dict(
        means=np.array([[0, 0, 3], [0.1, 0, 3.5]], np.float32), log_scales=np.array([[log_s] * 3, [-1] * 3], np.float32),
        quats=np.array([[1, 0, 0, 0], [1, 0.2, 0, 0]], np.float32), opacity_logits=np.zeros(2, np.float32),
        sh=0.2 * rng.standard_normal((2, 4, 3)).astype(np.float32), sh_degree=1))
    proj, T = render.project(scene, cam, op), render.tile_count(cam, op)
    proj.rect = torch.tensor([[0, 0, cam["width"] - 1, cam["height"] - 1]] * 2, dtype=torch.int16, device="cuda")
    proj.depth = torch.tensor([1.0, 2.0], device="cuda")
    proj.ntiles = torch.full((2,), T, dtype=torch.int32, device="cuda")
    b = render.bin_and_sort(proj, cam, op, 2 * T)
    f = render.composite_forward(scene, cam, op, proj, b)
    g = render.composite_backward(scene, cam, op, proj, b, f, torch.ones_like(f.rgb), torch.ones_like(f.alpha))
    return f, {k: to_np(v).astype(np.float64) for k, v in g.items()}


@pytest.mark.parametrize("mode", [{}, dict(colour_mode=1), dict(kernel_degree=3), dict(kbuffer=2)])
@pytest.mark.parametrize("rs", [0, 1])
def test_subnormal_direction_norm(rs, mode):
    kw = {}
    if rs:
        qe, te = synth.rs_end_pose(0.05, 2.0)
        kw = dict(q_end=qe, t_end=te, rolling_shutter=1)
    cam, op = synth.camera("fisheye" if rs else "pinhole", 21, 19, fx=16.0, fy=16.0, **kw), synth.options(**mode)
    f0, g0 = _step(30.0, cam, op)
    for log_s in (44.0, 45.0, 46.0, 48.0, 50.0):
        f, g = _step(log_s, cam, op)
        assert torch.equal(f.rgb, f0.rgb) and torch.equal(f.alpha, f0.alpha)
        for k in g:
            assert np.isfinite(g[k]).all(), (log_s, k)
            # the same per-pixel terms (omega^2 is below 1e-24 throughout): only the order of the 399
            # pixels' FP32 sums may differ, 399 x 2^-24 = 2.4e-5 of the largest sum
            if k in ("opacity_logits", "sh"):
                assert np.abs(g[k] - g0[k]).max() <= 2.4e-5 * np.abs(g0[k]).max(), (log_s, k)
